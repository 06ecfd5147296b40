// air_raster.cu -- Section 2 step vi: the output image as a finest-level
// raster, each finest pixel from the leaf that covers it, either that leaf's
// value or a bilinear interpolation on the leaf's own level between adjacent
// pixels of differing resolution (the super-resolution step the paper allows
// and leaves open).
#include "air_handle.cuh"
#include "air_tree.cuh"

namespace air {

// One thread per finest pixel (x, y) of an (n0 2^Lm)^2 raster (for base images,
// trees without level maps and rasters of fewer pixels than maps_pixels; else
// k_raster_maps). The covering
// leaf is the deepest node containing the pixel. For the bilinear form, with
// s = Lm - L, the pixel centre on the level-L grid is
// u = (x + 1/2) 2^-s - 1/2 = (2x + 1 - 2^s) / 2^(s+1): its floor is an
// arithmetic shift and its fraction an exact dyadic number, so the weights
// carry no rounding.
__global__ void k_raster(TreeView t, int Lm, int mode, const float *__restrict__ val,
                         float *__restrict__ out) {
  const int nf = t.n0 << Lm;
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= (int64_t)nf * nf) return;
  const int x = (int)(k % nf), y = (int)(k / nf);
  const int leaf = descend(t, 0, Lm, x, y);
  if (mode == AIR_RASTER_NEAREST) {
    out[k] = val[leaf];
    return;
  }
  const int L = t.lvl[leaf];
  const int s = Lm - L;
  const int nl = t.n0 << L;
  const int nu = 2 * x + 1 - (1 << s), nv = 2 * y + 1 - (1 << s);
  const int i0 = nu >> (s + 1), j0 = nv >> (s + 1);
  const float sc = __int_as_float((127 - (s + 1)) << 23);  // 2^-(s+1)
  const float fu = (float)(nu - i0 * (2 << s)) * sc;
  const float fv = (float)(nv - j0 * (2 << s)) * sc;
  const int ia = min(max(i0, 0), nl - 1), ib = min(max(i0 + 1, 0), nl - 1);
  const int ja = min(max(j0, 0), nl - 1), jb = min(max(j0 + 1, 0), nl - 1);
  const float v00 = val[descend(t, 0, L, ia, ja)], v10 = val[descend(t, 0, L, ib, ja)];
  const float v01 = val[descend(t, 0, L, ia, jb)], v11 = val[descend(t, 0, L, ib, jb)];
  const float gu = 1.f - fu, gv = 1.f - fv;
  out[k] = (gu * gv) * v00 + (fu * gv) * v10 + (gu * fv) * v01 + (fu * fv) * v11;
}

// The same raster through the tree's level maps (air_tree.cuh), for images with
// at least one level: a thread takes the 2 x 2 finest pixels of one level
// Lm - 1 pixel. One map entry then tells the case:
//   a node with children: the four pixels are its children, finest leaves,
//     which keep their values (their index fractions are zero);
//   a leaf: the four pixels lie between it and its 8 neighbours at its level;
//   none: a coarser leaf, level L <= Lm - 2; the four pixels share the four
//     level-L pixels they lie between (the cell boundary x = 2^(s-1) mod 2^s,
//     s = Lm - L >= 2, is even).
// Before, every pixel descended from its base pixel through up to Lm child
// links five times: 45 us for a 2048^2 raster of which 2.5 us are its writes.
// VEC: out is 8-byte aligned.
template <bool VEC>
__global__ void __launch_bounds__(256) k_raster_maps(TreeView t, const int32_t *__restrict__ lmap, int Lm,
                                                     int mode, const float *__restrict__ val,
                                                     float *__restrict__ out) {
  const int nh = t.n0 << (Lm - 1);
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= (int64_t)nh * nh) return;
  const int jc = (int)(q / nh), ic = (int)(q - (int64_t)jc * nh);
  float v[4];  // pixels (2 ic + (e & 1), 2 jc + (e >> 1))
  int k;       // the level Lm - 1 node, or -1
  if (Lm == 1) k = jc * t.n0 + ic;
  else k = __ldg(lmap + level_map_offset(t.n0, Lm - 1) + q);
  const int c = k >= 0 ? t.child[k] : -1;
  if (c >= 0) {
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] = val[c + e];
  } else {
    int L = Lm - 1;
    if (k < 0) {  // a coarser leaf
      while (k < 0) {
        --L;
        const int s = Lm - 1 - L;
        if (L == 0) k = (jc >> s) * t.n0 + (ic >> s);
        else k = __ldg(lmap + level_map_offset(t.n0, L) + (int64_t)(jc >> s) * (t.n0 << L) + (ic >> s));
      }
    }
    if (mode == AIR_RASTER_NEAREST) {
      const float x = val[k];
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] = x;
    } else {
      const int s = Lm - L, nl = t.n0 << L;
      const float sc = __int_as_float((127 - (s + 1)) << 23);  // 2^-(s+1)
      // columns and rows of level-L pixels the two finest columns and rows lie
      // between: [i0, i0 + 1], and for s = 1 one further for the second
      int i0[2], j0[2];
      float fu[2], fv[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int nu = 2 * (2 * ic + e) + 1 - (1 << s), nv = 2 * (2 * jc + e) + 1 - (1 << s);
        i0[e] = nu >> (s + 1);
        j0[e] = nv >> (s + 1);
        fu[e] = (float)(nu - i0[e] * (2 << s)) * sc;
        fv[e] = (float)(nv - j0[e] * (2 << s)) * sc;
      }
      float w[3][3];  // values of level-L pixels (i0[0] + a, j0[0] + b)
      const int na = i0[1] - i0[0] + 2;  // 2 or 3, the same for both axes
#pragma unroll
      for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int a = 0; a < 3; ++a)
          if (a < na && b < na) {
            const int ii = min(max(i0[0] + a, 0), nl - 1), jj = min(max(j0[0] + b, 0), nl - 1);
            w[b][a] = val[map_deepest(t, lmap, L, ii, jj)];
          }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int x = e & 1, y = e >> 1;
        const bool dx = x && na == 3, dy = y && na == 3;
        const float v00 = dy ? (dx ? w[1][1] : w[1][0]) : (dx ? w[0][1] : w[0][0]);
        const float v10 = dy ? (dx ? w[1][2] : w[1][1]) : (dx ? w[0][2] : w[0][1]);
        const float v01 = dy ? (dx ? w[2][1] : w[2][0]) : (dx ? w[1][1] : w[1][0]);
        const float v11 = dy ? (dx ? w[2][2] : w[2][1]) : (dx ? w[1][2] : w[1][1]);
        const float gu = 1.f - fu[x], gv = 1.f - fv[y];
        v[e] = (gu * gv) * v00 + (fu[x] * gv) * v10 + (gu * fv[y]) * v01 + (fu[x] * fv[y]) * v11;
      }
    }
  }
  float *o = out + (int64_t)(2 * jc) * (2 * nh) + 2 * ic;
  if (VEC) {
    *reinterpret_cast<float2 *>(o) = make_float2(v[0], v[1]);
    *reinterpret_cast<float2 *>(o + 2 * nh) = make_float2(v[2], v[3]);
  } else {
    o[0] = v[0];
    o[1] = v[1];
    o[2 * nh] = v[2];
    o[2 * nh + 1] = v[3];
  }
}

// Pixels from which k_raster_maps is the faster one. A raster of fewer pixels is
// bound by the latency of one thread, which k_raster_maps makes longer, and by
// the launch. Calls with k_raster and with k_raster_maps, us, one to nine levels:
// 512^2 pixels 22 to 27 and 23 to 28; 1024^2 nearest 24.4 to 27.1 and 24.6 to
// 29.4, bilinear 26.3 to 34.9 and 26.2 to 32.1; 1536^2 nearest 29.8 to 31.4 and
// 29.3 to 33.1, bilinear 38.8 to 51.4 and 33.4 to 39.6; 2048^2 nearest 32.7 to
// 36.2 and 27.3 to 32.5, bilinear 42.4 to 49.0 and 33.2 to 39.4.
static int64_t maps_pixels(int mode) { return (int64_t)(mode == AIR_RASTER_NEAREST ? 3 : 2) << 20; }

static bool is_device_ptr(const void *p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

air_status render_raster(air_grid *g, int32_t quantity, int32_t band, int32_t mode, float *out,
                         int64_t n_out) {
  if (!out) return set_error(AIR_ERR_ARG, "out must not be NULL");
  if (mode != AIR_RASTER_NEAREST && mode != AIR_RASTER_BILINEAR)
    return set_error(AIR_ERR_ARG, "unknown raster mode %d", mode);
  if (quantity != AIR_RASTER_INTENSITY && quantity != AIR_RASTER_SUM && quantity != AIR_RASTER_COLDENS)
    return set_error(AIR_ERR_ARG, "unknown raster quantity %d", quantity);
  if (!g->raster.ok) return set_error(AIR_ERR_ARG, "no single-view adaptive image to rasterise");
  if (quantity == AIR_RASTER_INTENSITY && (band < 0 || band >= g->gv.n_bands))
    return set_error(AIR_ERR_ARG, "band %d out of range", band);
  if (quantity == AIR_RASTER_INTENSITY && !g->ws.I)
    return set_error(AIR_ERR_ARG, "the image's band intensities were streamed to host memory");
  const int n0 = g->raster.n0, Lm = g->raster.Lm;
  const int64_t nf = (int64_t)n0 << Lm;
  if (nf > (1 << 30)) return set_error(AIR_ERR_ARG, "raster side %lld too large", (long long)nf);
  const int64_t n = nf * nf;
  if (n_out < n) return set_error(AIR_ERR_CAPACITY, "raster needs %lld floats, out holds %lld", (long long)n, (long long)n_out);
  Workspace &w = g->ws;
  const TreeView t = w.tree(n0, Lm);
  const float *val = quantity == AIR_RASTER_COLDENS ? t.N
                     : (quantity == AIR_RASTER_SUM ? t.p : t.I + (int64_t)band * t.cap);
  cudaStream_t st = g->stream;
  const bool dev = is_device_ptr(out);
  float *dst = out;
  if (!dev) {
    cudaError_t e = ensure((void **)&g->raster.scratch, &g->raster.scratch_b, sizeof(float) * (size_t)n);
    if (e != cudaSuccess) return cuda_fail(e, "raster staging");
    dst = g->raster.scratch;
  }
  const int64_t blocks = (n + 255) / 256;
  if (blocks > 0x7fffffff) return set_error(AIR_ERR_ARG, "raster too large");
  if (n >= maps_pixels(mode) && (Lm == 1 || (Lm > 1 && g->raster.lmap))) {
    const unsigned quads = (unsigned)((n / 4 + 255) / 256);
    if (((uintptr_t)dst & 7) == 0) k_raster_maps<true><<<quads, 256, 0, st>>>(t, g->raster.lmap, Lm, mode, val, dst);
    else k_raster_maps<false><<<quads, 256, 0, st>>>(t, g->raster.lmap, Lm, mode, val, dst);
  } else {
    k_raster<<<(unsigned)blocks, 256, 0, st>>>(t, Lm, mode, val, dst);
  }
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess && !dev) e = cudaMemcpyAsync(out, dst, sizeof(float) * (size_t)n, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_fail(e, "air_render_raster");
  return AIR_OK;
}

}  // namespace air

extern "C" AIR_API air_status air_render_raster(air_grid *g, int32_t quantity, int32_t band,
                                                int32_t mode, float *out, int64_t n_out) {
  air::clear_error();
  if (!g) return air::set_error(AIR_ERR_ARG, "grid handle is NULL");
  return air::render_raster(g, quantity, band, mode, out, n_out);
}
