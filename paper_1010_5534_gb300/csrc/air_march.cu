// air_march.cu -- launches of the per-ray march (device code in air_march.cuh,
// the kernel and its forms in air_march_kernel.cuh).
#include <algorithm>

#include "air_march_kernel.cuh"

namespace air {

__global__ void k_band_sum(const float *__restrict__ I, int n_bands, int64_t stride, int64_t first,
                           int64_t count, const int32_t *__restrict__ list, float *__restrict__ p,
                           int64_t ioff) {
  const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= count) return;
  const int64_t k = list ? (int64_t)list[r] : first + r;
  float s = 0.f;
  for (int b = 0; b < n_bands; ++b) s += I[(int64_t)b * stride + (k - ioff)];
  p[k] = s;
}

// Band sums of the new nodes of sweep q, counted on the device, unless they are
// more than `most` (their threads then held all bands and summed them).
__global__ void k_band_sum_dev(const float *I, int n_bands, int64_t stride, const SweepState *S, int q,
                               int64_t most, float *__restrict__ p) {
  wait_prior_grid();
  const int64_t first = S->slot[q & 3].n, end = S->slot[(q + 1) & 3].n;
  if (end - first > most) return;
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  for (int64_t k = first + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < end; k += step) {
    float s = 0.f;
    for (int b = 0; b < n_bands; ++b) s += I[(int64_t)b * stride + k];
    p[k] = s;
  }
}

// Rays whose threads (one per band chunk) fill the GPU twice in the form for
// few rays.
static int64_t few_rays(int NBT, int chunks) {
  const int blocks = NBT <= 4 ? MinBlocks<4, -1>::value : MinBlocks<8, -1>::value;
  return (int64_t)sm_count() * blocks * kMarchBlock * 2 / chunks;
}

// Compiled in air_march_<NBT>.cu and air_march_axis.cu.
extern template cudaError_t march_general<1>(const MarchLaunch &);
extern template cudaError_t march_general<2>(const MarchLaunch &);
extern template cudaError_t march_general<4>(const MarchLaunch &);
extern template cudaError_t march_general<8>(const MarchLaunch &);
extern template cudaError_t march_general<16>(const MarchLaunch &);
extern template cudaError_t march_axis_one<0>(const MarchLaunch &);
extern template cudaError_t march_axis_one<1>(const MarchLaunch &);
extern template cudaError_t march_axis_one<2>(const MarchLaunch &);

// Threads that the parts of a wide launch should fill (wide_parts): twice those
// resident at once (32-band clumps: 8.27 ms; filled once 9.15, four times 8.62).
static int64_t wide_fill_threads() { return (int64_t)sm_count() * kWideBlocks * kMarchBlock * 2; }

// Inclined rays with more than 8 bands per thread go to the wide form. (Bands in
// registers up to 8: the 8-band cone, 1500^2 fixed, 1.09 ms, 1.17 in the wide
// form; 5 hot bands 300 us, 318. With 32 bands the wide form's one walk wins over
// four: clumps 11.8 -> 7.9 ms, and 8 views x 16 bands 16.4 -> 13.2.) Rays that
// move along no axis (cells too large, see make_geom) take the same forms.
static bool is_wide(int nbt, int moving) { return moving != 1 && nbt > 8; }

// The march kernel with NBT bands per thread (the wide form: per chunk, any
// even number, and `fill` threads to fill).
static cudaError_t launch_nbt(int NBT, bool few, int64_t fill, const GridView &g, const RayGeom &rg,
                              const RaySource &src, const RayOut &out, const MarchTune &tune,
                              cudaStream_t st) {
  const int moving = (rg.Dhi[0] != 0.f) + (rg.Dhi[1] != 0.f) + (rg.Dhi[2] != 0.f);
  const bool wide = is_wide(NBT, moving) && !few;
  const int chunks = (g.n_bands + NBT - 1) / NBT;
  int64_t threads;
  if (src.mode == 0) {
    threads = src.count;
  } else if (src.mode == 1) {
    const int tw = src.tile_w, th = 32 / tw;
    const int64_t tiles = (int64_t)((src.n0 + tw - 1) / tw) * ((src.n0 + th - 1) / th);
    threads = tiles * 32;
  } else {
    threads = 1;  // the count is on the device; the grid is sized per form
  }
  if (threads <= 0) return cudaSuccess;
  const int64_t warps = (int64_t)sm_count() * (kMarchBlock / 32) *
                        (wide ? kWideBlocks : (few ? (NBT <= 4 ? MinBlocks<4, -1>::value : MinBlocks<8, -1>::value) : 4));
  RaySource rs = src;
  rs.width = NBT;
  rs.fill = fill;
  rs.rpw = moving == 1 ? 32 : rays_per_warp(threads, chunks * (wide ? wide_parts(threads, std::min(NBT, g.n_bands), fill) : 1), warps);
  const int64_t per_block = kMarchBlock / 32 * rs.rpw;
  const int64_t blocks = (threads + per_block - 1) / per_block;
  if (blocks > 0x7fffffff) return cudaErrorInvalidValue;
  const MarchLaunch m{g, rg, rs, out, blocks, chunks, tune.fp64_level, st, few};
  if (wide) {
    const cudaError_t e = march_wide(m, threads);
    return e != cudaSuccess ? e : cudaGetLastError();
  }
  cudaError_t le;
  if (NBT == 1 && moving == 1) {
    le = rg.Dhi[0] != 0.f ? march_axis_one<0>(m) : (rg.Dhi[1] != 0.f ? march_axis_one<1>(m) : march_axis_one<2>(m));
  } else {
    le = NBT == 1 ? march_general<1>(m)
         : NBT == 2 ? march_general<2>(m)
         : NBT == 4 ? march_general<4>(m)
         : NBT == 8 ? march_general<8>(m) : march_general<16>(m);
  }
  if (le != cudaSuccess) return le;
  return cudaGetLastError();
}

// The kernel's width for a number of bands per thread.
static int width_of(int nbt) { return nbt <= 1 ? 1 : (nbt <= 2 ? 2 : (nbt <= 4 ? 4 : (nbt <= 8 ? 8 : 16))); }

cudaError_t launch_march(const GridView &g, const Camera &cam, const RaySource &rays,
                         const RayOut &out, const MarchTune &tune, cudaStream_t st, int *launches) {
  *launches = 0;
  // default: every band in one thread up to 8 bands; above, chunks of 8 for rays
  // along an axis, and the wide form for inclined ones
  int nbt = g.cell_fmt == kCellLam ? 1 : width_of(tune.nbt > 0 ? tune.nbt : default_bands_per_thread(g.n_bands));
  RayGeom rg = make_geom(g, cam, rays.n0);
  rg.tab = rays.axtab;
  rg.tab_slot = rays.axtab_slot;
  rg.tab_byj = rays.axtab_byj;
  const int moving = (rg.Dhi[0] != 0.f) + (rg.Dhi[1] != 0.f) + (rg.Dhi[2] != 0.f);
  if (rays.mode == 0 && rays.count <= 0) return cudaSuccess;
  RaySource src = rays;
  if (moving > 1 && src.mode == 0 && src.base && src.first == 0 && src.count == (int64_t)src.n0 * src.n0) {
    // a base image in node order is the fixed image of its resolution: a warp
    // takes 8 x 4 pixels, whose rays stay closer than those of 32 in a row
    src.mode = 1;
    src.tile_w = 8;
  }

  // A launch of few inclined rays takes as long as its longest ray, and a ray's
  // time is that of one warp working alone, so its bands are spread over more
  // threads, at most four each (unless the caller has set a width other than the
  // default's: setting that one leaves the default as it is, so the autotuner's
  // widths include it), and it takes the form DIR = -1. `few`: the rays that fill that form's threads
  // twice. Where the count is on the device, both launches are queued and the one
  // that it is not for returns. (Inclined cone, 101^2 base, 4 bands, 30 sweeps,
  // the march: 3.40 ms; with one band per thread 3.75, two 3.71.) Rays along an
  // axis keep the chunks of large launches: their series (column_group) is chosen
  // by the largest opacity of the chunk, so another width gives other last bits.
  const bool free_width = tune.nbt <= 0 || (g.n_bands <= 8 && nbt == width_of(g.n_bands));
  const int narrow = !free_width || moving == 1 ? nbt : std::min(nbt, 4);
  const int nchunks = (g.n_bands + narrow - 1) / narrow;
  if (tune.nbt <= 0 && g.n_bands > 8 && moving > 1) nbt = 16;  // inclined: the wide form
  const bool wide = is_wide(nbt, moving);
  // there is a form for few rays (its 8 or 16 cells ahead are wasted in bricks of
  // 1 or 2 cells: 100^2 pixels, one band, 208 and 213 us, 176 and 135 without it)
  const bool lone = moving > 1 && narrow <= 8 && !(g.kind == AIR_GRID_AMR && g.B <= 2);
  const int64_t few = lone ? few_rays(narrow, nchunks) : 0;
  if (wide && tune.nbt <= 0) nbt = wide_width(g, kMarchBlock);
  const int64_t fill = wide && tune.nbt <= 0 ? wide_fill_threads() : 0;
  const int chunks = (g.n_bands + nbt - 1) / nbt;
  const int64_t total = src.mode == 0 ? src.count : (src.mode == 1 ? (int64_t)src.n0 * src.n0 : 0);
  cudaError_t e;
  if (src.mode != 2) {
    const bool is_few = total <= few;
    *launches = 1;
    e = launch_nbt(is_few ? narrow : nbt, is_few && lone, fill, g, rg, src, out, tune, st);
    if (e != cudaSuccess || !out.p) return e;
    if (is_few ? nchunks == 1 : chunks == 1 && (!wide || wide_parts(total, g.n_bands, fill) == 1)) return e;
    const int64_t first = src.mode == 0 ? src.first : 0;
    *launches = 2;
    if (src.list) {
      k_band_sum<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(out.I, g.n_bands, out.stride, 0, total,
                                                                  src.list, out.p, out.ioff);
      return cudaGetLastError();
    }
    return launch_band_sum(out.I, g.n_bands, out.stride, first, total, out.p, st, out.ioff);
  }
  RaySource s2 = src;
  s2.few = few;
  if (few > 0) {
    s2.part = 1;
    e = launch_nbt(narrow, lone, fill, g, rg, s2, out, tune, st);
    if (e != cudaSuccess) return e;
    *launches = 1;
    s2.part = 2;
  }
  e = launch_nbt(nbt, false, fill, g, rg, s2, out, tune, st);
  ++*launches;
  if (e != cudaSuccess || !out.p) return e;
  int64_t most = chunks > 1 ? INT64_MAX : (few > 0 && nchunks > 1 ? few : 0);
  if (wide && g.n_bands > 2) most = std::max(most, fill / 2);  // dealt to parts up to there
  if (most > 0) {
    ++*launches;
    return launch_pdl(k_band_sum_dev, dim3((unsigned)(sm_count() * 8)), dim3(256), 0, st,
                      (const float *)out.I, g.n_bands, out.stride, (const SweepState *)src.sweep, src.q, most,
                      out.p);
  }
  return cudaSuccess;
}

// Column-table entries (axis_table_entry), one per thread.
__global__ void k_axis_table(GridView g, RayGeom rg, int A, int byj, int n0, int64_t slot,
                             int32_t *tab) {
  const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= 2 * slot) return;
  const int s = x >= slot ? 1 : 0;
  const int64_t e = x - s * slot;
  int L = 0;
  while ((int64_t)n0 * ((((int64_t)1) << (L + 1)) - 1) <= e) ++L;
  const int p = (int)(e - (int64_t)n0 * ((((int64_t)1) << L) - 1));
  tab[x] = axis_table_entry(g, rg, (A + 1 + s) % 3, L, p, (byj >> s) & 1);
}

cudaError_t launch_axis_table(const GridView &g, const Camera &cam, int n0, int lmax,
                              int32_t *tab, int *byj, int64_t *slot, bool *ok, cudaStream_t st) {
  const RayGeom rg = make_geom(g, cam, n0);
  int A = 0;
  *ok = axis_table_view(rg, &A, byj);
  *slot = axis_table_slot(n0, lmax);
  if (!*ok) return cudaSuccess;
  const int64_t n = 2 * *slot;
  k_axis_table<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(g, rg, A, *byj, n0, *slot, tab);
  return cudaGetLastError();
}

cudaError_t launch_band_sum(const float *I, int n_bands, int64_t stride, int64_t first,
                            int64_t count, float *p, cudaStream_t st, int64_t ioff) {
  if (count <= 0) return cudaSuccess;
  const int block = 256;
  k_band_sum<<<(unsigned)((count + block - 1) / block), block, 0, st>>>(I, n_bands, stride, first,
                                                                       count, nullptr, p, ioff);
  return cudaGetLastError();
}

}  // namespace air
