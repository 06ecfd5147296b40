// air_march.cu -- launches of the per-ray march (device code in air_march.cuh,
// the kernel and its forms in air_march_kernel.cuh).
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

// Band sums of the new nodes of sweep q, counted on the device.
__global__ void k_band_sum_dev(const float *__restrict__ I, int n_bands, int64_t stride,
                               const SweepState *__restrict__ S, int q, float *__restrict__ p) {
  wait_prior_grid();
  const int64_t first = S->slot[q & 3].n, end = S->slot[(q + 1) & 3].n;
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  for (int64_t k = first + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < end; k += step) {
    float s = 0.f;
    for (int b = 0; b < n_bands; ++b) s += I[(int64_t)b * stride + k];
    p[k] = s;
  }
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

static cudaError_t launch_nbt(int NBT, const GridView &g, const Camera &cam, const RaySource &src,
                              const RayOut &out, const MarchTune &tune, cudaStream_t st) {
  const int chunks = (g.n_bands + NBT - 1) / NBT;
  const bool dev = src.mode == 2;
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
  const int64_t blocks = (threads + kMarchBlock - 1) / kMarchBlock;
  if (blocks > 0x7fffffff) return cudaErrorInvalidValue;
  RayGeom rg = make_geom(g, cam, src.n0);
  rg.tab = src.axtab;
  rg.tab_slot = src.axtab_slot;
  rg.tab_byj = src.axtab_byj;
  const int moving = (rg.Dhi[0] != 0.f) + (rg.Dhi[1] != 0.f) + (rg.Dhi[2] != 0.f);
  const MarchLaunch m{g, rg, src, out, blocks, chunks, tune.fp64_level, st};
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
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (dev && chunks > 1 && out.p)
    return launch_pdl(k_band_sum_dev, dim3((unsigned)(sm_count() * 8)), dim3(256), 0, st,
                      (const float *)out.I, g.n_bands, out.stride, (const SweepState *)src.sweep, src.q, out.p);
  if (chunks > 1 && out.p) {
    const int64_t first = src.mode == 0 ? src.first : 0;
    const int64_t count = src.mode == 0 ? src.count : (int64_t)src.n0 * src.n0;
    if (src.list) {
      k_band_sum<<<(unsigned)((count + 255) / 256), 256, 0, st>>>(out.I, g.n_bands, out.stride, 0,
                                                                  count, src.list, out.p, out.ioff);
      return cudaGetLastError();
    }
    return launch_band_sum(out.I, g.n_bands, out.stride, first, count, out.p, st, out.ioff);
  }
  return cudaSuccess;
}

cudaError_t launch_march(const GridView &g, const Camera &cam, const RaySource &src,
                         const RayOut &out, const MarchTune &tune, cudaStream_t st) {
  // default: every band in one thread up to 8 bands, chunks of 8 above
  // (32-band adaptive / fixed images of the large grid, one view: 4 bands
  // 1315 / 1365 ms, 8 bands 1251 / 1328 ms, 16 bands 1512 / 1653 ms)
  int nbt = tune.nbt;
  if (nbt <= 0) nbt = default_bands_per_thread(g.n_bands);
  if (g.cell_fmt == kCellLam) nbt = 1;  // one band
  if (nbt <= 1) return launch_nbt(1, g, cam, src, out, tune, st);
  if (nbt <= 2) return launch_nbt(2, g, cam, src, out, tune, st);
  if (nbt <= 4) return launch_nbt(4, g, cam, src, out, tune, st);
  if (nbt <= 8) return launch_nbt(8, g, cam, src, out, tune, st);
  return launch_nbt(16, g, cam, src, out, tune, st);
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
