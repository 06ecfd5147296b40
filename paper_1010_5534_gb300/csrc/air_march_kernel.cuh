// air_march_kernel.cuh -- the march kernel and its launch, as templates over
// the bands one thread carries. Each width is compiled in a translation unit
// of its own (air_march_<width>.cu, air_march_axis.cu), in parallel: one unit
// with every form took 150 s of a build, the slowest of these takes a quarter.
#pragma once
#include <algorithm>

#include "air_march.cuh"
#include "air_refine.cuh"

namespace air {

// One launch of the march, as launch_march resolved it.
struct MarchLaunch {
  const GridView &g;
  const RayGeom &rg;
  const RaySource &src;
  const RayOut &out;
  int64_t blocks;  // of kMarchBlock / 32 warps, src.rpw rays each; with the count on the device, unused
  int chunks;      // band chunks
  int fp64_level;
  cudaStream_t st;
  bool few;        // inclined rays that leave most threads idle: the form DIR = -1
};

// Resident blocks per SM of the one-band kernels of rays parallel to an axis
// (DIR = 1 + A). Measured on the cone-shock bench image, one process, each
// variant twice (AIR / fixed 4096^2 image, ms): 12 blocks with 8-cell groups
// 5.39 / 4.89, 10 blocks 5.22 / 4.82, 8 blocks 5.02 / 4.30, 8 blocks with
// 16-cell groups 4.92 / 4.37 (the form kept). A separate form for launches
// of at most one wave (more registers, deeper load groups) is then the same
// kernel, so there is one.
constexpr int kAxisBlocks = 8;
constexpr int kAxisBlocksSmall = 6;  // bricks of 4 or 8 cells: two bricks' records in registers

// DIR = -1 has the registers of two or three blocks (see DdaChunk).
template <int NBT, int DIR>
struct MinBlocks {
  static constexpr int value = DIR == -1 ? (NBT <= 4 ? 3 : 2)
                               : DIR == -2 ? (NBT <= 1 ? 6 : (NBT <= 2 ? 5 : 4))
                               : DIR >= 4 && DIR <= 6 ? kAxisBlocksSmall
                               : DIR >= 1 ? kAxisBlocks
                               : (NBT <= 1 ? 6 : (NBT <= 2 ? 5 : (NBT <= 4 ? 4 : (NBT <= 8 ? 3 : 2))));
};

constexpr int kMarchBlock = 128;

// Node k's ray: trace it and store its column density, step count and band
// intensities (and their sum when one chunk holds every band).
template <int NBT, bool AMR, int FMT, int DIR>
__device__ __forceinline__ void march_one(const GridView &g, const RayGeom &rg, const RaySource &src,
                                          const RayOut &out, int fp64_level, const BandCtx &bc,
                                          BandRegs<NBT> &br, int chunk, int b0, int nbh,
                                          int64_t k) {
  if (src.use_prop) {
    // the pixel's values from the proposal wave when it traced the pixel
    // (the same trace, so the same bits); else trace it here
    const Proposal &pr = src.prop;
    const int L = src.lvl[k], i = src.pi[k], j = src.pj[k];
    const int64_t b = (int64_t)(j >> L) * src.n0 + (i >> L);
    const int64_t q = prop_index(pr.depth + 4 * b, pr.off[b], L, i, j);
    if (q >= 0) {
      if (chunk == 0) {
        out.N[k] = pr.N[q];
        out.steps[k] = pr.steps[q];
      }
      for (int c = 0; c < nbh; ++c)
        out.I[(int64_t)(b0 + c) * out.stride + k] = pr.I[(int64_t)(b0 + c) * pr.stride + q];
      if (out.p && gridDim.y == 1) out.p[k] = pr.p[q];
      return;
    }
    if (chunk == 0) {
      if (atomicAdd(&src.sweep->slot[src.q & 3].missed, 1ull) == 0ull) atomicAdd(&src.sweep->fb_waves, 1);
      atomicAdd(&src.sweep->fb_total, 1ull);
    }
  }
  RTState<NBT> st;
  trace_ray<NBT, AMR, FMT, DIR>(st, g, rg, src.lvl[k], src.pi[k], src.pj[k], fp64_level, bc, br);
  if (chunk == 0) {
    out.N[k] = st.N;
    out.steps[k] = st.steps;
    if (out.tau0) out.tau0[k] = bc.band[0].kap * st.N;
    if (out.maxlev) out.maxlev[k] = (uint8_t)st.maxlev;
  }
#pragma unroll
  for (int b = 0; b < NBT; ++b)
    if (b < nbh) out.I[(int64_t)(b0 + b) * out.stride + (k - out.ioff)] = st.I[b];
  if (out.p && gridDim.y == 1) {
    float p = 0.f;
#pragma unroll
    for (int b = 0; b < NBT; ++b)
      if (b < nbh) p += st.I[b];
    out.p[k] = p;
  }
}

template <int NBT, bool AMR, int FMT, int DIR>
__global__ void __launch_bounds__(kMarchBlock, MinBlocks<NBT, DIR>::value)
    k_march(GridView g, RayGeom rg, RaySource src, RayOut out, int fp64_level) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int chunk = blockIdx.y;
  const int b0 = chunk * NBT;
  const int nbh = min(NBT, g.n_bands - b0);
  chunk_fill<NBT, FMT>(smem, g, b0);
  const BandCtx bc = chunk_ctx<NBT, FMT>(smem, g, nbh);
  // (what fills the shared memory was written when the grid was loaded)
  wait_prior_grid();
  __syncthreads();
  BandRegs<NBT> br;
  band_regs<NBT, FMT>(br, bc);

  if (src.mode == 2) {
    // new nodes of a sweep counted on the device: warp w of the grid takes rays
    // [rpw w, + rpw), and more from a work counter until the rays run out
    SweepSlot &s0 = src.sweep->slot[src.q & 3];
    const int64_t first = s0.n, count = src.sweep->slot[(src.q + 1) & 3].n - first;
    if ((src.part == 1 && count > src.few) || (src.part == 2 && count <= src.few)) return;
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (kMarchBlock / 32);
    const int rpw = DIR == -1 || DIR == -2 ? rays_per_warp(count, gridDim.y, warps) : 32;
    for (int64_t w = (int64_t)blockIdx.x * (kMarchBlock / 32) + (threadIdx.x >> 5); rpw * w < count;) {
      const int64_t r = rpw * w + lane;
      if (lane < rpw && r < count) march_one<NBT, AMR, FMT, DIR>(g, rg, src, out, fp64_level, bc, br, chunk, b0,
                                                   nbh, first + r);
      if (count <= rpw * warps) return;
      __syncwarp();
      long long next = 0;
      if (lane == 0) next = (long long)atomicAdd(&s0.ray_ctr[chunk], 1ull);
      w = warps + __shfl_sync(0xffffffffu, next, 0);
    }
    return;
  }
  if ((int)(threadIdx.x & 31) >= src.rpw) return;
  const int64_t r = ((int64_t)blockIdx.x * (kMarchBlock / 32) + (threadIdx.x >> 5)) * src.rpw + (threadIdx.x & 31);
  int L, i, j;
  int64_t k;
  if (src.mode == 0) {
    if (r >= src.count) return;
    k = src.list ? (int64_t)src.list[r] : src.first + r;
    L = src.lvl[k];
    i = src.pi[k];
    j = src.pj[k];
  } else {
    const int res = src.n0;
    const int tw = src.tile_w, th = 32 / tw;
    // res <= 2^16: the tiles of 32 pixels number at most 2^27 (+ a row), so
    // 32-bit division does (64-bit division is long and uses FP64 units)
    const uint32_t tiles_x = (uint32_t)(res + tw - 1) / (uint32_t)tw;
    const uint32_t warp = (uint32_t)(r >> 5);
    const uint32_t lane = (uint32_t)(r & 31);
    const uint32_t ty = warp / tiles_x;
    i = (int)((warp - ty * tiles_x) * tw + lane % (uint32_t)tw);
    j = (int)(ty * th + lane / (uint32_t)tw);
    if (i >= res || j >= res) return;
    k = (int64_t)j * res + i;
    L = 0;
  }
  RTState<NBT> st;
  trace_ray<NBT, AMR, FMT, DIR>(st, g, rg, L, i, j, fp64_level, bc, br);
  if (chunk == 0) {
    out.N[k] = st.N;
    out.steps[k] = st.steps;
    if (out.tau0) out.tau0[k] = bc.band[0].kap * st.N;
    if (out.maxlev) out.maxlev[k] = (uint8_t)st.maxlev;
  }
#pragma unroll
  for (int b = 0; b < NBT; ++b)
    if (b < nbh) out.I[(int64_t)(b0 + b) * out.stride + (k - out.ioff)] = st.I[b];
  if (out.p && gridDim.y == 1) {
    float p = 0.f;
#pragma unroll
    for (int b = 0; b < NBT; ++b)
      if (b < nbh) p += st.I[b];
    out.p[k] = p;
  }
}

// The wide form: bands [blockIdx.y width, + width) in wide_parts() parts. A
// warp takes rpw rays of a part at a time (a block of four warps at a time waited
// for its slowest ray: 32-band clumps 8.9 ms, 7.7 by warps).
// Resident blocks per SM (8 views x 16 bands, batched: 6 blocks 14.95 ms, 5 14.73,
// 4 13.51, 3 14.01; 32-band clumps: 12.8, 12.2, 9.3, 9.2: the sums of more blocks
// leave too little L1 for the cells).
constexpr int kWideBlocks = 4;
// The kernel's limit of dynamic shared memory. It is a property of the function,
// shared by every thread that launches it, so it is set to one value above what
// any launch takes (wide_width: 54 KB), not to each launch's own.
constexpr int kWideShared = 64 * 1024;

template <bool AMR, int FMT>
__device__ __forceinline__ void wide_one(const GridView &g, const RayGeom &rg, const RaySource &src,
                                         const RayOut &out, int fp64_level, const WideCtx &wc, int b0,
                                         bool all, int L, int i, int j, int64_t k) {
  if (src.use_prop) {  // as in march_one
    const Proposal &pr = src.prop;
    const int64_t b = (int64_t)(j >> L) * src.n0 + (i >> L);
    const int64_t q = prop_index(pr.depth + 4 * b, pr.off[b], L, i, j);
    if (q >= 0) {
      if (b0 == 0) {
        out.N[k] = pr.N[q];
        out.steps[k] = pr.steps[q];
      }
      for (int c = 0; c < wc.nbh; ++c)
        out.I[(int64_t)(b0 + c) * out.stride + k] = pr.I[(int64_t)(b0 + c) * pr.stride + q];
      if (out.p && all) out.p[k] = pr.p[q];
      return;
    }
    if (b0 == 0) {
      if (atomicAdd(&src.sweep->slot[src.q & 3].missed, 1ull) == 0ull) atomicAdd(&src.sweep->fb_waves, 1);
      atomicAdd(&src.sweep->fb_total, 1ull);
    }
  }
  RTState<0> st;
  trace_wide<AMR, FMT>(st, g, rg, L, i, j, fp64_level, wc);
  if (b0 == 0) {
    out.N[k] = st.N;
    out.steps[k] = st.steps;
    if (out.tau0) out.tau0[k] = wc.band[0].kap * st.N;
    if (out.maxlev) out.maxlev[k] = (uint8_t)st.maxlev;
  }
  float p = 0.f;
  for (int q = 0; q < wc.pairs; ++q) {
    const float4 s = wc.sums[q * blockDim.x];
    float *I = out.I + (int64_t)(b0 + 2 * q) * out.stride + (k - out.ioff);
    I[0] = s.x;
    p += s.x;
    if (2 * q + 1 < wc.nbh) {
      I[out.stride] = s.z;
      p += s.z;
    }
  }
  if (out.p && all) out.p[k] = p;
}

template <bool AMR, int FMT>
__global__ void __launch_bounds__(kMarchBlock, kWideBlocks)
    k_march_wide(GridView g, RayGeom rg, RaySource src, RayOut out, int fp64_level) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int c0 = blockIdx.y * src.width, nb = min(src.width, g.n_bands - c0);
  wide_fill<FMT>(smem, g, c0, src.width);
  float4 *sums = reinterpret_cast<float4 *>(smem + wide_tab_bytes(FMT == kCellXq, g.n_tbins, src.width));
  wait_prior_grid();
  __syncthreads();
  int64_t first = src.first, count = src.count;
  if (src.mode == 2) {
    first = src.sweep->slot[src.q & 3].n;
    count = src.sweep->slot[(src.q + 1) & 3].n - first;
    if ((src.part == 1 && count > src.few) || (src.part == 2 && count <= src.few)) return;
  }
  const int tw = src.tile_w, th = src.mode == 1 ? 32 / tw : 1;
  const uint32_t tiles_x = src.mode == 1 ? (uint32_t)(src.n0 + tw - 1) / (uint32_t)tw : 1u;
  if (src.mode == 1) count = 32 * (int64_t)tiles_x * ((src.n0 + th - 1) / th);
  const int parts = wide_parts(count, nb, src.fill);
  // items of rpw rays and one part; a warp takes its first by its place in the
  // grid and, where the count is on the device, more from the work counter
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (kMarchBlock / 32);
  const int rpw = src.mode == 2 ? rays_per_warp(count, gridDim.y * parts, warps) : src.rpw;
  const int64_t rounds = (count + rpw - 1) / rpw, items = rounds * parts;
  for (int64_t it = (int64_t)blockIdx.x * (kMarchBlock / 32) + (threadIdx.x >> 5); it < items;) {
    const int part = parts == 1 ? 0 : (int)(it / rounds);
    const int64_t r = (it - part * rounds) * rpw + lane;
    int b0;
    const WideCtx wc = wide_ctx<FMT>(smem, sums, src.width, nb, part, parts, &b0);
    bool mine = lane < rpw && r < count && wc.pairs > 0;
    int64_t k = first + r;
    int L = 0, i = 0, j = 0;
    if (src.mode == 1) {
      // (32-bit division as in k_march)
      const uint32_t tile = (uint32_t)(r >> 5), x = (uint32_t)(r & 31), ty = tile / tiles_x;
      i = (int)((tile - ty * tiles_x) * tw + x % (uint32_t)tw);
      j = (int)(ty * th + x / (uint32_t)tw);
      mine = mine && i < src.n0 && j < src.n0;
      k = (int64_t)j * src.n0 + i;
    } else if (mine) {
      if (src.mode == 0 && src.list) k = (int64_t)src.list[r];
      L = src.lvl[k];
      i = src.pi[k];
      j = src.pj[k];
    }
    if (mine) wide_one<AMR, FMT>(g, rg, src, out, fp64_level, wc, c0 + b0, gridDim.y == 1 && parts == 1, L, i, j, k);
    if (items <= warps) return;
    __syncwarp();
    long long next = 0;
    if (lane == 0) next = (long long)atomicAdd(&src.sweep->slot[src.q & 3].ray_ctr[blockIdx.y], 1ull);
    it = warps + __shfl_sync(0xffffffffu, next, 0);
  }
}

template <bool AMR, int FMT>
static cudaError_t march_wide_form(const MarchLaunch &m, int64_t rays) {
  const int width = m.src.width;
  const size_t smem = wide_tab_bytes(FMT == kCellXq, m.g.n_tbins, width) + wide_sum_bytes(width, kMarchBlock);
  if (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(k_march_wide<AMR, FMT>, cudaFuncAttributeMaxDynamicSharedMemorySize, kWideShared);
    if (e != cudaSuccess) return e;
  }
  const int64_t blocks = m.src.mode == 2 ? (int64_t)sm_count() * kWideBlocks
                                         : m.blocks * wide_parts(rays, std::min(width, m.g.n_bands), m.src.fill);
  if (blocks > 0x7fffffff) return cudaErrorInvalidValue;
  return launch_pdl(k_march_wide<AMR, FMT>, dim3((unsigned)blocks, m.chunks), dim3(kMarchBlock), smem, m.st, m.g,
                    m.rg, m.src, m.out, m.fp64_level);
}

// Inclined rays in the wide form (m.src.width, m.src.fill set); `rays`: the
// launch's threads per band chunk where the host knows them.
static inline cudaError_t march_wide(const MarchLaunch &m, int64_t rays) {
  const bool amr = m.g.kind == AIR_GRID_AMR;
  if (m.g.cell_fmt == kCellRho) return amr ? march_wide_form<true, kCellRho>(m, rays) : march_wide_form<false, kCellRho>(m, rays);
  return amr ? march_wide_form<true, kCellXq>(m, rays) : march_wide_form<false, kCellXq>(m, rays);
}

// The launch grid of form DIR: blocks over the rays, or, with the count on
// the device, one wave of the form's resident blocks taking work from the
// counter.
template <int NBT, int DIR>
static dim3 march_grid(const MarchLaunch &m) {
  return dim3((unsigned)(m.src.mode == 2 ? sm_count() * MinBlocks<NBT, DIR>::value : m.blocks), m.chunks);
}

template <int NBT, bool AMR, int FMT, int DIR>
static cudaError_t march_form(const MarchLaunch &m) {
  const size_t smem = chunk_bytes<NBT>(FMT == kCellXq, m.g.n_tbins);
  return launch_pdl(k_march<NBT, AMR, FMT, DIR>, march_grid<NBT, DIR>(m), dim3(kMarchBlock), smem, m.st,
                    m.g, m.rg, m.src, m.out, m.fp64_level);
}

template <int NBT, bool AMR, int FMT>
static cudaError_t march_any(const MarchLaunch &m) {
  const int moving = (m.rg.Dhi[0] != 0.f) + (m.rg.Dhi[1] != 0.f) + (m.rg.Dhi[2] != 0.f);
  if constexpr (NBT > 1)  // (one band: march_axis_one)
    if (moving == 1) return march_form<NBT, AMR, FMT, -3>(m);
  // (inclined rays with more bands per thread: march_wide)
  if constexpr (NBT <= 8) return m.few ? march_form<NBT, AMR, FMT, -1>(m) : march_form<NBT, AMR, FMT, -2>(m);
  return cudaErrorInvalidValue;
}

// Rays in any direction, NBT bands per thread.
template <int NBT>
cudaError_t march_general(const MarchLaunch &m) {
  const bool amr = m.g.kind == AIR_GRID_AMR;
  if (m.g.cell_fmt == kCellRho) return amr ? march_any<NBT, true, kCellRho>(m) : march_any<NBT, false, kCellRho>(m);
  if (m.g.cell_fmt == kCellXq) return amr ? march_any<NBT, true, kCellXq>(m) : march_any<NBT, false, kCellXq>(m);
  // per-cell Lambda exists for one-band grids only
  if constexpr (NBT == 1) return amr ? march_any<1, true, kCellLam>(m) : march_any<1, false, kCellLam>(m);
  return cudaErrorInvalidValue;
}

// One-band grids, every ray parallel to grid axis A: the form DIR = 1 + A, or
// 4 + A for bricks of 4 or 8 cells, 13 + A for 1 or 2, 7 + A or 10 + A for grids
// of 16^3 bricks with per-cell Lambda, the ordinary one-band grid (constant
// strides would serve 32^3 bricks and several bands too; not tried there).
template <int A, int FMT>
static cudaError_t march_axis_fmt(const MarchLaunch &m) {
  if (m.g.kind != AIR_GRID_AMR) return march_form<1, false, FMT, 1 + A>(m);
  if (m.g.B <= 2) return march_form<1, true, FMT, 13 + A>(m);
  if (m.g.B <= 8) return march_form<1, true, FMT, 4 + A>(m);
  if constexpr (FMT == kCellLam)
    if (m.g.B == 16) return m.rg.Dhi[A] > 0.f ? march_form<1, true, FMT, 7 + A>(m) : march_form<1, true, FMT, 10 + A>(m);
  return march_form<1, true, FMT, 1 + A>(m);
}
template <int A>
cudaError_t march_axis_one(const MarchLaunch &m) {
  if (m.g.cell_fmt == kCellRho) return march_axis_fmt<A, kCellRho>(m);
  if (m.g.cell_fmt == kCellXq) return march_axis_fmt<A, kCellXq>(m);
  return march_axis_fmt<A, kCellLam>(m);
}

}  // namespace air
