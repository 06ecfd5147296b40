// air_march_kernel.cuh -- the march kernel and its launch, as templates over
// the bands one thread carries. Each width is compiled in a translation unit
// of its own (air_march_<width>.cu, air_march_axis.cu), in parallel: one unit
// with every form took 150 s of a build, the slowest of these takes a quarter.
#pragma once
#include "air_march.cuh"
#include "air_refine.cuh"

namespace air {

// One launch of the march, as launch_march resolved it.
struct MarchLaunch {
  const GridView &g;
  const RayGeom &rg;
  const RaySource &src;
  const RayOut &out;
  int64_t blocks;  // of kMarchBlock rays; with the count on the device, unused
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
constexpr int kAxisBlocksSmall = 6;  // bricks of at most 8 cells: two bricks' records in registers

// DIR = -1 has the registers of two or three blocks (see DdaChunk).
template <int NBT, int DIR>
struct MinBlocks {
  static constexpr int value = DIR == -1 ? (NBT <= 4 ? 3 : 2)
                               : DIR == -2 ? (NBT <= 1 ? 6 : (NBT <= 2 ? 5 : (NBT <= 8 ? 4 : 3)))
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
  band_regs<NBT>(br, bc);

  if (src.mode == 2) {
    // new nodes of a sweep counted on the device: block b takes chunk b of
    // blockDim.x rays, and more from a work counter until the rays run out
    SweepSlot &s0 = src.sweep->slot[src.q & 3];
    const int64_t first = s0.n, count = src.sweep->slot[(src.q + 1) & 3].n - first;
    if ((src.part == 1 && count > src.few) || (src.part == 2 && count <= src.few)) return;
    __shared__ long long s_chunk;
    for (int64_t r0 = (int64_t)blockIdx.x * blockDim.x; r0 < count; r0 = s_chunk * blockDim.x) {
      const int64_t r = r0 + threadIdx.x;
      if (r < count) march_one<NBT, AMR, FMT, DIR>(g, rg, src, out, fp64_level, bc, br, chunk, b0,
                                                   nbh, first + r);
      if (count <= (int64_t)gridDim.x * blockDim.x) return;
      __syncthreads();
      if (threadIdx.x == 0) s_chunk = gridDim.x + (long long)atomicAdd(&s0.ray_ctr[chunk], 1ull);
      __syncthreads();
    }
    return;
  }
  const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
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
  // 16 bands per thread leave no registers for the form for few rays
  if constexpr (NBT <= 8)
    if (m.few) return march_form<NBT, AMR, FMT, -1>(m);
  return march_form<NBT, AMR, FMT, -2>(m);
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
// 4 + A for bricks of at most 8 cells, 7 + A or 10 + A for grids of 16^3 bricks
// with per-cell Lambda (the ordinary one-band grid).
template <int A, int FMT>
static cudaError_t march_axis_fmt(const MarchLaunch &m) {
  if (m.g.kind != AIR_GRID_AMR) return march_form<1, false, FMT, 1 + A>(m);
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
