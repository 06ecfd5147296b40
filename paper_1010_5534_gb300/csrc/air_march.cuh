// air_march.cuh -- per-ray march (Parkin 2010, Section 1 and Section 2 step ii):
// follow one ray per pixel through the grid and sum, per crossed cell, the
// column density N = sum rho ds and the emergent intensity of the absorbed
// emission, front to back, I_b = sum_k (j_k/alpha_k)(1 - e^-dtau_k) e^-tau_<k.
//
// One thread marches one ray with a chunk of bands: their sums in registers (up
// to 8 bands, or 16 along an axis), or in shared memory (the wide form, up to 32
// bands of an inclined ray). A warp takes up to 32 neighbouring pixels, so their
// cell fetches fall in the same or adjacent cells.
//
// Traversal: the ray's position is kept as an integer finest-level cell
// coordinate plus a ray parameter t (world length). Inside a block of cells
// (the whole uniform grid, or one AMR brick) an Amanatides-Woo DDA in FP32
// local coordinates yields the exact chord of each cell. AMR bricks are found
// through a dense map over the finest cells (at the finest brick level that
// fits 2^24 entries, with an octree descent below it); a brick is left
// through the face with the smallest exit parameter and the next brick is the
// one holding the finest cell across that face, so no cell is skipped or
// visited twice. A ray along one grid axis crosses every brick whole, and its
// walk (march_amr_axis) carries no ray parameter. Bricks at level >= fp64_level
// compute their entry point and exit parameter in FP64. Coarser bricks compute the entry point in
// double-float (pairs of FP32 with error-free sums and products), since FP64
// issues at a small fraction of the FP32 rate on this GPU. Either way the
// entry point is expressed relative to the entry cell, so FP32 rounding inside
// a brick scales with the distance marched in it.
//
// Accumulation in FP32: N and I_b are Kahan-compensated sums. The absorption
// coefficient is alpha_b = kappa_b rho with kappa_b fixed per band, so the
// optical depth is tau_b = kappa_b N exactly, taken from the compensated N;
// T_b = e^-tau_b = 2^(-kappa_b log2(e) N) is recomputed at every cell with the
// hardware base-2 exponential (ex2.approx: relative error about 2^-22, plus
// the rounding of its argument, |tau| 2^-24 relative), so no error is carried
// from one cell to the next. The cell term is j ds T (1 - e^-dtau)/dtau from
// a Taylor polynomial for dtau < 1/4, and (j/alpha)(T_prev - T_next) above.
#pragma once
#include <cfloat>
#include <cmath>

#include "air_internal.cuh"

namespace air {

template <int NBT>
struct RTState {
  float N, cN;
  float T[NBT], I[NBT], cI[NBT];
  uint32_t steps;
  int maxlev;  // deepest brick level crossed
  // T[] is not that of the current N: cells that emit nothing left it behind.
  // It is then 2^(nk (tN + tp)), formed as fma(nk, tp, nk tN).
  bool stale;
  float tN, tp;
};

// NBT = 0, the wide form of inclined rays: any number of bands per thread (up
// to kWideBands), their sums in shared memory (WideCtx).
template <>
struct RTState<0> {
  float N, cN;
  uint32_t steps;
  int maxlev;
  bool due;  // cells that emit nothing since the last one that emits
};

// Emission table of a band chunk in shared memory (kCellXq): per table bin
// the pairs {Lambda_b, next bin's Lambda_b - Lambda_b} of the chunk's NBT bands
// side by side, so a cell's look-up is one 16-byte load per two bands and one
// fused multiply-add per band. (Before: two 4-byte loads from two places and a
// subtraction per band.) Rows of four and more bands are padded by 16 bytes,
// so that rows of neighbouring bins start in different banks.
template <int NBT>
__host__ __device__ constexpr int tab_row() {  // floats per bin
  return 2 * NBT + (NBT >= 4 ? 4 : 0);
}
template <int NBT>
__host__ __device__ constexpr size_t tab_bytes(int n_tbins) {
  return (sizeof(float) * (size_t)(tab_row<NBT>() * n_tbins) + 15) & ~(size_t)15;
}
// Fill the table of bands [b0, b0 + NBT) (zero beyond n_bands) by one block.
// (Eight entries' loads in flight: a block that goes from chunk to chunk fills
// its table again and again, see batch_tables.)
template <int NBT>
__device__ __forceinline__ void tab_fill(float *tab, const GridView &g, int b0) {
  const int ts = g.n_tbins + 1;
#pragma unroll 8
  for (int x = threadIdx.x; x < NBT * g.n_tbins; x += blockDim.x) {
    const int k = x / NBT, b = x - k * NBT;
    float v = 0.f, d = 0.f;
    if (b0 + b < g.n_bands) {
      v = g.table[(b0 + b) * ts + k];
      d = g.table[(b0 + b) * ts + k + 1] - v;
    }
    tab[k * tab_row<NBT>() + 2 * b] = v;
    tab[k * tab_row<NBT>() + 2 * b + 1] = d;
  }
}

// Shared memory of a band chunk: its table (kCellXq) and its bands' constants.
template <int NBT>
__host__ __device__ constexpr size_t chunk_bytes(bool table, int n_tbins) {
  return (table ? tab_bytes<NBT>(n_tbins) : 0) + sizeof(BandConst) * NBT;
}

struct BandCtx {
  const float *tab;      // shared: the chunk's table (tab_fill)
  const BandConst *band; // shared: the chunk's bands (zero opacity beyond the last)
  int nbh;
};

// The wide form (RTState<0>). A band's T is 2^(nk N) at every point of the ray,
// so its only state is its compensated sum, two words, and only a cell that
// emits needs them. They lie in shared memory, one float4 {I, c, I, c} per pair
// of bands and thread: a thread's registers do not grow with its bands, so one
// walk through the cells serves up to 32 bands, where 8 bands in registers took
// 124 of them and a walk for every 8 bands. A chunk of cells with an emitting
// one (wide_chunk) goes through the bands pair by pair: constants and sums are
// read once, and every cell of the chunk is added to them.
constexpr int kWideBands = 32;
struct WideCtx {
  const float *tab;       // the first pair's table entries (kCellXq), rows of `row` floats
  const BandConst *band;  // the first band's constants
  float4 *sums;           // [pairs][blockDim.x], this thread's column
  int row, pairs;
  int nbh;                // bands; an odd one's partner has zero opacity and table
};
// Floats per table bin: 4 modulo 8, so that rows of neighbouring bins start in
// different banks.
__host__ __device__ constexpr int wide_row(int width) { return (2 * width + 7) / 8 * 8 + 4; }
// Table and constants of `width` (even) bands, and the sums of a block.
__host__ __device__ constexpr size_t wide_tab_bytes(bool table, int n_tbins, int width) {
  return (table ? sizeof(float) * (size_t)wide_row(width) * n_tbins : 0) + sizeof(BandConst) * width;
}
__host__ __device__ constexpr size_t wide_sum_bytes(int width, int threads) {
  return sizeof(float4) * (size_t)(width / 2) * threads;
}
// Fill table and constants of bands [b0, b0 + width) at `sm` by one block (zero
// beyond n_bands).
template <int FMT>
__device__ __forceinline__ void wide_fill(unsigned char *sm, const GridView &g, int b0, int width) {
  BandConst *band = reinterpret_cast<BandConst *>(sm);
  for (int b = threadIdx.x; b < width; b += blockDim.x)
    band[b] = b0 + b < g.n_bands ? g.bands[b0 + b] : BandConst{0.f, 0.f, -0.f, 0xffffffffu};
  if (FMT == kCellXq) {
    float *tab = reinterpret_cast<float *>(band + width);
    const int ts = g.n_tbins + 1, row = wide_row(width);
#pragma unroll 8
    for (int x = threadIdx.x; x < width * g.n_tbins; x += blockDim.x) {
      const int k = x / width, b = x - k * width;
      float v = 0.f, d = 0.f;
      if (b0 + b < g.n_bands) {
        v = g.table[(b0 + b) * ts + k];
        d = g.table[(b0 + b) * ts + k + 1] - v;
      }
      *reinterpret_cast<float2 *>(tab + k * row + 2 * b) = make_float2(v, d);
    }
  }
}
// Part `part` of `parts` of the chunk at `sm` (nb of its `width` bands exist);
// *first: its first band within the chunk. parts <= the chunk's pairs.
template <int FMT>
__device__ __forceinline__ WideCtx wide_ctx(unsigned char *sm, float4 *sums, int width, int nb, int part,
                                            int parts, int *first) {
  const int pairs = (nb + 1) / 2, per = (pairs + parts - 1) / parts;
  const int q0 = min(part * per, pairs);
  WideCtx c;
  c.band = reinterpret_cast<const BandConst *>(sm) + 2 * q0;
  c.tab = reinterpret_cast<const float *>(sm + sizeof(BandConst) * width) + 4 * q0;
  c.sums = sums + threadIdx.x;
  c.row = wide_row(width);
  c.pairs = min(per, pairs - q0);
  c.nbh = min(2 * c.pairs, nb - 2 * q0);
  *first = 2 * q0;
  return c;
}
// Parts that a chunk's bands are dealt to for `rays` rays, so that the rays'
// parts are at least about `fill` threads: a walk of its own for each part, but
// a launch that leaves the GPU idle takes as long as its longest ray.
__host__ __device__ __forceinline__ int wide_parts(int64_t rays, int nb, int64_t fill) {
  int parts = 1;
  while (2 * parts <= (nb + 1) / 2 && 2 * parts * rays <= fill) parts *= 2;
  return parts;
}

// Bands of a chunk of the wide form: all of them, or as equal parts as let the
// shared memory of four blocks fit an SM (and kWideBands).
static inline int wide_width(const GridView &g, int threads) {
  int chunks = (g.n_bands + kWideBands - 1) / kWideBands;
  for (;; ++chunks) {
    const int width = ((g.n_bands + chunks - 1) / chunks + 1) & ~1;
    const size_t b = wide_tab_bytes(g.cell_fmt == kCellXq, g.n_tbins, width) + wide_sum_bytes(width, threads);
    if (b <= 54 * 1024 || width <= 8) return width;
  }
}

// Rays that a warp takes at a time, of `rays` inclined rays in `chunks` chunks
// or parts, for `warps` warps at work at once. The lanes of a warp meet brick
// faces and emitting cells at different steps, so a warp of 32 rays issues a
// multiple of one ray's instructions (of 32 lanes 7 to 14 are active); a launch
// of few rays spreads them over the idle warps. (The march of the inclined cone
// above 3.65 -> 3.40 ms, 8 views x 16 bands 12.34 -> 11.92. Rays along an axis
// share their steps and their cache lines: 126 -> 158 us, so they stay together.)
__host__ __device__ __forceinline__ int rays_per_warp(int64_t rays, int chunks, int64_t warps) {
  int rpw = 32;
  while (rpw > 1 && rays * chunks <= warps * (rpw / 2)) rpw >>= 1;
  return rpw;
}

// Fill a chunk's shared memory at `sm` by one block.
template <int NBT, int FMT>
__device__ __forceinline__ void chunk_fill(unsigned char *sm, const GridView &g, int b0) {
  if (FMT == kCellXq) tab_fill<NBT>(reinterpret_cast<float *>(sm), g, b0);
  BandConst *band = reinterpret_cast<BandConst *>(sm + (FMT == kCellXq ? tab_bytes<NBT>(g.n_tbins) : 0));
  for (int b = threadIdx.x; b < NBT; b += blockDim.x)
    band[b] = b0 + b < g.n_bands ? g.bands[b0 + b] : BandConst{0.f, 0.f, -0.f, 0xffffffffu};
}
template <int NBT, int FMT>
__device__ __forceinline__ BandCtx chunk_ctx(const unsigned char *sm, const GridView &g, int nbh) {
  BandCtx bc;
  bc.tab = reinterpret_cast<const float *>(sm);
  bc.band = reinterpret_cast<const BandConst *>(sm + (FMT == kCellXq ? tab_bytes<NBT>(g.n_tbins) : 0));
  bc.nbh = nbh;
  return bc;
}

// Per-band constants in registers. One band keeps them for the whole ray; with
// more, the column march of axis rays does (band_load), and so does every ray of
// a grid whose emission has no table (kCellRho): there a band's arithmetic is so
// short that a load per band and cell shows (400^2 inclined pixels, 5 bands: 537 us
// with the constants in shared memory, 455 in registers). With a table the cells of inclined rays read their band's constants
// from shared memory (one 16-byte load that every lane shares, against 24
// registers at 8 bands).
template <int NBT, int FMT>
constexpr bool kRegConst = NBT == 1 || (NBT > 1 && FMT == kCellRho);
template <int NBT>
struct BandRegs {
  float kap[NBT];  // kappa_b
  float ik[NBT];   // 1 / kappa_b (0 where kappa_b = 0)
  float nk[NBT];   // -kappa_b log2(e): T_b = 2^(nk_b N)
  float kmax;      // largest kappa_b of the chunk
  uint32_t xz;     // table coordinates below xz emit nothing in any band (kCellXq)
};

template <>
struct BandRegs<0> {
  uint32_t xz;
};

template <int NBT>
__device__ __forceinline__ BandConst band_const(const BandCtx &bc, int b) {
  const float4 c = *reinterpret_cast<const float4 *>(bc.band + b);
  return BandConst{c.x, c.y, c.z, __float_as_uint(c.w)};
}
template <int NBT>
__device__ __forceinline__ void band_load(BandRegs<NBT> &br, const BandCtx &bc) {
  br.kmax = 0.f;
#pragma unroll
  for (int b = 0; b < NBT; ++b) {
    const BandConst c = band_const<NBT>(bc, b);
    br.kap[b] = c.kap;
    br.ik[b] = c.ik;
    br.nk[b] = c.nk;
    br.kmax = fmaxf(br.kmax, c.kap);
  }
}
// What a ray starts with: xz, and the constants that stay in registers.
template <int NBT, int FMT>
__device__ __forceinline__ void band_regs(BandRegs<NBT> &br, const BandCtx &bc) {
  br.xz = 0xffffffffu;
#pragma unroll
  for (int b = 0; b < NBT; ++b) br.xz = min(br.xz, bc.band[b].xz);
  if (kRegConst<NBT, FMT>) band_load<NBT>(br, bc);
}

// Whether a cell emits nothing in any band of the chunk, from its auxiliary
// word: rho Lambda = 0 (kCellLam), or a table coordinate below which every
// band's table is zero (kCellXq). Cool gas has no X-ray emission, and most of
// a grid's volume is cool. Such a cell adds zero to every I_b and only its
// rho ds to N, so the march leaves the band arithmetic out where the sums'
// bits allow it (rt_term, march_column).
template <int FMT>
__device__ __forceinline__ bool cell_dark(uint32_t aux, uint32_t xz) {
  return FMT == kCellLam ? aux == 0u : (FMT == kCellXq ? aux < xz : false);
}

// 2^x by the hardware approximation (PTX ex2.approx.ftz.f32).
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// The wide form's start: sums of zero.
__device__ __forceinline__ void wide_init(RTState<0> &r, const WideCtx &wc) {
  r.N = 0.f;
  r.cN = 0.f;
  r.steps = 0;
  r.maxlev = 0;
  r.due = false;
  for (int q = 0; q < wc.pairs; ++q) wc.sums[q * blockDim.x] = make_float4(0.f, 0.f, 0.f, 0.f);
}

template <int NBT>
__device__ __forceinline__ void rt_init(RTState<NBT> &r) {
  r.N = 0.f;
  r.cN = 0.f;
  r.steps = 0;
  r.maxlev = 0;
  r.stale = false;
  r.tN = 0.f;
  r.tp = 0.f;
#pragma unroll
  for (int b = 0; b < NBT; ++b) {
    r.T[b] = 1.f;
    r.I[b] = 0.f;
    r.cI[b] = 0.f;
  }
}

// T[] brought up to the current N after cells that emit nothing.
template <int NBT>
__device__ __forceinline__ void rt_refresh(RTState<NBT> &r, const BandCtx &bc) {
#pragma unroll
  for (int b = 0; b < NBT; ++b) {
    const float nk = bc.band[b].nk;
    r.T[b] = ex2_approx(fmaf(nk, r.tp, __fmul_rn(nk, r.tN)));
  }
  r.stale = false;
}

// After dark cells up to N = tN + tp.
template <int NBT>
__device__ __forceinline__ void rt_dark(RTState<NBT> &r, float tN, float tp) {
  if (!r.stale) {
#pragma unroll
    for (int b = 0; b < NBT; ++b) kahan_add(r.I[b], r.cI[b], 0.f);
    r.stale = true;
  }
  r.tN = tN;
  r.tp = tp;
}

// Lambda of bands 2 q and 2 q + 1 at table row `row` (tab_fill) and weight w.
template <int NBT>
__device__ __forceinline__ void tab_pair(const float *row, int q, float w, float &l0, float &l1) {
  if (NBT == 1) {
    const float2 t = *reinterpret_cast<const float2 *>(row);
    l0 = fmaf(w, t.y, t.x);
  } else {
    const float4 t = *reinterpret_cast<const float4 *>(row + 4 * q);
    l0 = fmaf(w, t.y, t.x);
    l1 = fmaf(w, t.w, t.z);
  }
}

// Transfer step of one cell chord of length ds: density rho, and aux =
// rho Lambda (kCellLam, as float bits) or the table coordinate of T (kCellXq).
// With dtau = 0 (kappa_b = 0 or rho = 0) the series form gives the optically
// thin term j ds T exactly, so no separate case is needed.
// Both forms of the cell term are evaluated and the one for the cell's dtau
// is selected, which keeps the band loop free of divergent branches.
//
// A cell that emits nothing (cell_dark) leaves I_b and T_b out. Adding its
// zero term can change a compensated sum once (it moves a residue that is
// not yet below half an ulp into the sum) and never again, so the zero is
// added at the first dark cell after an emitting one and skipped at the rest;
// T_b is formed at the next emitting cell from N, as it would have been. (One
// band: the zero is added and T formed each time, six operations.)
// Where N overflows, every cell takes the full path. All bits are those of
// the full path.
//
// The products that feed the compensated sums (rho ds, and each form's final
// product) are rounded explicitly (__fmul_rn), so the compiler cannot fuse
// them into the sums' subtractions: every instantiation (band chunking, form)
// rounds alike and gives the same bits.

// The band terms of a cell that brought the column density to N.
template <int NBT, int FMT>
__device__ __forceinline__ void rt_bands(RTState<NBT> &r, float rho, uint32_t aux, float rds, float N,
                                         const BandCtx &bc, const BandRegs<NBT> &br) {
  if (FMT != kCellRho && NBT > 1 && r.stale) rt_refresh<NBT>(r, bc);
  float w = 0.f;
  const float *row = bc.tab;
  if (FMT == kCellXq) {
    row += (int)(aux >> kXqFracBits) * tab_row<NBT>();
    w = (float)(aux & ((1u << kXqFracBits) - 1u)) * (1.0f / (float)(1u << kXqFracBits));
  }
#pragma unroll
  for (int q = 0; q < (NBT + 1) / 2; ++q) {
    if (NBT <= 2 || 2 * q < bc.nbh) {
      float lam[2] = {1.f, 1.f};
      if (FMT == kCellXq) tab_pair<NBT>(row, q, w, lam[0], lam[1]);
#pragma unroll
      for (int e = 0; e < (NBT == 1 ? 1 : 2); ++e) {
        const int b = 2 * q + e;
        const BandConst c = kRegConst<NBT, FMT> ? BandConst{br.kap[b], br.ik[b], br.nk[b], 0u} : band_const<NBT>(bc, b);
        const float dtau = c.kap * rds;
        const float Tn = ex2_approx(c.nk * N);
        // rho Lambda_b
        const float rl = FMT == kCellLam ? __uint_as_float(aux) : (FMT == kCellXq ? rho * lam[e] : rho);
        const float t_small = __fmul_rn(rl * rds, r.T[b] * one_minus_exp_over_x(dtau));
        const float t_large = __fmul_rn(rl * c.ik, r.T[b] - Tn);
        const float term = dtau < 0.25f ? t_small : t_large;
        r.T[b] = Tn;
        kahan_add(r.I[b], r.cI[b], term);
      }
    }
  }
}

// The band terms of dark cells up to column density N.
template <int NBT>
__device__ __forceinline__ void rt_dark_to(RTState<NBT> &r, float N, const BandRegs<NBT> &br) {
  if (NBT == 1) {
    kahan_add(r.I[0], r.cI[0], 0.f);
    r.T[0] = ex2_approx(br.nk[0] * N);
  } else {
    rt_dark<NBT>(r, N, 0.f);
  }
}

// The band terms of a chunk of K cells in the wide form (cell u lies on the ray
// where in[u]): the operations of rt_bands and rt_dark in their order, for one
// pair of bands after the other. N0: the column density before the chunk.
template <int FMT, int K>
__device__ __forceinline__ void wide_chunk(RTState<0> &r, const bool (&in)[K], const float (&rh)[K],
                                           const uint32_t (&xv)[K], const float (&rds)[K],
                                           const float (&N)[K], float N0, const WideCtx &wc, uint32_t xz) {
  uint32_t emits = 0u, zero = 0u;  // cells that emit; those with dark cells before them
#pragma unroll
  for (int u = 0; u < K; ++u)
    if (in[u]) {
      if (cell_dark<FMT>(xv[u], xz) && N[u] <= FLT_MAX) {
        r.due = true;
      } else {
        emits |= 1u << u;
        if (r.due) zero |= 1u << u;
        r.due = false;
      }
    }
  if (!emits) return;
  const bool start = N0 == 0.f;  // T = 1, whatever the opacity
  int row[K];
  float w[K];
#pragma unroll
  for (int u = 0; u < K; ++u) {
    row[u] = FMT == kCellXq ? (int)(xv[u] >> kXqFracBits) * wc.row : 0;
    w[u] = FMT == kCellXq ? (float)(xv[u] & ((1u << kXqFracBits) - 1u)) * (1.0f / (float)(1u << kXqFracBits)) : 0.f;
  }
#pragma unroll 1
  for (int q = 0; q < wc.pairs; ++q) {
    const float4 ca = *reinterpret_cast<const float4 *>(wc.band + 2 * q);
    const float4 cb = *reinterpret_cast<const float4 *>(wc.band + 2 * q + 1);
    float4 s = wc.sums[q * blockDim.x];
    float T0 = start ? 1.f : ex2_approx(ca.z * N0);
    float T1 = start ? 1.f : ex2_approx(cb.z * N0);
#pragma unroll
    for (int u = 0; u < K; ++u) {
      const float Tn0 = ex2_approx(ca.z * N[u]);
      const float Tn1 = ex2_approx(cb.z * N[u]);
      if (emits >> u & 1u) {
        if (zero >> u & 1u) {
          kahan_add(s.x, s.y, 0.f);
          kahan_add(s.z, s.w, 0.f);
        }
        float rl0 = rh[u], rl1 = rh[u];  // rho Lambda_b
        if (FMT == kCellXq) {
          const float4 t = *reinterpret_cast<const float4 *>(wc.tab + row[u] + 4 * q);
          rl0 *= fmaf(w[u], t.y, t.x);
          rl1 *= fmaf(w[u], t.w, t.z);
        }
        const float d0 = ca.x * rds[u], d1 = cb.x * rds[u];  // dtau
        const float small0 = __fmul_rn(rl0 * rds[u], T0 * one_minus_exp_over_x(d0));
        const float small1 = __fmul_rn(rl1 * rds[u], T1 * one_minus_exp_over_x(d1));
        const float large0 = __fmul_rn(rl0 * ca.y, T0 - Tn0);
        const float large1 = __fmul_rn(rl1 * cb.y, T1 - Tn1);
        kahan_add(s.x, s.y, d0 < 0.25f ? small0 : large0);
        kahan_add(s.z, s.w, d1 < 0.25f ? small1 : large1);
      }
      T0 = Tn0;
      T1 = Tn1;
    }
    wc.sums[q * blockDim.x] = s;
  }
}

// DARK = false: without the test (for callers that have made it).
template <int NBT, int FMT, bool DARK = true>
__device__ __forceinline__ void rt_term(RTState<NBT> &r, float rho, uint32_t aux, float ds,
                                        const BandCtx &bc, const BandRegs<NBT> &br) {
  const float rds = __fmul_rn(rho, ds);
  kahan_add(r.N, r.cN, rds);
  if (DARK && cell_dark<FMT>(aux, br.xz) && r.N <= FLT_MAX) rt_dark_to<NBT>(r, r.N, br);
  else rt_bands<NBT, FMT>(r, rho, aux, rds, r.N, bc, br);
}

// Cells that the DDA steps through, and requests, before it sums the first of
// them (march_block). DIR = -1, the form for launches that leave most of the
// GPU's threads idle, goes further ahead: there a ray's time is its number of
// chunks times the L2's latency (800 cycles), and registers are free.
constexpr int kWideAhead = 4;  // (8: batched 16 bands 13.5 -> 14.4 ms)
template <int NBT, int DIR>
struct DdaChunk {
  static constexpr int value = NBT == 0 ? kWideAhead : DIR != -1 ? 4 : (NBT <= 2 ? 16 : 8);
};

// Fields of cell idx: rho and the auxiliary word of the format.
template <int FMT, typename Idx>
__device__ __forceinline__ void load_cell(const void *__restrict__ cells, Idx idx, float &rho,
                                          uint32_t &aux) {
  if (FMT == kCellRho) {
    rho = __ldg((const float *)cells + idx);
    aux = 0u;
  } else {
    const uint2 c = __ldg((const uint2 *)cells + idx);
    rho = __uint_as_float(c.x);
    aux = c.y;
  }
}

// (1 - e^-x) / x for 0 <= x < 1/64 from its Taylor series truncated after
// x^3 (remainder < x^4 / 5! < 5e-10).
__device__ __forceinline__ float one_minus_exp_over_x_short(float x) {
  float g = -1.0f / 24.0f;
  g = fmaf(g, x, 1.0f / 6.0f);
  g = fmaf(g, x, -0.5f);
  g = fmaf(g, x, 1.0f);
  return g;
}

// The transfer steps of a group of U column cells, all with chord ds. Inside
// the group the column density and the band intensities are summed in plain
// FP32 (partial sums from zero, the cell terms added with one fused
// multiply-add each), and the group's partial sums are added to the running
// sums with Kahan compensation; the error of a plain sum of U = 16 positive
// terms is at most 15 u of the group's sum (u = 2^-24), so the column's sums
// stay within about 16 u of exact. T_b at each cell is 2^(nk_b N_k) with N_k
// the running column density plus the group's partial sum, its exponent
// formed as fma(nk_b, partial, nk_b N_start).
// FORM 3: every dtau of the group below 2^-12: (1 - e^-x) / x taken to first
// order, 1 - x / 2 (remainder < x^2 / 6 < 1e-8), as T + (-kappa_b / 2 T)(rho
// ds); used for one-band grids with per-cell Lambda, the format whose
// instantiations are few enough to afford another form;
// FORM 2: below 1/64 (the short series); FORM 1: below 1/4 (the full series);
// FORM 0: the form is selected per cell and band.
// rh: the cells' rho, or their rho ds already formed (kCellLam).
template <int NBT, int FMT, int FORM, int U>
__device__ __forceinline__ void column_group(RTState<NBT> &r, const float (&rh)[U],
                                             const uint32_t (&xv)[U], float ds, const BandCtx &bc,
                                             const BandRegs<NBT> &br) {
  float pN = 0.f, pI[NBT], nN0[NBT], hk[NBT];
  const float N0 = r.N;
#pragma unroll
  for (int b = 0; b < NBT; ++b) {
    pI[b] = 0.f;
    nN0[b] = __fmul_rn(br.nk[b], N0);  // log2 T_b at the group's start
    hk[b] = -0.5f * br.kap[b];         // exact: a power-of-two scaling
  }
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const float rho = rh[u];
    const float rds = FMT == kCellLam ? rho : __fmul_rn(rho, ds);
    pN = __fadd_rn(pN, rds);
    float w = 0.f;
    const float *row = bc.tab;
    if (FMT == kCellXq) {
      row += (int)(xv[u] >> kXqFracBits) * tab_row<NBT>();
      w = (float)(xv[u] & ((1u << kXqFracBits) - 1u)) * (1.0f / (float)(1u << kXqFracBits));
    }
    float lam[2] = {1.f, 1.f};
#pragma unroll
    for (int b = 0; b < NBT; ++b) {
      if (NBT <= 2 || (b & ~1) < bc.nbh) {
        if (FMT == kCellXq && (b & 1) == 0) tab_pair<NBT>(row, b >> 1, w, lam[0], lam[1]);
        const float Tn = ex2_approx(fmaf(br.nk[b], pN, nN0[b]));
        // rho Lambda_b
        const float rl = FMT == kCellLam ? __uint_as_float(xv[u]) : __fmul_rn(rho, lam[b & 1]);
        float P, Q;
        if (FORM == 3) {
          // T (1 - dtau / 2) with dtau = kappa_b (rho ds)
          P = __fmul_rn(rl, rds);
          Q = fmaf(__fmul_rn(hk[b], r.T[b]), rds, r.T[b]);
        } else if (FORM == 2) {
          const float dtau = __fmul_rn(br.kap[b], rds);
          P = __fmul_rn(rl, rds);
          Q = __fmul_rn(r.T[b], one_minus_exp_over_x_short(dtau));
        } else {
          const float dtau = __fmul_rn(br.kap[b], rds);
          const float Ps = __fmul_rn(rl, rds);
          const float Qs = __fmul_rn(r.T[b], one_minus_exp_over_x(dtau));
          if (FORM == 1) {
            P = Ps;
            Q = Qs;
          } else {
            const bool small = dtau < 0.25f;
            P = small ? Ps : __fmul_rn(rl, br.ik[b]);
            Q = small ? Qs : __fsub_rn(r.T[b], Tn);
          }
        }
        pI[b] = fmaf(P, Q, pI[b]);
        r.T[b] = Tn;
      }
    }
  }
  kahan_add(r.N, r.cN, pN);
#pragma unroll
  for (int b = 0; b < NBT; ++b)
    if (NBT <= 2 || (b & ~1) < bc.nbh) kahan_add(r.I[b], r.cI[b], pI[b]);
}

// A group whose cells all emit nothing: N alone, summed as column_group sums
// it; its zero partial sums change I_b as theirs do (once after an emitting
// group or cell, see rt_term), and T_b waits for the next emitting group.
// False where N overflows: the caller then takes the full path.
template <int NBT, int FMT, int U>
__device__ __forceinline__ bool column_group_dark(RTState<NBT> &r, const float (&rh)[U], float ds,
                                                  const BandRegs<NBT> &br) {
  float pN = 0.f;
#pragma unroll
  for (int u = 0; u < U; ++u) pN = __fadd_rn(pN, FMT == kCellLam ? rh[u] : __fmul_rn(rh[u], ds));
  // N + pN plus the compensation is finite if twice the larger sum is
  if (!(r.N + pN <= 0.5f * FLT_MAX)) return false;
  if (NBT == 1) {
    kahan_add(r.I[0], r.cI[0], 0.f);
    r.T[0] = ex2_approx(fmaf(br.nk[0], pN, __fmul_rn(br.nk[0], r.N)));
  } else {
    rt_dark<NBT>(r, r.N, pN);
  }
  kahan_add(r.N, r.cN, pN);
  return true;
}

// Largest of U non-negative floats (their bits compare as integers; three
// operands per instruction).
template <int U>
__device__ __forceinline__ float max_of(const float (&v)[U]) {
  int m = __float_as_int(v[0]);
#pragma unroll
  for (int u = 1; u + 1 < U; u += 2) m = __vimax3_s32(m, __float_as_int(v[u]), __float_as_int(v[u + 1]));
  if (U % 2 == 0) m = max(m, __float_as_int(v[U - 1]));
  return __int_as_float(m);
}

// One group of U column cells, fetched into rh and xv: the dark path, or the
// transfer form chosen from kmax (rho_max ds) for the group's largest rho,
// which bounds every cell's dtau = kappa_b (rho ds) (FP32 rounding is
// monotonic).
template <int NBT, int FMT, int U>
__device__ __forceinline__ void column_cells(RTState<NBT> &r, float (&rh)[U],
                                             const uint32_t (&xv)[U], float ds, const BandCtx &bc,
                                             const BandRegs<NBT> &br) {
  if (FMT == kCellLam) {
    // only rho ds is used from here on (the record holds rho Lambda)
#pragma unroll
    for (int u = 0; u < U; ++u) rh[u] = __fmul_rn(rh[u], ds);
  }
  if (FMT != kCellRho) {
    uint32_t x = xv[0];
#pragma unroll
    for (int u = 1; u < U; ++u) x = FMT == kCellLam ? x | xv[u] : max(x, xv[u]);
    if (cell_dark<FMT>(x, br.xz) && column_group_dark<NBT, FMT, U>(r, rh, ds, br)) return;
    if (NBT > 1 && r.stale) rt_refresh<NBT>(r, bc);
  }
  const float m = max_of<U>(rh);
  const float dmax = br.kmax * (FMT == kCellLam ? m : __fmul_rn(m, ds));
  if (FMT == kCellLam && dmax < 0x1p-12f) column_group<NBT, FMT, 3, U>(r, rh, xv, ds, bc, br);
  else if (dmax < 0.015625f) column_group<NBT, FMT, 2, U>(r, rh, xv, ds, bc, br);
  else if (dmax < 0.25f) column_group<NBT, FMT, 1, U>(r, rh, xv, ds, bc, br);
  else column_group<NBT, FMT, 0, U>(r, rh, xv, ds, bc, br);
}

// n cells of one column (cell idx, idx + d, ...), every one crossed whole
// with the same chord ds: the path of a ray parallel to a grid axis, which
// enters each block of cells through a face and leaves through the opposite
// one. No DDA is needed. Cells are fetched U at a time (U loads in flight per
// thread) and summed as a group (column_cells).
// TAIL = false: n is known to be a multiple of U.
template <int NBT, int FMT, int U, bool TAIL, typename Idx>
__device__ __forceinline__ void march_column(RTState<NBT> &r, const void *__restrict__ cells, Idx idx,
                                             Idx d, int n, float ds, const BandCtx &bc,
                                             const BandRegs<NBT> &br) {
  r.steps += (uint32_t)n;
  int k = 0;
  for (; k + U <= n; k += U) {
    float rh[U];
    uint32_t xv[U];
#pragma unroll
    for (int u = 0; u < U; ++u) load_cell<FMT>(cells, idx + (Idx)u * d, rh[u], xv[u]);
    idx += (Idx)U * d;
    column_cells<NBT, FMT, U>(r, rh, xv, ds, bc, br);
  }
  // the rest (all of a brick of fewer than U cells) one by one, fetched 4 at
  // a time (8 at a time spilled 240 bytes in the one-axis kernels)
  for (; TAIL && k < n; k += 4) {
    float rh[4];
    uint32_t xv[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (k + u < n) load_cell<FMT>(cells, idx + (Idx)u * d, rh[u], xv[u]);
    idx += (Idx)4 * d;
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (k + u < n) rt_term<NBT, FMT>(r, rh[u], xv[u], ds, bc, br);
  }
}

// The column of a 16^3 brick along axis A (16 cells, one group), at cells =
// its lowest cell: strides are constants here, so the 16 loads need no address
// arithmetic, and along x a load takes two records. Integer instructions issue
// at half the rate of FP32 ones on this GPU and bound the general form (78% of
// their peak; 48 of a group's 260 instructions formed addresses).
template <int NBT, int FMT, int A, bool POS>
__device__ __forceinline__ void march_column16(RTState<NBT> &r, const void *__restrict__ cells,
                                               float ds, const BandCtx &bc, const BandRegs<NBT> &br) {
  constexpr int st = A == 0 ? 1 : (A == 1 ? 16 : 256);
  float rh[16];
  uint32_t xv[16];
  r.steps += 16u;
  if (A == 0 && FMT != kCellRho) {
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const uint4 c = __ldg((const uint4 *)cells + u);
      const int p = POS ? 2 * u : 15 - 2 * u, q = POS ? 2 * u + 1 : 14 - 2 * u;
      rh[p] = __uint_as_float(c.x);
      xv[p] = c.y;
      rh[q] = __uint_as_float(c.z);
      xv[q] = c.w;
    }
  } else {
#pragma unroll
    for (int u = 0; u < 16; ++u) load_cell<FMT>(cells, (POS ? u : 15 - u) * st, rh[u], xv[u]);
  }
  column_cells<NBT, FMT, 16>(r, rh, xv, ds, bc, br);
}

// Cells fetched per group in the column march: 16 in the compiled one-axis
// form (8 blocks per SM), 8 where the column march runs inside a general
// kernel (oblique-capable single-view and batched kernels, more registers
// taken by the 3-axis DDA).
template <int DIR>
struct ColumnUnroll {
  static constexpr int value = 16;
};

// DDA through a block of nx x ny x nz cells, entered in cell (lx, ly, lz),
// for a ray that moves along two or three grid axes (a ray along one axis
// takes march_column). Q: entry point relative to the low corner of the
// entry cell (in cells), Dl: direction (cells per unit t), inv = 1 / Dl (0
// where Dl = 0), tend: block exit relative to the entry. cells points at the
// block's cell (0, 0, 0); cell (x, y, z) is record z*sz + y*sy + x.
//
// After k steps along axis a the next face of that axis is crossed at
// t = (k + [Dl > 0] - Q) / Dl = k |inv| + q, evaluated as one fused
// multiply-add from the exact float count k, so the rounding of a boundary
// parameter does not grow with the number of cells marched. Parameters are
// measured from the entry cell, so their FP32 rounding scales with the
// distance marched inside the block, not with the ray's distance from the
// origin.
//
// Which cells a ray crosses does not depend on their fields, so the walk runs
// K cells ahead of the sums: it steps through a chunk of cells, asking
// for each record as its index is known, and only then sums the chunk. One
// load latency is paid per chunk instead of one per cell, and the step's own
// dependent operations overlap the loads.
template <int NBT, int FMT, int K, typename Idx, class Ctx>
__device__ __forceinline__ void march_block(RTState<NBT> &r, const float Q[3], const float Dl[3],
                                            const float inv[3], float tend, int lx, int ly, int lz,
                                            int nx, int ny, int nz, Idx sy, Idx sz,
                                            const void *__restrict__ cells, const Ctx &bc,
                                            const BandRegs<NBT> &br) {
  const float INF = FLT_MAX;
  const bool p0 = Dl[0] > 0.f, p1 = Dl[1] > 0.f, p2 = Dl[2] > 0.f;
  const float a0 = fabsf(inv[0]), a1 = fabsf(inv[1]), a2 = fabsf(inv[2]);
  const float q0 = Dl[0] != 0.f ? ((p0 ? 1.f : 0.f) - Q[0]) * inv[0] : INF;
  const float q1 = Dl[1] != 0.f ? ((p1 ? 1.f : 0.f) - Q[1]) * inv[1] : INF;
  const float q2 = Dl[2] != 0.f ? ((p2 ? 1.f : 0.f) - Q[2]) * inv[2] : INF;
  // last step count that stays inside the block, per axis
  const float km0 = (float)(p0 ? nx - 1 - lx : lx);
  const float km1 = (float)(p1 ? ny - 1 - ly : ly);
  const float km2 = (float)(p2 ? nz - 1 - lz : lz);
  const Idx d0 = p0 ? (Idx)1 : (Idx)-1, d1 = p1 ? sy : -sy, d2 = p2 ? sz : -sz;
  float k0 = 0.f, k1 = 0.f, k2 = 0.f;
  float tm0 = q0, tm1 = q1, tm2 = q2;
  Idx idx = (Idx)lz * sz + (Idx)ly * sy + (Idx)lx;
  float tl = 0.f;
  bool more = true;
  do {
    float ds[K], rh[K];
    uint32_t xv[K];
    bool in[K];  // cell u of the chunk lies in the block
#pragma unroll
    for (int u = 0; u < K; ++u) {
      in[u] = more;
      if (more) load_cell<FMT>(cells, idx, rh[u], xv[u]);
      const float tmin = fminf(fminf(tm0, tm1), tm2);
      const float tn = fminf(tmin, tend);
      ds[u] = fmaxf(tn - tl, 0.f);
      tl = tn;
      // step the axis whose face comes first; an axis that is not stepped
      // keeps its count and so its boundary parameter
      if (tm0 == tmin) {
        k0 += 1.f;
        tm0 = fmaf(k0, a0, q0);
        idx += d0;
      } else if (tm1 == tmin) {
        k1 += 1.f;
        tm1 = fmaf(k1, a1, q1);
        idx += d1;
      } else {
        k2 += 1.f;
        tm2 = fmaf(k2, a2, q2);
        idx += d2;
      }
      more = more && tmin < tend && k0 <= km0 && k1 <= km1 && k2 <= km2;
    }
    // the chunk's column density, and whether any of its cells emits. A
    // zero-length chord (a ray grazing an edge or corner) adds nothing and is
    // not counted as a step.
    float N[K];
    const float N0 = r.N;
    uint32_t x = 0u;
#pragma unroll
    for (int u = 0; u < K; ++u) {
      N[u] = r.N;
      if (in[u]) {
        r.steps += ds[u] > 0.f ? 1u : 0u;
        ds[u] = __fmul_rn(rh[u], ds[u]);  // rho ds from here on
        kahan_add(r.N, r.cN, ds[u]);
        N[u] = r.N;
        x = FMT == kCellLam ? x | xv[u] : max(x, xv[u]);
      }
    }
    if constexpr (NBT == 0) {
      if (cell_dark<FMT>(x, br.xz) && r.N <= FLT_MAX) r.due = true;
      else wide_chunk<FMT, K>(r, in, rh, xv, ds, N, N0, bc, br.xz);
    } else if (cell_dark<FMT>(x, br.xz) && r.N <= FLT_MAX) {
      rt_dark_to<NBT>(r, r.N, br);
    } else {
#pragma unroll
      for (int u = 0; u < K; ++u)
        if (in[u]) {
          if (NBT > 1 && cell_dark<FMT>(xv[u], br.xz) && N[u] <= FLT_MAX) rt_dark_to<NBT>(r, N[u], br);
          else rt_bands<NBT, FMT>(r, rh[u], xv[u], ds[u], N[u], bc, br);
        }
    }
  } while (more);  // until the block is left (through its far face, or by rounding)
}

// march_block for a block of one cell, at `cells`, one band: a brick of one cell
// has no walk, and a chunk's other steps are wasted (three inclined views, batched:
// 1170 us, 972 without them).
template <int FMT>
__device__ __forceinline__ void march_cell(RTState<1> &r, const float Q[3], const float Dl[3], const float inv[3],
                                           float tend, const void *__restrict__ cells, const BandCtx &bc,
                                           const BandRegs<1> &br) {
  float rho;
  uint32_t aux;
  load_cell<FMT>(cells, 0, rho, aux);
  float tn = fminf(tend, FLT_MAX);
#pragma unroll
  for (int a = 0; a < 3; ++a)
    if (Dl[a] != 0.f) tn = fminf(tn, ((Dl[a] > 0.f ? 1.f : 0.f) - Q[a]) * inv[a]);
  const float ds = fmaxf(tn, 0.f);
  r.steps += ds > 0.f ? 1u : 0u;
  rt_term<1, FMT>(r, rho, aux, ds, bc, br);
}

// Per-launch ray geometry, resolved on the host in FP64: the pixel centre
// (uc, vc) is the world point C + uc u + vc v (C = image centre - grid origin),
// its grid coordinate (finest-cell units) that point divided by the cell size
// h; rays travel along D = d / h (cells per unit t).
struct RayGeom {
  double C[3], U[3], V[3], h[3], invh[3], D[3], invD[3];
  double H, pix0;  // image half-extent, pixel size at level 0
  float Dhi[3], Dlo[3];  // D as a double-float pair
  float invDhi[3];       // 1 / Dhi, correctly rounded (0 where D = 0); for a
                         // brick at 2^s finest cells per cell, 1 / (Dhi 2^-s)
                         // is exactly invDhi 2^s
  // FP32 copies for what FP32 can decide: the grid coordinate of a pixel
  // centre is fO + uc fU + vc fV to within eO finest cells (eO infinite where
  // these numbers are too large or too small for FP32)
  float fO[3], fU[3], fV[3], eO[3], fH, fpix0;
  // Axis views whose u and v are grid axes too: the cell of every pixel
  // column on each fixed axis, from axis_table_entry (exactly the set-up's
  // FP64 operations, once per column instead of once per ray), or NULL.
  // Fixed axis s = (A + 1 + s) % 3 (A the ray's axis): entries
  // tab[s * tab_slot + tab_n0 (2^L - 1) + p] for levels L = 0, 1, ..., with
  // p the pixel's j when bit s of tab_byj is set, else its i; -1 where the
  // column misses the grid.
  const int32_t *tab;
  int64_t tab_slot;
  int tab_n0, tab_byj;
};

// 2^-L exactly (0 <= L < 1023).
__device__ __forceinline__ double exp2_neg(int L) {
  return __longlong_as_double((long long)(1023 - L) << 52);
}

// Pixel centre -> ray in finest-cell units, clipped to the box: F(t) = O + t D,
// t >= t0. The pixel size at level L is pix0 2^-L (exact scaling), so a pixel
// of an adaptive image and the same pixel of a fixed image get the same ray.
// The grid coordinate x / h is the correctly rounded quotient (a product with
// 1/h and one residual correction), so a pixel centre that lies exactly on a
// cell face maps exactly onto it, and the half-open rule picks the higher cell.
//
// FP64 costs this GPU 16 SM cycles per warp instruction and 67 cycles of
// latency, conversions to and from FP64 as much as arithmetic, against a
// quarter of a cycle for FP32 (measured). So FP64 is kept to the values that
// are used; what only decides is decided in FP32 where a bound on its error
// allows: whether the ray misses the box, through which face it enters, and
// that it enters before it leaves. What FP32 leaves open goes to
// ray_setup_full, so every result has the bits of that path. About 30 FP64
// instructions instead of 80 for a ray that hits the box, none for most rays
// that miss it.
static __device__ __noinline__ bool ray_setup_full(const GridView &g, const RayGeom &rg, int L, int i,
                                                  int j, double O[3], double &t0, int &eax) {
  const double pix = rg.pix0 * exp2_neg(L);
  const double uc = fma((double)i + 0.5, pix, -rg.H);
  const double vc = fma((double)j + 0.5, pix, -rg.H);
  t0 = -DBL_MAX;
  eax = -1;
  double t1 = DBL_MAX;
  bool hit = true;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const double x = fma(vc, rg.V[a], fma(uc, rg.U[a], rg.C[a]));
    const double q = x * rg.invh[a];
    O[a] = fma(fma(-q, rg.h[a], x), rg.invh[a], q);
    if (rg.D[a] == 0.0) {
      if (!(O[a] >= 0.0 && O[a] < (double)g.nf[a])) hit = false;
    } else {
      double ta = -O[a] * rg.invD[a], tb = ((double)g.nf[a] - O[a]) * rg.invD[a];
      if (ta > tb) {
        const double y = ta;
        ta = tb;
        tb = y;
      }
      if (ta > t0) {
        t0 = ta;
        eax = a;  // the box face the ray enters through
      }
      t1 = fmin(t1, tb);
    }
  }
  return hit && t0 < t1;
}

__device__ __forceinline__ int clampi(int x, int lo, int hi) { return x < lo ? lo : (x > hi ? hi : x); }

// Exact FP64 value of a finite float by integer operations (zeros and
// subnormals by a conversion).
__device__ __forceinline__ double widen(float f) {
  const uint32_t u = __float_as_uint(f), m = u & 0x7fffffffu;
  if (m < 0x00800000u) return (double)f;
  return __hiloint2double((int)((u & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(u << 29));
}
// Exact FP64 value of an integer.
__device__ __forceinline__ double widen_int(int n) {
  return abs(n) < (1 << 24) ? widen((float)n) : (double)n;
}
__device__ __forceinline__ double pick(int a, double x0, double x1, double x2) {
  return a == 0 ? x0 : (a == 1 ? x1 : x2);
}

// Double-float values (unevaluated sums of two FP32 numbers).
struct F2 {
  float hi, lo;
};
__device__ __forceinline__ F2 f2_from(double x) {
  F2 r;
  r.hi = (float)x;
  r.lo = (float)(x - widen(r.hi));
  return r;
}

// Of: O as double-floats.
__device__ __forceinline__ bool ray_setup(const GridView &g, const RayGeom &rg, int L, int i, int j,
                                          double O[3], F2 Of[3], double &t0, int &eax) {
  const float ic = (float)i + 0.5f, jc = (float)j + 0.5f;  // exact: i, j < 2^20
  {
    // the box widened by the error of the pixel centre's coordinate; 2^-20
    // relative covers the roundings of each parameter (16 units, 5 occur)
    const float pix = rg.fpix0 * __int_as_float((127 - L) << 23);
    const float uc = fmaf(ic, pix, -rg.fH), vc = fmaf(jc, pix, -rg.fH);
    float tin = -FLT_MAX, tout = FLT_MAX;
    bool miss = false;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float o = fmaf(vc, rg.fV[a], fmaf(uc, rg.fU[a], rg.fO[a]));
      const float nf = (float)g.nf[a];
      const float e = fmaf(nf, 0x1p-20f, rg.eO[a]);
      if (rg.Dhi[a] == 0.f) {
        miss = miss || o < -e || o > nf + e;
      } else {
        const float ta = (-e - o) * rg.invDhi[a], tb = (nf + e - o) * rg.invDhi[a];
        const float x = fminf(ta, tb), y = fmaxf(ta, tb);
        tin = fmaxf(tin, x - fabsf(x) * 0x1p-20f);
        tout = fminf(tout, y + fabsf(y) * 0x1p-20f);
      }
    }
    if (miss || tin > tout) return false;
  }
  const double pix = rg.pix0 * exp2_neg(L);
  const double uc = fma(widen(ic), pix, -rg.H);
  const double vc = fma(widen(jc), pix, -rg.H);
  // bounds lo <= entry parameter <= hi per axis, and on the exit
  float lo[3], hi[3], tout = FLT_MAX;
  bool clear = true;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const double x = fma(vc, rg.V[a], fma(uc, rg.U[a], rg.C[a]));
    const double q = x * rg.invh[a];
    O[a] = fma(fma(-q, rg.h[a], x), rg.invh[a], q);
    Of[a] = f2_from(O[a]);
    const float nf = (float)g.nf[a], o = Of[a].hi;
    lo[a] = hi[a] = -FLT_MAX;
    if (rg.Dhi[a] == 0.f) {
      clear = clear && o > nf * 0x1p-20f && o < nf - nf * 0x1p-20f;
    } else {
      const float ta = -o * rg.invDhi[a], tb = (nf - o) * rg.invDhi[a];
      const float err = (nf + fabsf(o)) * fabsf(rg.invDhi[a]) * 0x1p-20f;
      lo[a] = fminf(ta, tb) - err;
      hi[a] = fminf(ta, tb) + err;
      tout = fminf(tout, fmaxf(ta, tb) - err);
    }
  }
  eax = lo[0] > hi[1] && lo[0] > hi[2] ? 0 : (lo[1] > hi[0] && lo[1] > hi[2] ? 1 : 2);
  const float tlo = eax == 0 ? lo[0] : (eax == 1 ? lo[1] : lo[2]);
  const float thi = eax == 0 ? hi[0] : (eax == 1 ? hi[1] : hi[2]);
  const float other = eax == 0 ? fmaxf(hi[1], hi[2]) : (eax == 1 ? fmaxf(hi[0], hi[2]) : fmaxf(hi[0], hi[1]));
  if (!(clear && tlo > other && thi < tout)) {
    double Ox[3], tx;  // of their own, so that O stays in registers
    int ex;
    const bool hit = ray_setup_full(g, rg, L, i, j, Ox, tx, ex);
    t0 = tx;
    eax = ex;
    return hit;
  }
  const float De = eax == 0 ? rg.Dhi[0] : (eax == 1 ? rg.Dhi[1] : rg.Dhi[2]);
  const int ne = eax == 0 ? g.nf[0] : (eax == 1 ? g.nf[1] : g.nf[2]);
  const double Oe = pick(eax, O[0], O[1], O[2]);
  const double dist = De > 0.f ? -Oe : widen_int(ne) - Oe;
  t0 = dist * pick(eax, rg.invD[0], rg.invD[1], rg.invD[2]);
  return true;
}

// ray_setup for a ray along grid axis A: only the two fixed coordinates are
// needed (the ray enters at the grid face and crosses every cell of its
// column), computed exactly as ray_setup computes them, so the cells are the
// same; c[A] is left for the caller. Half of ray_setup's FP64 work, which
// matters on a GPU whose FP64 rate is a small fraction of FP32's.
//
// With a column table (RayGeom::tab) the two cells are read from it: where u
// and v are grid axes, x_a depends on one pixel index only (the other term is
// an exact zero), and the table holds this function's result for every
// column (axis_table_entry), so the cells are the same bits.
//
// A is a constant where the kernel is compiled for one axis; the kernels for
// any direction hold one copy of this code and pass the view's axis.
static __device__ __noinline__ unsigned long long axis_cells_fp64(const GridView &g, const RayGeom &rg,
                                                           int A, int L, int i, int j);

// Cells on axes (A + 1) % 3 and (A + 2) % 3; false where the ray misses.
__device__ __forceinline__ bool axis_ray_setup(const GridView &g, const RayGeom &rg, int A, int L,
                                               int i, int j, int &c1, int &c2) {
  if (rg.tab) {
    const int o = rg.tab_n0 * ((1 << L) - 1);
    c1 = __ldg(rg.tab + o + ((rg.tab_byj & 1) ? j : i));
    c2 = __ldg(rg.tab + rg.tab_slot + o + ((rg.tab_byj & 2) ? j : i));
    return c1 >= 0 && c2 >= 0;
  }
  // a separate function, so that none of its FP64 work is executed ahead of
  // the branch on views that have a table
  const unsigned long long cc = axis_cells_fp64(g, rg, A, L, i, j);
  c1 = (int)(uint32_t)cc;
  c2 = (int)(uint32_t)(cc >> 32);
  return c1 >= 0 && c2 >= 0;
}

// The two fixed cells of pixel (L, i, j)'s ray along axis A in FP64: cell on
// axis (A + 1) % 3 in the low word, on (A + 2) % 3 in the high word, -1 where
// the ray misses the grid on that axis.
static __device__ __noinline__ unsigned long long axis_cells_fp64(const GridView &g, const RayGeom &rg,
                                                           int A, int L, int i, int j) {
  const double pix = rg.pix0 * exp2_neg(L);
  const double uc = fma((double)i + 0.5, pix, -rg.H);
  const double vc = fma((double)j + 0.5, pix, -rg.H);
  int c[2];
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const int a0 = A + 1 + s, a = a0 >= 3 ? a0 - 3 : a0;
    const double x = fma(vc, rg.V[a], fma(uc, rg.U[a], rg.C[a]));
    const double q = __dmul_rn(x, rg.invh[a]);
    const double o = fma(fma(-q, rg.h[a], x), rg.invh[a], q);
    c[s] = (o >= 0.0 && o < (double)g.nf[a]) ? (int)o : -1;  // o >= 0: truncation is floor
  }
  return (unsigned long long)(uint32_t)c[0] | ((unsigned long long)(uint32_t)c[1] << 32);
}

// One column-table entry: the cell on grid axis a of level-L pixel column p
// (its i when by_j is false, else its j; the other index is 0, whose term is
// an exact zero), computed with axis_ray_setup's operations; -1 where the
// column misses the grid.
__device__ __forceinline__ int axis_table_entry(const GridView &g, const RayGeom &rg, int a, int L,
                                                int p, bool by_j) {
  const double pix = rg.pix0 * exp2_neg(L);
  const double uc = fma((double)(by_j ? 0 : p) + 0.5, pix, -rg.H);
  const double vc = fma((double)(by_j ? p : 0) + 0.5, pix, -rg.H);
  const double x = fma(vc, rg.V[a], fma(uc, rg.U[a], rg.C[a]));
  const double q = __dmul_rn(x, rg.invh[a]);
  const double o = fma(fma(-q, rg.h[a], x), rg.invh[a], q);
  return (o >= 0.0 && o < (double)g.nf[a]) ? (int)o : -1;
}

template <int NBT, int FMT, int K, class Ctx>
__device__ void march_uniform(RTState<NBT> &r, const GridView &g, const double O[3],
                              const RayGeom &rg, double t0, const Ctx &bc,
                              const BandRegs<NBT> &br) {
  float Q[3], Dl[3], inv[3];
  int lc[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const double F = fma(t0, rg.D[a], O[a]);
    lc[a] = clampi(__double2int_rd(F), 0, g.nf[a] - 1);
    Q[a] = (float)(F - widen_int(lc[a]));
    Dl[a] = rg.Dhi[a];
    inv[a] = rg.invDhi[a];
  }
  // the ray leaves through a face of the grid: no end parameter needed
  if (walk_index_fits(g.nf[0], g.nf[1], g.nf[2], K))
    march_block<NBT, FMT, K, int>(r, Q, Dl, inv, FLT_MAX, lc[0], lc[1], lc[2], g.nf[0], g.nf[1], g.nf[2],
                               g.nf[0], g.nf[0] * g.nf[1], g.cells, bc, br);
  else
    march_block<NBT, FMT, K, int64_t>(r, Q, Dl, inv, FLT_MAX, lc[0], lc[1], lc[2], g.nf[0], g.nf[1],
                                   g.nf[2], (int64_t)g.nf[0], (int64_t)g.nf[0] * g.nf[1], g.cells,
                                   bc, br);
}

// Error-free transformations (Knuth's TwoSum and the fused-multiply-add form
// of Dekker's TwoProduct).
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}
__device__ __forceinline__ F2 f2_add_f(F2 a, float b) {
  float s, e;
  two_sum(a.hi, b, s, e);
  e += a.lo;
  F2 r;
  r.hi = s + e;
  r.lo = e - (r.hi - s);
  return r;
}
// (O + t D - anchor) in finest cells, accurate to FP32 rounding of the result:
// the products and sums that cancel are carried in double-float.
__device__ __forceinline__ float f2_offset(F2 O, F2 t, F2 D, float anchor) {
  const float p = t.hi * D.hi;
  float pe = fmaf(t.hi, D.hi, -p);            // exact error of t.hi * D.hi
  pe = fmaf(t.hi, D.lo, fmaf(t.lo, D.hi, pe));
  float s, se;
  two_sum(O.hi, p, s, se);
  const float a = s - anchor;                  // exact: s lies within a cell of anchor
  return a + ((se + O.lo) + pe);
}

// Dense brick-map entry of finest cell c (see GridView::bmap).
__device__ __forceinline__ int map_entry(const GridView &g, int c0, int c1, int c2) {
  const int sm = g.log2B + g.Lm - g.mapL;
  return __ldg(g.bmap + ((int64_t)(c2 >> sm) * g.nm[1] + (c1 >> sm)) * g.nm[0] + (c0 >> sm));
}

// Leaf brick holding finest cell c from its map entry: id, and its level in
// `lev`. Below the map level the brick octree is descended.
__device__ __forceinline__ int brick_of(const GridView &g, int e, const int c[3], int &lev) {
  if (e >= 0) {
    lev = e >> kMapLevelShift;
    return e & kMapIdMask;
  }
  const int s0 = g.log2B + g.Lm;
  lev = g.mapL;
  while (e < 0) {
    ++lev;
    const int sh = s0 - lev;
    const int oc = ((c[0] >> sh) & 1) | (((c[1] >> sh) & 1) << 1) | (((c[2] >> sh) & 1) << 2);
    e = __ldg(g.oct + (int64_t)(-e - 1) * 8 + oc);
  }
  return e;
}

// Brick by brick: find the leaf brick holding finest cell c, compute the
// entry point in it and the exit face (FP64 at levels >= fp64_level, else
// double-float), march its cells, step to the finest cell across the exit
// face. The map entry of the next brick is fetched before the current brick
// is marched, so its latency overlaps the march. Per-launch constants
// (direction, its inverse and its double-float split) are read from the
// kernel-parameter bank, not held per thread.
template <int NBT, int FMT, int K, class Ctx>
__device__ void march_amr(RTState<NBT> &r, const GridView &g, const double O[3], const F2 Of[3],
                          const RayGeom &rg, double t0, int eax, int fp64_level,
                          const Ctx &bc, const BandRegs<NBT> &br) {
  const int B = g.B, lb = g.log2B, Lm = g.Lm;
  int c[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    // the entry face's coordinate is 0 or nf to within rounding: its cell is
    // the first or the last
    if (a == eax) c[a] = rg.Dhi[a] > 0.f ? 0 : g.nf[a] - 1;
    else c[a] = clampi(__double2int_rd(rg.Dhi[a] == 0.f ? O[a] : fma(t0, rg.D[a], O[a])), 0, g.nf[a] - 1);
  }
  F2 t = f2_from(t0);
  const int max_iter = 4 * (g.nf[0] + g.nf[1] + g.nf[2]);
  const float ulp = fmaf((float)max(g.nf[0], max(g.nf[1], g.nf[2])), 0x1p-44f, (float)B * 0x1p-20f);
  int e = map_entry(g, c[0], c[1], c[2]);
  for (int it = 0; it < max_iter; ++it) {
    int lev;
    const int code = brick_of(g, e, c, lev);
    r.maxlev = max(r.maxlev, lev);
    const int shift = Lm - lev;
    const int sb = lb + shift;
    const int S = B << shift;
    const float scale = __int_as_float((127 - shift) << 23);  // 2^-shift
    const float up = __int_as_float((127 + shift) << 23);     // 2^shift
    int lc[3], anchor[3], bo[3];
    float Q[3], Dl[3], inv[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      bo[a] = (c[a] >> sb) << sb;
      lc[a] = (c[a] - bo[a]) >> shift;
      anchor[a] = bo[a] + (lc[a] << shift);
      Dl[a] = rg.Dhi[a] * scale;
      inv[a] = rg.invDhi[a] * up;
    }
    const bool deep = lev >= fp64_level;
    // entry point relative to the entry cell, and the exit face: smallest
    // parameter over the axes, measured from the entry
    float tend = FLT_MAX;
    int ax = -1;
    double te = 0.0;
    // On the axis the brick is entered through, the entry point is the face
    // itself, an integer finest coordinate: its offset is exact. On an axis
    // the ray does not move along, the offset O - anchor is constant and exact
    // in double-float. Only the other axes need the FP64 (or double-float)
    // position of the entry point.
    if (deep) {
      const double td = widen(t.hi) + widen(t.lo);
      // the two axes b1, b2 that are not the entry axis
      const int b1 = eax == 0 ? 1 : 0, b2 = eax == 2 ? 1 : 2;
      const double E1 = pick(b1, O[0], O[1], O[2]) - widen_int(b1 == 0 ? anchor[0] : anchor[1]);
      const double E2 = pick(b2, O[0], O[1], O[2]) - widen_int(b2 == 1 ? anchor[1] : anchor[2]);
      const float Q1 = (float)fma(td, pick(b1, rg.D[0], rg.D[1], rg.D[2]), E1) * scale;
      const float Q2 = (float)fma(td, pick(b2, rg.D[0], rg.D[1], rg.D[2]), E2) * scale;
      // exit parameters from the entry point in FP32, to within 2^-20 of the
      // brick's edge (5 roundings of 2^-24, and the entry point is within
      // 2^-24 of a cell) and 2^-44 of the grid's (td has 48 bits): they tell
      // the exit axis unless two faces are met almost together
      float x[3], xe[3];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        if (a == eax)
          Q[a] = (float)((Dl[a] > 0.f ? c[a] : c[a] + 1) - anchor[a]) * scale;
        else if (Dl[a] == 0.f)
          Q[a] = ((Of[a].hi - (float)anchor[a]) + Of[a].lo) * scale;
        else
          Q[a] = a == b1 ? Q1 : Q2;
        x[a] = Dl[a] == 0.f ? FLT_MAX : ((float)(Dl[a] > 0.f ? B - lc[a] : -lc[a]) - Q[a]) * inv[a];
        xe[a] = ulp * fabsf(inv[a]);
      }
      ax = x[0] <= x[1] && x[0] <= x[2] ? 0 : (x[1] <= x[2] ? 1 : 2);
      const float xm = ax == 0 ? x[0] + xe[0] : (ax == 1 ? x[1] + xe[1] : x[2] + xe[2]);
      const bool clear = (ax == 0 || xm < x[0] - xe[0]) && (ax == 1 || xm < x[1] - xe[1]) &&
                         (ax == 2 || xm < x[2] - xe[2]);
      double tmin;
      if (clear) {
        const int face = ax == 0 ? (Dl[0] > 0.f ? bo[0] + S : bo[0])
                                 : (ax == 1 ? (Dl[1] > 0.f ? bo[1] + S : bo[1])
                                            : (Dl[2] > 0.f ? bo[2] + S : bo[2]));
        tmin = (widen_int(face) - pick(ax, O[0], O[1], O[2])) * pick(ax, rg.invD[0], rg.invD[1], rg.invD[2]);
      } else {
        tmin = DBL_MAX;
        ax = -1;
#pragma unroll
        for (int a = 0; a < 3; ++a)
          if (Dl[a] != 0.f) {
            const double ta = (widen_int(Dl[a] > 0.f ? bo[a] + S : bo[a]) - O[a]) * rg.invD[a];
            if (ta < tmin) {
              tmin = ta;
              ax = a;
            }
          }
      }
      // te = max(tmin, td); tend = te - td (the difference's sign is exact)
      const double dt = tmin - td;
      const bool fwd = __double2hiint(dt) >= 0;
      te = fwd ? tmin : td;
      tend = fwd ? (float)dt : 0.f;
    } else {
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        F2 Dv;
        Dv.hi = rg.Dhi[a];
        Dv.lo = rg.Dlo[a];
        if (a == eax)
          Q[a] = (float)((Dl[a] > 0.f ? c[a] : c[a] + 1) - anchor[a]) * scale;
        else if (Dl[a] == 0.f)
          Q[a] = ((Of[a].hi - (float)anchor[a]) + Of[a].lo) * scale;
        else
          Q[a] = f2_offset(Of[a], t, Dv, (float)anchor[a]) * scale;
        if (Dl[a] != 0.f) {
          const float face = Dl[a] > 0.f ? (float)(B - lc[a]) : (float)(-lc[a]);
          const float ta = (face - Q[a]) * inv[a];
          if (ta < tend) {
            tend = ta;
            ax = a;
          }
        }
      }
      if (tend < 0.f) tend = 0.f;
    }
    // finest cell just across the exit face; the other coordinates, from the
    // exit point in this brick's frame, stay in this brick's range
    bool out = ax < 0;
    int cn[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      if (a == ax) {
        cn[a] = Dl[a] > 0.f ? bo[a] + S : bo[a] - 1;
        out = out || cn[a] < 0 || cn[a] >= g.nf[a];
      } else {
        const float x = fmaf(tend, Dl[a], Q[a]);  // local cells from the entry cell
        const int f = anchor[a] + (int)floorf(x * up);
        cn[a] = clampi(f, bo[a], bo[a] + S - 1);
      }
    }
    const int en = out ? 0 : map_entry(g, cn[0], cn[1], cn[2]);
    const int64_t boff = (int64_t)code << (3 * lb);
    const void *cb = FMT == kCellRho ? (const void *)((const float *)g.cells + boff)
                                     : (const void *)((const uint2 *)g.cells + boff);
    bool cell = false;
    if constexpr (NBT == 1) {
      cell = B == 1;
      if (cell) march_cell<FMT>(r, Q, Dl, inv, tend, cb, bc, br);
    }
    if (!cell)
      march_block<NBT, FMT, K, int>(r, Q, Dl, inv, tend, lc[0], lc[1], lc[2], B, B, B, B, B * B, cb, bc, br);
    if (out) break;
    // advance to the exit point
    if (deep) t = f2_from(te);
    else t = f2_add_f(t, tend);
    c[0] = cn[0];
    c[1] = cn[1];
    c[2] = cn[2];
    e = en;
    eax = ax;
  }
}

// A ray parallel to grid axis A (every face-on view: the bench's +z view, the
// paper's ring view). Such a ray enters the grid, and every brick after,
// through an A face and crosses each brick whole, through a column of B cells
// of the brick's level, each with the same chord: the cell width over the
// direction, |1 / D_A| 2^(Lm - level) (an exact power-of-two scaling of the
// per-launch FP32 reciprocal). The other two finest coordinates never change
// and the next brick is the one holding the finest cell just past the far
// face, so the walk is integer-exact: no entry or exit parameter is computed,
// in FP32 or FP64, and no cell can be skipped or counted twice. Every kernel
// form (and the batched kernel) sends such a ray here, so all give the same
// bits for it. The map entry of the next brick is fetched before the current
// brick's column is marched, so its latency overlaps the march.
// W16 = +1 / -1: bricks of 16^3 cells, rays towards higher / lower cells of
// the constant axis A (march_column16); 0: any brick and direction.
template <int NBT, int FMT, int U, bool TAIL, int W16 = 0, int CA = 0>
__device__ __forceinline__ void march_amr_axis(RTState<NBT> &r, const GridView &g, int A, int c1,
                                               int c2, const RayGeom &rg, const BandCtx &bc,
                                               const BandRegs<NBT> &br) {
  if (W16 != 0) A = CA;
  const int A1 = A == 2 ? 0 : A + 1, A2 = A == 0 ? 2 : A - 1;
  const int B = W16 != 0 ? 16 : g.B, lb = W16 != 0 ? 4 : g.log2B, Lm = g.Lm;
  const int nfA = A == 0 ? g.nf[0] : (A == 1 ? g.nf[1] : g.nf[2]);
  const bool pos = W16 != 0 ? W16 > 0 : (A == 0 ? rg.Dhi[0] : (A == 1 ? rg.Dhi[1] : rg.Dhi[2])) > 0.f;
  const float a1 = fabsf(A == 0 ? rg.invDhi[0] : (A == 1 ? rg.invDhi[1] : rg.invDhi[2]));
  // cell strides inside a brick, x fastest
  const int lA = A * lb, l1 = A1 * lb, l2 = A2 * lb;
  const int d = pos ? (1 << lA) : -(1 << lA);
  // the brick map along the ray: entry column + (cA >> sm) * step
  const int sm = lb + Lm - g.mapL;
  const int m0 = 1, m1 = g.nm[0], m2 = g.nm[0] * g.nm[1];  // at most 2^24 entries
  const int32_t *column = g.bmap + (c1 >> sm) * (A1 == 0 ? m0 : (A1 == 1 ? m1 : m2)) +
                          (c2 >> sm) * (A2 == 0 ? m0 : (A2 == 1 ? m1 : m2));
  const int step = A == 0 ? m0 : (A == 1 ? m1 : m2);
  int cA = pos ? 0 : nfA - 1;  // the ray enters through the grid face
  const int max_iter = 4 * nfA;
  int e = __ldg(column + (cA >> sm) * step);
  for (int it = 0; it < max_iter; ++it) {
    int lev;
    if (e >= 0) {
      lev = e >> kMapLevelShift;
      e &= kMapIdMask;
    } else {
      lev = g.mapL;
      while (e < 0) {
        ++lev;
        const int sh = lb + Lm - lev;
        const int oc = (((cA >> sh) & 1) << A) | (((c1 >> sh) & 1) << A1) | (((c2 >> sh) & 1) << A2);
        e = __ldg(g.oct + (int64_t)(-e - 1) * 8 + oc);
      }
    }
    r.maxlev = max(r.maxlev, lev);
    const int shift = Lm - lev;
    const int S = B << shift;
    const int cn = pos ? cA + S : cA - S;
    const bool out = cn < 0 || cn >= nfA;
    const int en = out ? 0 : __ldg(column + (cn >> sm) * step);
    const int idx = (pos ? 0 : (B - 1) << lA) + (((c1 >> shift) & (B - 1)) << l1) +
                    (((c2 >> shift) & (B - 1)) << l2);
    const float ds = a1 * __int_as_float((127 + shift) << 23);  // a1 2^shift
    const int64_t boff = (int64_t)e << (3 * lb);
    const void *cb = FMT == kCellRho ? (const void *)((const float *)g.cells + boff)
                                     : (const void *)((const uint2 *)g.cells + boff);
    if constexpr (W16 != 0) {
      const int low = (((c1 >> shift) & 15) << l1) + (((c2 >> shift) & 15) << l2);
      march_column16<NBT, FMT, CA, (W16 > 0)>(
          r, FMT == kCellRho ? (const void *)((const float *)cb + low) : (const void *)((const uint2 *)cb + low),
          ds, bc, br);
    } else {
      march_column<NBT, FMT, U, TAIL, int>(r, cb, idx, d, B, ds, bc, br);
    }
    if (out) break;
    cA = cn;
    e = en;
  }
}

// march_amr_axis for bricks of at most 8 cells, compiled on its own: a brick's
// cells are too few for a group, so each takes the compensated step, and a ray
// spends its time waiting for one short column after the other. Here the next
// brick's records (and the map entry of the one after) are on their way while
// a brick is summed. (One kernel with both walks spilled registers; the walk
// that waits for each column took 26 us a sweep on the ring grid, 8^3 bricks.)
// M: the largest brick edge, 8, or 2 for bricks of one or two cells, where eight
// cells' instructions per brick are wasted (a fixed image of 500^2 pixels through
// bricks of one cell 186 us with M = 8, 127 with 2).
template <int NBT, int FMT, int M>
__device__ __forceinline__ void march_amr_axis_small(RTState<NBT> &r, const GridView &g, int A,
                                                     int c1, int c2, const RayGeom &rg,
                                                     const BandCtx &bc, const BandRegs<NBT> &br) {
  const int A1 = A == 2 ? 0 : A + 1, A2 = A == 0 ? 2 : A - 1;
  const int B = g.B, lb = g.log2B, Lm = g.Lm;
  const int nfA = A == 0 ? g.nf[0] : (A == 1 ? g.nf[1] : g.nf[2]);
  const bool pos = (A == 0 ? rg.Dhi[0] : (A == 1 ? rg.Dhi[1] : rg.Dhi[2])) > 0.f;
  const float a1 = fabsf(A == 0 ? rg.invDhi[0] : (A == 1 ? rg.invDhi[1] : rg.invDhi[2]));
  const int lA = A * lb, l1 = A1 * lb, l2 = A2 * lb;
  const int d = pos ? (1 << lA) : -(1 << lA);
  const int sm = lb + Lm - g.mapL;
  const int m0 = 1, m1 = g.nm[0], m2 = g.nm[0] * g.nm[1];
  const int32_t *column = g.bmap + (c1 >> sm) * (A1 == 0 ? m0 : (A1 == 1 ? m1 : m2)) +
                          (c2 >> sm) * (A2 == 0 ? m0 : (A2 == 1 ? m1 : m2));
  const int step = A == 0 ? m0 : (A == 1 ? m1 : m2);
  int cA = pos ? 0 : nfA - 1;  // finest cell through which the next brick is entered
  int e = __ldg(column + (cA >> sm) * step);
  float rh[M], nrh[M], ds = 0.f, nds = 0.f;
  uint32_t xv[M], nxv[M];
  bool have = false, more = true;
  while (true) {
    if (more) {  // ask for the brick at cA
      int lev;
      if (e >= 0) {
        lev = e >> kMapLevelShift;
        e &= kMapIdMask;
      } else {
        lev = g.mapL;
        while (e < 0) {
          ++lev;
          const int sh = lb + Lm - lev;
          const int oc = (((cA >> sh) & 1) << A) | (((c1 >> sh) & 1) << A1) | (((c2 >> sh) & 1) << A2);
          e = __ldg(g.oct + (int64_t)(-e - 1) * 8 + oc);
        }
      }
      r.maxlev = max(r.maxlev, lev);
      const int shift = Lm - lev;
      const int idx = (pos ? 0 : (B - 1) << lA) + (((c1 >> shift) & (B - 1)) << l1) +
                      (((c2 >> shift) & (B - 1)) << l2);
      nds = a1 * __int_as_float((127 + shift) << 23);  // a1 2^shift
      const int64_t at = ((int64_t)e << (3 * lb)) + idx;
#pragma unroll
      for (int u = 0; u < M; ++u)
        if (u < B) load_cell<FMT>(g.cells, at + u * d, nrh[u], nxv[u]);
      cA = pos ? cA + (B << shift) : cA - (B << shift);
    }
    const bool next = more;
    more = next && cA >= 0 && cA < nfA;
    if (more) e = __ldg(column + (cA >> sm) * step);
    if (have) {
      r.steps += (uint32_t)B;
      // the whole brick's column dark: N alone (see rt_term; the zero terms
      // of several dark cells change a sum as one does)
      uint32_t x = 0u;
      float tot = 0.f;
#pragma unroll
      for (int u = 0; u < M; ++u)
        if (u < B) {
          x = FMT == kCellLam ? x | xv[u] : max(x, xv[u]);
          tot += rh[u];
        }
      if (FMT != kCellRho && cell_dark<FMT>(x, br.xz) && fmaf(tot, ds, r.N) <= 0.5f * FLT_MAX) {
#pragma unroll
        for (int u = 0; u < M; ++u)
          if (u < B) kahan_add(r.N, r.cN, __fmul_rn(rh[u], ds));
        kahan_add(r.I[0], r.cI[0], 0.f);
        r.T[0] = ex2_approx(br.nk[0] * r.N);
      } else {
#pragma unroll
        for (int u = 0; u < M; ++u)
          if (u < B) rt_term<NBT, FMT, false>(r, rh[u], xv[u], ds, bc, br);
      }
    }
    if (!next) break;
#pragma unroll
    for (int u = 0; u < M; ++u) {
      rh[u] = nrh[u];
      xv[u] = nxv[u];
    }
    ds = nds;
    have = true;
  }
}

// The uniform grid's version: the whole column of nf[A] cells.
template <int NBT, int FMT, int U>
__device__ __forceinline__ void march_uniform_axis(RTState<NBT> &r, const GridView &g, int A, int c1,
                                                   int c2, const RayGeom &rg, const BandCtx &bc,
                                                   const BandRegs<NBT> &br) {
  const bool pos = (A == 0 ? rg.Dhi[0] : (A == 1 ? rg.Dhi[1] : rg.Dhi[2])) > 0.f;
  const float ds = fabsf(A == 0 ? rg.invDhi[0] : (A == 1 ? rg.invDhi[1] : rg.invDhi[2]));
  const int nfA = A == 0 ? g.nf[0] : (A == 1 ? g.nf[1] : g.nf[2]);
  const int64_t s1 = g.nf[0], s2 = (int64_t)g.nf[0] * g.nf[1];
  const int64_t stA = A == 0 ? 1 : (A == 1 ? s1 : s2);
  const int64_t st1 = A == 0 ? s1 : (A == 1 ? s2 : 1), st2 = A == 0 ? s2 : (A == 1 ? 1 : s1);
  const int64_t idx = (pos ? 0 : (int64_t)(nfA - 1) * stA) + (int64_t)c1 * st1 + (int64_t)c2 * st2;
  march_column<NBT, FMT, U, true, int64_t>(r, g.cells, idx, pos ? stA : -stA, nfA, ds, bc, br);
}

// Pixel (L, i, j)'s ray along grid axis A through either kind of grid. DIR: the
// kernel's form (trace_ray).
template <int NBT, bool AMR, int FMT, int DIR, int U>
__device__ __forceinline__ void march_axis(RTState<NBT> &st, const GridView &g, const RayGeom &rg,
                                           int A, int L, int i, int j, const BandCtx &bc,
                                           BandRegs<NBT> &br) {
  int c1, c2;
  if (!axis_ray_setup(g, rg, A, L, i, j, c1, c2)) return;
  if (NBT > 1) band_load<NBT>(br, bc);
  if constexpr (!AMR) march_uniform_axis<NBT, FMT, U>(st, g, A, c1, c2, rg, bc, br);
  else if constexpr (DIR >= 13) march_amr_axis_small<NBT, FMT, 2>(st, g, A, c1, c2, rg, bc, br);
  else if constexpr (DIR >= 7) march_amr_axis<NBT, FMT, U, false, (DIR < 10 ? 1 : -1), (DIR - 1) % 3>(st, g, A, c1, c2, rg, bc, br);
  else if constexpr (DIR >= 4) march_amr_axis_small<NBT, FMT, 8>(st, g, A, c1, c2, rg, bc, br);
  else march_amr_axis<NBT, FMT, U, (DIR <= 0)>(st, g, A, c1, c2, rg, bc, br);
}

// One ray (pixel (L, i, j)) through the grid, bands [b0, b0 + NBT) of bc/br.
// DIR, the kernel's form:
//   0: any direction (the batched kernel);
//   1 + A: every ray of the launch is parallel to grid axis A, one band (bricks
//     of 16 cells and more, or a uniform grid); 4 + A: the same with bricks of
//     4 or 8 cells; 13 + A: of 1 or 2; 7 + A and 10 + A: with 16^3 bricks,
//     towards higher and lower cells;
//   -1: inclined rays in launches of few rays (DdaChunk); -2: inclined rays;
//   -3: rays parallel to some axis, any number of bands.
template <int NBT, bool AMR, int FMT, int DIR = 0>
__device__ __forceinline__ void trace_ray(RTState<NBT> &st, const GridView &g, const RayGeom &rg,
                                          int L, int i, int j, int fp64_level, const BandCtx &bc,
                                          BandRegs<NBT> &br) {
  rt_init<NBT>(st);
  constexpr int U = ColumnUnroll<DIR>::value;
  if constexpr (DIR >= 1) {
    march_axis<NBT, AMR, FMT, DIR, U>(st, g, rg, (DIR - 1) % 3, L, i, j, bc, br);
    return;
  }
  if constexpr (DIR == 0 || DIR == -3) {
    const bool m0 = rg.Dhi[0] != 0.f, m1 = rg.Dhi[1] != 0.f, m2 = rg.Dhi[2] != 0.f;
    if (DIR == -3 || m0 + m1 + m2 == 1) {
      march_axis<NBT, AMR, FMT, DIR, U>(st, g, rg, m0 ? 0 : (m1 ? 1 : 2), L, i, j, bc, br);
      return;
    }
  }
  if constexpr (DIR <= 0 && DIR != -3) {
    double O[3], t0;
    F2 Of[3];
    int eax;
    if (!ray_setup(g, rg, L, i, j, O, Of, t0, eax)) return;
    constexpr int K = DdaChunk<NBT, DIR>::value;
    if (AMR) march_amr<NBT, FMT, K>(st, g, O, Of, rg, t0, eax, fp64_level, bc, br);
    else march_uniform<NBT, FMT, K>(st, g, O, rg, t0, bc, br);
  }
}

// An inclined ray in the wide form; its sums are left in wc.sums.
template <bool AMR, int FMT>
__device__ __forceinline__ void trace_wide(RTState<0> &st, const GridView &g, const RayGeom &rg, int L,
                                           int i, int j, int fp64_level, const WideCtx &wc) {
  wide_init(st, wc);
  BandRegs<0> br;
  br.xz = 0xffffffffu;
  for (int b = 0; b < wc.nbh; ++b) br.xz = min(br.xz, wc.band[b].xz);
  double O[3], t0;
  F2 Of[3];
  int eax;
  if (!ray_setup(g, rg, L, i, j, O, Of, t0, eax)) return;
  constexpr int K = DdaChunk<0, -2>::value;
  if (AMR) march_amr<0, FMT, K>(st, g, O, Of, rg, t0, eax, fp64_level, wc, br);
  else march_uniform<0, FMT, K>(st, g, O, rg, t0, wc, br);
  if (st.due)  // the last cells were dark
    for (int q = 0; q < wc.pairs; ++q) {
      float4 s = wc.sums[q * blockDim.x];
      kahan_add(s.x, s.y, 0.f);
      kahan_add(s.z, s.w, 0.f);
      wc.sums[q * blockDim.x] = s;
    }
}

// World camera -> per-launch ray geometry (FP64, host).
static inline RayGeom make_geom(const GridView &g, const Camera &cam, int n0) {
  RayGeom rg;
  for (int a = 0; a < 3; ++a) {
    rg.C[a] = cam.c[a] - g.lo[a];
    rg.U[a] = cam.u[a];
    rg.V[a] = cam.v[a];
    rg.h[a] = g.h[a];
    rg.invh[a] = 1.0 / g.h[a];
    rg.D[a] = cam.d[a] / g.h[a];
    rg.invD[a] = cam.d[a] != 0.0 ? 1.0 / rg.D[a] : 0.0;
    rg.Dhi[a] = (float)rg.D[a];
    // a direction component too small for FP32 (the ray moves less than
    // 1e-30 cells per unit length along that axis) is taken as zero
    if (!(fabsf(rg.Dhi[a]) >= 1e-30f)) {
      rg.D[a] = 0.0;
      rg.invD[a] = 0.0;
      rg.Dhi[a] = 0.f;
    }
    rg.Dlo[a] = (float)(rg.D[a] - (double)rg.Dhi[a]);
    rg.invDhi[a] = rg.Dhi[a] != 0.f ? 1.0f / rg.Dhi[a] : 0.f;
  }
  rg.H = cam.H;
  rg.pix0 = (2.0 * cam.H) / (double)n0;
  rg.fH = (float)rg.H;
  rg.fpix0 = (float)rg.pix0;
  for (int a = 0; a < 3; ++a) {
    rg.fO[a] = (float)(rg.C[a] * rg.invh[a]);
    rg.fU[a] = (float)(rg.U[a] * rg.invh[a]);
    rg.fV[a] = (float)(rg.V[a] * rg.invh[a]);
    // roundings of FP32: at most 8 units of each product (32 allowed)
    const double reach = (fabs(rg.C[a]) + 2.0 * rg.H * (fabs(rg.U[a]) + fabs(rg.V[a]))) * rg.invh[a];
    const bool fits = rg.H < 1e25 && rg.pix0 > 1e-25 && rg.invh[a] < 1e25 && rg.invh[a] > 1e-25 && reach < 1e15;
    rg.eO[a] = fits ? (float)(reach * 0x1p-20) : HUGE_VALF;
  }
  rg.tab = nullptr;
  rg.tab_slot = 0;
  rg.tab_n0 = n0;
  rg.tab_byj = 0;
  return rg;
}

// Whether the view's rays run along one grid axis A with u and v along the
// other two (each with one nonzero component); then *byj gets bit s set when
// fixed axis (A + 1 + s) % 3 follows v (the pixel's j).
static inline bool axis_table_view(const RayGeom &rg, int *A, int *byj) {
  const int moving = (rg.Dhi[0] != 0.f) + (rg.Dhi[1] != 0.f) + (rg.Dhi[2] != 0.f);
  if (moving != 1) return false;
  *A = rg.Dhi[0] != 0.f ? 0 : (rg.Dhi[1] != 0.f ? 1 : 2);
  *byj = 0;
  for (int s = 0; s < 2; ++s) {
    const int a = (*A + 1 + s) % 3;
    const bool u = rg.U[a] != 0.0, v = rg.V[a] != 0.0;
    if (u == v) return false;
    if (v) *byj |= 1 << s;
  }
  return true;
}


}  // namespace air
