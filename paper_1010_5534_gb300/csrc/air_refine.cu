// air_refine.cu -- the adaptive image (Parkin 2010, Section 2 steps iii-vi):
// truncation-error scan (Section 3, Eq. 2), 2:1 level balance between adjacent
// pixels, quadtree refinement with a warp-ballot prefix sum that compacts the
// new rays, and the leaf output with the band flux.
//
// The image quadtree is a node list: the base image row-major (node j*n0 + i),
// then four consecutive children per refined node, in the order of the
// parents. Each node stores its level, (i, j) at that level and the index of
// its first child (-1 for a leaf). The pixel at level L holding (i, j) is
// found by descending from the base node through the child links; this gives
// the deepest existing node at a level <= L, which is the value a missing
// neighbour takes in the stencil.
#include <algorithm>
#include <atomic>
#include <cfloat>

#include "air_tree.cuh"

namespace air {

// Step iii: flag every leaf below max_level whose xi >= xi_crit.
// ---- warp-ballot prefix sums ------------------------------------------------
// A block covers kScanItems = kScanRounds * kScanBlock consecutive items;
// round r holds items [r * kScanBlock, (r + 1) * kScanBlock) of the block, one
// per thread, so every load is coalesced and the block-local order is the
// global order.

struct PredFlag {
  const uint32_t *flag;
  __device__ bool operator()(int64_t k) const { return flag[k] != 0; }
};

template <class Pred>
__global__ void __launch_bounds__(kScanBlock) k_count(Pred pred, int64_t n, int32_t *bcount) {
  __shared__ int32_t wsum[kScanBlock / 32];
  const int64_t start = (int64_t)blockIdx.x * kScanItems;
  int32_t cnt = 0;
  for (int rr = 0; rr < kScanRounds; ++rr) {
    const int64_t k = start + (int64_t)rr * kScanBlock + threadIdx.x;
    const bool p = k < n && pred(k);
    cnt += __popc(__ballot_sync(0xffffffffu, p));
  }
  if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = cnt;
  __syncthreads();
  if (threadIdx.x == 0) {
    int32_t s = 0;
    for (int w = 0; w < kScanBlock / 32; ++w) s += wsum[w];
    bcount[blockIdx.x] = s;
  }
}

// Exclusive scan of the per-block counts in one block; total -> *total.
__global__ void __launch_bounds__(1024) k_scan_blocks(const int32_t *bcount, int64_t nb,
                                                      int64_t *boff, int64_t *total) {
  __shared__ int64_t part[1024];
  const int64_t per = (nb + 1023) / 1024;
  const int64_t a = threadIdx.x * per, b = min(nb, a + per);
  int64_t s = 0;
  for (int64_t x = a; x < b; ++x) s += bcount[x];
  part[threadIdx.x] = s;
  __syncthreads();
  for (int off = 1; off < 1024; off <<= 1) {
    const int64_t v = threadIdx.x >= off ? part[threadIdx.x - off] : 0;
    __syncthreads();
    part[threadIdx.x] += v;
    __syncthreads();
  }
  int64_t run = part[threadIdx.x] - s;
  for (int64_t x = a; x < b; ++x) {
    boff[x] = run;
    run += bcount[x];
  }
  if (threadIdx.x == 1023) *total = part[1023];
}

// ---- open-leaf list -----------------------------------------------------------
// The leaves below the top level, in ascending node order: the only nodes a
// sweep can flag. Steps iii and iv run over this list instead of every node;
// children are still emitted in parent (node) order, so the quadtree is the
// same. Flags of nodes outside the list are kept at zero (a refined node's
// flag is cleared when its children are emitted, children start at zero).

// Level-map entries of the four children (first index c0, level l) of the
// level-(l - 1) pixel (i, j); only levels l < Lm have maps.
__device__ __forceinline__ void set_level_map(int32_t *lmap, int n0, int l, int i, int j,
                                              int64_t c0) {
  const int64_t nl = (int64_t)n0 << l;
  int32_t *row = lmap + level_map_offset(n0, l) + (int64_t)(2 * j) * nl + 2 * i;
  row[0] = (int32_t)c0;
  row[1] = (int32_t)(c0 + 1);
  row[nl] = (int32_t)(c0 + 2);
  row[nl + 1] = (int32_t)(c0 + 3);
}

__global__ void k_iota(int32_t *list, int64_t m) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < m) list[i] = (int32_t)i;
}

__global__ void k_xi_scan_list(TreeView t, const int32_t *__restrict__ open, int64_t m,
                               double xi_crit, int xi_norm, int refine_on,
                               uint32_t *__restrict__ flag, const int32_t *lmap) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m) return;
  const int64_t k = open[i];
  flag[k] = xi_flag(t, NodeLookup{0, lmap}, k, xi_crit, xi_norm, refine_on);
}

__global__ void k_balance_list(TreeView t, const int32_t *__restrict__ open, int64_t m,
                               uint32_t *__restrict__ flag, uint32_t *__restrict__ err,
                               const int32_t *lmap) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += stride) {
    const int k = open[i];
    if (flag[k] != 0) balance_from(t, NodeLookup{0, lmap}, k, flag, err);
  }
}

// Three selections over the list, per entry k = open[i]: flagged (refined
// this sweep), kept (not flagged: stays an open leaf), and flagged with
// children below the top level (its four children join the list).
struct ListSel {
  bool f, keep, co;
};
__device__ __forceinline__ ListSel list_sel(const TreeView &t, const int32_t *open, int64_t m,
                                            const uint32_t *flag, int Lm, int64_t i, int &k) {
  ListSel q{false, false, false};
  k = 0;
  if (i < m) {
    k = open[i];
    q.f = flag[k] != 0;
    q.keep = !q.f;
    q.co = q.f && t.lvl[k] + 1 < Lm;
  }
  return q;
}

__global__ void __launch_bounds__(kScanBlock) k_count3(TreeView t, const int32_t *open, int64_t m,
                                                       const uint32_t *flag, int Lm,
                                                       int32_t *bcount, int64_t nb) {
  __shared__ int32_t wsum[3][kScanBlock / 32];
  const int64_t start = (int64_t)blockIdx.x * kScanItems;
  int32_t c0 = 0, c1 = 0, c2 = 0;
  for (int rr = 0; rr < kScanRounds; ++rr) {
    int k;
    const ListSel q = list_sel(t, open, m, flag, Lm, start + (int64_t)rr * kScanBlock + threadIdx.x, k);
    c0 += __popc(__ballot_sync(0xffffffffu, q.f));
    c1 += __popc(__ballot_sync(0xffffffffu, q.keep));
    c2 += __popc(__ballot_sync(0xffffffffu, q.co));
  }
  if ((threadIdx.x & 31) == 0) {
    wsum[0][threadIdx.x >> 5] = c0;
    wsum[1][threadIdx.x >> 5] = c1;
    wsum[2][threadIdx.x >> 5] = c2;
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    int32_t s = 0;
    for (int w = 0; w < kScanBlock / 32; ++w) s += wsum[threadIdx.x][w];
    bcount[threadIdx.x * nb + blockIdx.x] = s;
  }
}

// Block b of the launch scans selection b's per-block counts.
__global__ void __launch_bounds__(1024) k_scan_blocks3(const int32_t *bcount, int64_t nb,
                                                       int64_t *boff, int64_t *total) {
  __shared__ int64_t part[1024];
  const int32_t *bc = bcount + blockIdx.x * nb;
  int64_t *bo = boff + blockIdx.x * nb;
  const int64_t per = (nb + 1023) / 1024;
  const int64_t a = threadIdx.x * per, b = min(nb, a + per);
  int64_t s = 0;
  for (int64_t x = a; x < b; ++x) s += bc[x];
  part[threadIdx.x] = s;
  __syncthreads();
  for (int off = 1; off < 1024; off <<= 1) {
    const int64_t v = threadIdx.x >= off ? part[threadIdx.x - off] : 0;
    __syncthreads();
    part[threadIdx.x] += v;
    __syncthreads();
  }
  int64_t run = part[threadIdx.x] - s;
  for (int64_t x = a; x < b; ++x) {
    bo[x] = run;
    run += bc[x];
  }
  if (threadIdx.x == 1023) total[blockIdx.x] = part[1023];
}

// Step iv over the list, and the next list: kept entries first (in order),
// then the children below the top level (in order).
__global__ void __launch_bounds__(kScanBlock) k_emit3(TreeView t, const int32_t *open, int64_t m,
                                                      uint32_t *flag, int Lm, const int64_t *boff,
                                                      const int64_t *total, int64_t nb,
                                                      int64_t n_old, int32_t *next, int32_t *lmap) {
  __shared__ int32_t wsum[3][kScanBlock / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t start = (int64_t)blockIdx.x * kScanItems;
  int64_t run0 = boff[blockIdx.x], run1 = boff[nb + blockIdx.x], run2 = boff[2 * nb + blockIdx.x];
  const int64_t keep_total = total[1];
  const uint32_t below = (1u << lane) - 1u;
  for (int rr = 0; rr < kScanRounds; ++rr) {
    int k;
    const ListSel q = list_sel(t, open, m, flag, Lm, start + (int64_t)rr * kScanBlock + threadIdx.x, k);
    const uint32_t b0 = __ballot_sync(0xffffffffu, q.f);
    const uint32_t b1 = __ballot_sync(0xffffffffu, q.keep);
    const uint32_t b2 = __ballot_sync(0xffffffffu, q.co);
    if (lane == 0) {
      wsum[0][warp] = __popc(b0);
      wsum[1][warp] = __popc(b1);
      wsum[2][warp] = __popc(b2);
    }
    __syncthreads();
    int32_t p0 = 0, p1 = 0, p2 = 0, t0 = 0, t1 = 0, t2 = 0;
#pragma unroll
    for (int w = 0; w < kScanBlock / 32; ++w) {
      const int32_t v0 = wsum[0][w], v1 = wsum[1][w], v2 = wsum[2][w];
      p0 += w < warp ? v0 : 0;
      p1 += w < warp ? v1 : 0;
      p2 += w < warp ? v2 : 0;
      t0 += v0;
      t1 += v1;
      t2 += v2;
    }
    if (q.f) {
      const int64_t c0 = n_old + 4 * (run0 + p0 + __popc(b0 & below));
      const int L = t.lvl[k] + 1, i = t.pi[k], j = t.pj[k];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        t.lvl[c0 + c] = (int8_t)L;
        t.pi[c0 + c] = 2 * i + (c & 1);
        t.pj[c0 + c] = 2 * j + (c >> 1);
        t.child[c0 + c] = -1;
        flag[c0 + c] = 0u;
      }
      t.child[k] = (int32_t)c0;
      flag[k] = 0u;
      if (q.co) {
        const int64_t r2 = keep_total + 4 * (run2 + p2 + __popc(b2 & below));
#pragma unroll
        for (int c = 0; c < 4; ++c) next[r2 + c] = (int32_t)(c0 + c);
        if (lmap) set_level_map(lmap, t.n0, L, i, j, c0);
      }
    } else if (q.keep) {
      next[run1 + p1 + __popc(b1 & below)] = k;
    }
    run0 += t0;
    run1 += t1;
    run2 += t2;
    __syncthreads();
  }
}

// ---- the sweep with counts on the device ----------------------------------
// The same steps over the sweep's open list, whose length its slot holds
// (SweepSlot::m), in two launches; grids are a few blocks per SM and loop over the items. The first flags and counts,
// the second ranks and emits: each of its blocks adds up the chunk counts in
// front of its chunk (and in all, to know the totals) from the two count
// arrays, a few kilobytes that lie in L2. (With a counting and a scanning
// launch between them a sweep took 12 us more, whatever its size.)
//
// counts: two sets (q & 1) of [flagged | below the top level][nb_cap] chunk
// counts. The set of the current sweep is zero when it starts; the emit kernel
// zeroes the other one for the next. A flag word holds its leaf's position in
// the open list (see FlagCount).

__device__ __forceinline__ FlagCount sweep_counts(uint32_t *counts, int64_t nb_cap, int set) {
  uint32_t *c = counts + 2 * nb_cap * set;
  return FlagCount{c, c + nb_cap};
}

// The first slot, the first open list (the m base pixels), flag words with
// their positions, and the counts of the first set zeroed.
__global__ void k_open_init(SweepState *S, int64_t n, int32_t *list, uint32_t *flag, int64_t m,
                            uint32_t *counts, int64_t nb_cap) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < m) {
    list[i] = (int32_t)i;
    flag[i] = (uint32_t)i << 1;
  }
  if (i < scan_chunks(m)) counts[i] = counts[nb_cap + i] = 0u;
  if (blockIdx.x == 0) {
    SweepSlot &s = S->slot[0];
    if (threadIdx.x < kMaxBands) s.ray_ctr[threadIdx.x] = 0ull;
    if (threadIdx.x == 0) {
      s.n = n;
      s.m = m;
      s.n_refined = 0;
      s.sweeps = 0;
      s.done = m == 0;
      s.missed = 0ull;
      S->fb_total = 0ull;
      S->fb_waves = 0;
    }
  }
}

// Scan and balance in one pass. No flag of the open list is set when a sweep
// starts, so a thread only ever sets flags: a leaf whose xi reaches xi_crit is
// flagged, and the thread that sets a flag -- the scan's or a balance
// expansion's -- expands it. Every flag is expanded once, and the flags reach
// the same closure as a scan of every leaf followed by the balance.
__global__ void __launch_bounds__(kScanBlock)
    k_scan_balance_dev(TreeView t, const int32_t *open, const SweepState *S,
                       int q, double xi_crit, int xi_norm, int refine_on, uint32_t *flag,
                       uint32_t *counts, int64_t nb_cap, uint32_t *err, const int32_t *lmap) {
  wait_prior_grid();
  const SweepSlot &sl = S->slot[q & 3];
  if (sl.done) return;
  const int64_t m = sl.m;
  const FlagCount fc = sweep_counts(counts, nb_cap, q & 1);
  const NodeLookup look{0, lmap};
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  __shared__ unsigned long long queue[kScanBlock / 32][kWarpQueue];
  // whole warps run the loop: a warp's 32 entries lie in one chunk
  for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); i0 < m; i0 += stride) {
    const int64_t i = i0 + (threadIdx.x & 31);
    const int k = i < m ? open[i] : 0;
    bool mine = i < m && xi_flag(t, look, k, xi_crit, xi_norm, refine_on) &&
                (atomicOr(flag + k, 1u) & 1u) == 0u;
    const bool below = mine && t.lvl[k] + 1 < t.Lm;
    const unsigned nf = __popc(__ballot_sync(0xffffffffu, mine));
    const unsigned nc = __popc(__ballot_sync(0xffffffffu, below));
    if ((threadIdx.x & 31) == 0 && nf) {
      atomicAdd(fc.flagged + i0 / kScanItems, nf);
      if (nc) atomicAdd(fc.below + i0 / kScanItems, nc);
    }
    if (lmap) {
      int L = 0, pi = 0, pj = 0;
      if (mine) {
        L = t.lvl[k];
        pi = t.pi[k];
        pj = t.pj[k];
      }
      balance_warp(t, lmap, mine, L, pi, pj, flag, err, fc, queue[threadIdx.x >> 5]);
    } else if (mine) {
      balance_from(t, look, k, flag, err, fc);
    }
  }
}

// Sums of a and b over the block (to every thread).
__device__ __forceinline__ void block_sum4(uint32_t (&v)[4], uint32_t (&sh)[4][kScanBlock / 32]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) v[q] = __reduce_add_sync(0xffffffffu, v[q]);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) {
#pragma unroll
    for (int q = 0; q < 4; ++q) sh[q][threadIdx.x >> 5] = v[q];
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    uint32_t s = 0;
#pragma unroll
    for (int w = 0; w < kScanBlock / 32; ++w) s += sh[q][w];
    v[q] = s;
  }
}

// Step iv over the list, and the next list: kept entries first (in order),
// then the children below the top level (in order). Block 0 writes the next
// slot and the host's report.
__global__ void __launch_bounds__(kScanBlock)
    k_emit3d(TreeView t, const int32_t *open, int32_t *next, SweepState *S, int q, uint32_t *flag,
             uint32_t *counts, int64_t nb_cap, const uint32_t *err, SweepReport *rep, uint32_t tag, int32_t *lmap) {
  wait_prior_grid();
  __shared__ uint32_t sums[4][kScanBlock / 32];
  __shared__ int32_t wsum[3][kScanBlock / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const SweepSlot &sl = S->slot[q & 3];
  const int done = sl.done;
  const int64_t m = sl.m, n_old = sl.n;
  if (done && blockIdx.x != 0) return;
  const int cur = q & 1;
  const FlagCount fc = sweep_counts(counts, nb_cap, cur);
  const int64_t nb = done ? 0 : scan_chunks(m);
  // totals, and the counts in front of the block's first chunk
  uint32_t v[4] = {0u, 0u, 0u, 0u};
  for (int64_t x = threadIdx.x; x < nb; x += kScanBlock) {
    const uint32_t a = fc.flagged[x], b = fc.below[x];
    v[0] += a;
    v[1] += b;
    if (x < blockIdx.x) {
      v[2] += a;
      v[3] += b;
    }
  }
  block_sum4(v, sums);
  const int64_t nflag = v[0], nbelow = v[1], keep_total = m - nflag;
  if (blockIdx.x == 0) {
    SweepSlot &sn = S->slot[(q + 1) & 3];
    if (threadIdx.x < kMaxBands) sn.ray_ctr[threadIdx.x] = 0ull;
    if (threadIdx.x == 0) {
      const int64_t m1 = keep_total + 4 * nbelow;
      const int sweeps = sl.sweeps + (nflag ? 1 : 0);
      const int end = done || nflag == 0 || m1 == 0;  // flagged nothing, or no leaf is left to scan
      const int64_t n1 = n_old + 4 * nflag, refined = sl.n_refined + nflag;
      sn.n = n1;
      sn.m = m1;
      sn.n_refined = refined;
      sn.sweeps = sweeps;
      sn.done = end;
      sn.missed = 0ull;
      SweepReport &r = rep[q & 3];
      r.n = n1;
      r.n_refined = refined;
      r.sweeps = sweeps;
      r.done = end;
      r.err = *err;
      __threadfence_system();
      *(volatile unsigned long long *)&r.progress = ((unsigned long long)tag << 32) | (unsigned)(q + 1);
    }
  }
  if (nflag == 0) return;
  // the other set of counts, for the next sweep's list
  {
    const FlagCount fo = sweep_counts(counts, nb_cap, cur ^ 1);
    const int64_t nn = scan_chunks(keep_total + 4 * nbelow);
    for (int64_t x = (int64_t)blockIdx.x * kScanBlock + threadIdx.x; x < nn; x += (int64_t)gridDim.x * kScanBlock)
      fo.flagged[x] = fo.below[x] = 0u;
  }
  int64_t front0 = v[2], front2 = v[3];  // flagged, below: entries before chunk c
  const uint32_t below = (1u << lane) - 1u;
  for (int64_t c = blockIdx.x; c < nb; c += gridDim.x) {
    const int64_t start = c * kScanItems;
    int64_t run0 = front0, run1 = start - front0, run2 = front2;
    for (int rr = 0; rr < kScanRounds; ++rr) {
      const int64_t at = start + (int64_t)rr * kScanBlock + threadIdx.x;
      int k = 0;
      bool f = false, co = false;
      if (at < m) {
        k = open[at];
        f = (flag[k] & 1u) != 0u;
      }
      const bool keep = at < m && !f;
      // a flagged node's fields, loaded before the ranks are formed
      int L = 0, i = 0, j = 0;
      if (f) {
        L = t.lvl[k] + 1;
        i = t.pi[k];
        j = t.pj[k];
        co = L < t.Lm;
      }
      const uint32_t b0 = __ballot_sync(0xffffffffu, f);
      const uint32_t b1 = __ballot_sync(0xffffffffu, keep);
      const uint32_t b2 = __ballot_sync(0xffffffffu, co);
      if (lane == 0) {
        wsum[0][warp] = __popc(b0);
        wsum[1][warp] = __popc(b1);
        wsum[2][warp] = __popc(b2);
      }
      __syncthreads();
      int32_t p0 = 0, p1 = 0, p2 = 0, t0 = 0, t1 = 0, t2 = 0;
#pragma unroll
      for (int w = 0; w < kScanBlock / 32; ++w) {
        const int32_t v0 = wsum[0][w], v1 = wsum[1][w], v2 = wsum[2][w];
        p0 += w < warp ? v0 : 0;
        p1 += w < warp ? v1 : 0;
        p2 += w < warp ? v2 : 0;
        t0 += v0;
        t1 += v1;
        t2 += v2;
      }
      if (f) {
        const int64_t c0 = n_old + 4 * (run0 + p0 + __popc(b0 & below));
        const int64_t r2 = keep_total + 4 * (run2 + p2 + __popc(b2 & below));
#pragma unroll
        for (int ch = 0; ch < 4; ++ch) {
          t.lvl[c0 + ch] = (int8_t)L;
          t.pi[c0 + ch] = 2 * i + (ch & 1);
          t.pj[c0 + ch] = 2 * j + (ch >> 1);
          t.child[c0 + ch] = -1;
          flag[c0 + ch] = co ? (uint32_t)(r2 + ch) << 1 : 0u;
        }
        t.child[k] = (int32_t)c0;
        flag[k] = 0u;
        if (co) {
#pragma unroll
          for (int ch = 0; ch < 4; ++ch) next[r2 + ch] = (int32_t)(c0 + ch);
          if (lmap) set_level_map(lmap, t.n0, L, i, j, c0);
        }
      } else if (keep) {
        const int64_t r1 = run1 + p1 + __popc(b1 & below);
        next[r1] = k;
        flag[k] = (uint32_t)r1 << 1;
      }
      run0 += t0;
      run1 += t1;
      run2 += t2;
      __syncthreads();
    }
    if (c + gridDim.x < nb) {  // the counts up to the block's next chunk
      uint32_t w4[4] = {0u, 0u, 0u, 0u};
      for (int64_t x = c + threadIdx.x; x < c + gridDim.x; x += kScanBlock) {
        w4[0] += fc.flagged[x];
        w4[1] += fc.below[x];
      }
      block_sum4(w4, sums);
      front0 += w4[0];
      front2 += w4[1];
    }
  }
}

// Step vi: copy the selected nodes (leaves, or all) to the output arrays.

// The fields of every round's node are loaded before the ranks are formed,
// so their latency overlaps the block's ballots and barriers. The leaves in
// front of the block are those of the flux blocks before it and of the chunks
// before it within its flux block (counts of k_flux_partial). The former are
// added up here, or, above kFluxDirect flux blocks, read from their prefix sums
// block_off. (A counting and a scanning launch of their own took 25 us for 7.7 M
// nodes; but every block adding up all the counts before it is quadratic work.)
__global__ void __launch_bounds__(kScanBlock) k_emit_out(TreeView t, OutView o, int all, int64_t n,
                                                         const int32_t *chunk_leaves,
                                                         const int32_t *block_leaves,
                                                         const int64_t *block_off) {
  wait_prior_grid();
  __shared__ int32_t wsum[kScanBlock / 32];
  __shared__ uint32_t fsum[kScanBlock / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t start = (int64_t)blockIdx.x * kScanItems;
  uint32_t front = 0;
  if (!all) {
    const int fb = blockIdx.x / kFluxChunks, c0 = fb * kFluxChunks;
    if (!block_off)
      for (int x = threadIdx.x; x < fb; x += kScanBlock) front += (uint32_t)block_leaves[x];
    else if (threadIdx.x == kScanBlock - 1)
      front = (uint32_t)block_off[fb];  // (at most 2^31 nodes)
    if (c0 + (int)threadIdx.x < (int)blockIdx.x) front += (uint32_t)chunk_leaves[c0 + threadIdx.x];
    front = __reduce_add_sync(0xffffffffu, front);
    if (lane == 0) fsum[warp] = front;
  }
  bool sel[kScanRounds];
  int lv[kScanRounds], pi[kScanRounds], pj[kScanRounds], cl[kScanRounds];
  float N[kScanRounds], P[kScanRounds], I0[kScanRounds];
#pragma unroll
  for (int rr = 0; rr < kScanRounds; ++rr) {
    const int64_t k = start + (int64_t)rr * kScanBlock + threadIdx.x;
    sel[rr] = false;
    if (k < n) {
      cl[rr] = t.child[k];
      sel[rr] = all || cl[rr] < 0;
      lv[rr] = t.lvl[k];
      pi[rr] = t.pi[k];
      pj[rr] = t.pj[k];
      N[rr] = t.N[k];
      P[rr] = t.p[k];
      I0[rr] = o.I ? t.I[k] : 0.f;  // no tree intensities are read without o.I
    }
  }
  int64_t run = start;
  if (!all) {
    __syncthreads();
    uint32_t f = 0;
#pragma unroll
    for (int w = 0; w < kScanBlock / 32; ++w) f += fsum[w];
    run = f;
  }
#pragma unroll
  for (int rr = 0; rr < kScanRounds; ++rr) {
    const int64_t k = start + (int64_t)rr * kScanBlock + threadIdx.x;
    const uint32_t bal = __ballot_sync(0xffffffffu, sel[rr]);
    if (lane == 0) wsum[warp] = __popc(bal);
    __syncthreads();
    int32_t before = 0, tot = 0;
#pragma unroll
    for (int w = 0; w < kScanBlock / 32; ++w) {
      const int32_t v = wsum[w];
      before += w < warp ? v : 0;
      tot += v;
    }
    if (sel[rr]) {
      const int64_t r = run + before + __popc(bal & ((1u << lane) - 1u));
      if (o.level) o.level[r] = lv[rr];
      if (o.i) o.i[r] = pi[rr];
      if (o.j) o.j[r] = pj[rr];
      if (o.is_leaf) o.is_leaf[r] = cl[rr] < 0;
      if (o.N) o.N[r] = N[rr];
      if (o.p) o.p[r] = P[rr];
      if (o.I) {
        o.I[r] = I0[rr];
#pragma unroll 4
        for (int b = 1; b < o.n_bands; ++b) o.I[(int64_t)b * o.stride + r] = t.I[(int64_t)b * t.cap + k];
      }
    }
    run += tot;
    __syncthreads();
  }
}

// Base image, row-major: node j*n0 + i.
__global__ void k_init_base(TreeView t) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t n = (int64_t)t.n0 * t.n0;
  if (k >= n) return;
  t.lvl[k] = 0;
  t.pi[k] = (int32_t)(k % t.n0);
  t.pj[k] = (int32_t)(k / t.n0);
  t.child[k] = -1;
}

// ---- band flux and step count --------------------------------------------
// Per block: sum over selected pixels of I_b x 4^-level in FP64, times area0,
// and of the step counts (integers); a second kernel adds the block partials
// of each band in a fixed order (strided per thread, then a tree), so the
// result does not depend on scheduling.
//
// A block takes kFluxPerBlock entries and kFluxBands bands (blockIdx.y; the last
// row of blocks sums the step counts): leaf flags and levels are read once for
// the bands of a block, and bands run beside one another. (One block summed
// every band of 8192 entries, band after band, before: 85 us for 0.8 M leaves
// of four bands.)
__global__ void __launch_bounds__(256) k_flux_partial(FluxArgs a) {
  wait_prior_grid();
  __shared__ int32_t chunk_sum[kFluxChunks];
  __shared__ double sh[kFluxBands][8];
  __shared__ unsigned long long shs[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t start = (int64_t)blockIdx.x * kFluxPerBlock;
  const int64_t end = min(a.n, start + kFluxPerBlock);
  double *outp = a.partial + (int64_t)blockIdx.x * (a.n_bands + 1);
  const int b0 = blockIdx.y * kFluxBands;
  if (b0 >= a.n_bands) {
    unsigned long long st = 0;
    for (int64_t k = start + threadIdx.x; k < end; k += blockDim.x) st += a.steps[k];
    for (int off = 16; off > 0; off >>= 1) st += __shfl_xor_sync(0xffffffffu, st, off);
    if (lane == 0) shs[warp] = st;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < 8; ++w) st += shs[w];
      outp[0] = (double)st;
    }
    return;
  }
  float hi[kFluxBands], lo[kFluxBands];
  double rest[kFluxBands];
#pragma unroll
  for (int q = 0; q < kFluxBands; ++q) {
    hi[q] = lo[q] = 0.f;
    rest[q] = 0.0;
  }
  // four entries per thread at a time, their loads issued together (a leaf's
  // intensity is not made to wait for its flag)
  constexpr int R = 4;
  const bool count = a.chunk_leaves && b0 == 0;
  if (count) {
    if (threadIdx.x < kFluxChunks) chunk_sum[threadIdx.x] = 0;
    __syncthreads();
  }
  for (int64_t k0 = start + threadIdx.x; k0 - threadIdx.x < end; k0 += R * blockDim.x) {
    bool leaf[R];
    int L[R];
    float I[R][kFluxBands];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int64_t k = k0 + r * blockDim.x;
      const bool in = k < end;
      leaf[r] = in && (!a.child || a.child[k] < 0);
      L[r] = in && a.lvl ? a.lvl[k] : 0;
#pragma unroll
      for (int q = 0; q < kFluxBands; ++q)
        I[r][q] = in && b0 + q < a.n_bands ? a.I[(int64_t)(b0 + q) * a.stride + k] : 0.f;
    }
    if (count) {
#pragma unroll
      for (int r = 0; r < R; ++r) {  // 256 nodes of a round lie in one chunk
        const int c = __popc(__ballot_sync(0xffffffffu, leaf[r]));
        if (lane == 0 && c) atomicAdd(&chunk_sum[(int)(k0 + r * blockDim.x - start) / kScanItems], c);
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r)
      if (leaf[r]) {
#pragma unroll
        for (int q = 0; q < kFluxBands; ++q)
          if (b0 + q < a.n_bands) flux_add(I[r][q], L[r], hi[q], lo[q], rest[q]);
      }
  }
#pragma unroll
  for (int q = 0; q < kFluxBands; ++q)
    if (b0 + q < a.n_bands) rest[q] += (double)hi[q] + (double)lo[q];
  const double s4 = flux_warp_sum(rest);
  if ((lane & 7) == 0) sh[lane >> 3][warp] = s4;
  __syncthreads();
  if (count) {
    const int nc = (int)((end - start + kScanItems - 1) / kScanItems);
    if (threadIdx.x < nc) a.chunk_leaves[(int64_t)blockIdx.x * kFluxChunks + threadIdx.x] = chunk_sum[threadIdx.x];
    if (threadIdx.x == 32) {
      int s = 0;
      for (int c = 0; c < nc; ++c) s += chunk_sum[c];
      a.block_leaves[blockIdx.x] = s;
    }
  }
  if (threadIdx.x < kFluxBands && b0 + (int)threadIdx.x < a.n_bands) {
    double s = sh[threadIdx.x][0];
    for (int w = 1; w < 8; ++w) s += sh[threadIdx.x][w];
    outp[b0 + threadIdx.x + 1] = s * a.area0;
  }
}

// One block per output: block 0 the step count, block b + 1 band b. The host
// reads its copy in page-locked memory once the stream has been waited for (a
// copy of its own behind the kernel cost 4 us per image).
__global__ void __launch_bounds__(256) k_flux_final(FluxArgs a, int64_t nblocks) {
  wait_prior_grid();
  __shared__ double sh[8];
  const int b = (int)blockIdx.x - 1;
  double s = 0.0;
  for (int64_t x = threadIdx.x; x < nblocks; x += blockDim.x) s += a.partial[x * (a.n_bands + 1) + b + 1];
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) s += sh[w];
    a.host[b < 0 ? a.n_bands : b] = s;
    if (b >= 0 && a.flux) a.flux[b] = s;
  }
}

// ---- host launchers ----------------------------------------------------------

static inline unsigned nblk(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

cudaError_t launch_init_base(const TreeView &t, cudaStream_t st) {
  const int64_t n = (int64_t)t.n0 * t.n0;
  k_init_base<<<nblk(n, 256), 256, 0, st>>>(t);
  return cudaGetLastError();
}

int sm_count() {
  static std::atomic<int> sms{0};
  int n = sms.load(std::memory_order_relaxed);
  if (n == 0) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) {
      cudaGetLastError();
      n = 1;
    }
    sms.store(n, std::memory_order_relaxed);
  }
  return n;
}

// Blocks for a grid-stride launch: enough for `per_sm` blocks on every SM.
static unsigned stride_blocks(int64_t n, int block, int per_sm) {
  const int64_t cap = (int64_t)sm_count() * per_sm;
  const int64_t need = (n + block - 1) / block;
  return (unsigned)(need < cap ? need : cap);
}

int64_t scan_blocks(int64_t n) { return scan_chunks(n); }

cudaError_t launch_list_init(int32_t *list, int64_t m, cudaStream_t st) {
  if (m <= 0) return cudaSuccess;
  k_iota<<<nblk(m, 256), 256, 0, st>>>(list, m);
  return cudaGetLastError();
}

cudaError_t launch_list_scan(const TreeView &t, const int32_t *open, int64_t m, double xi_crit,
                             int xi_norm, int refine_on, uint32_t *flag, cudaStream_t st,
                             const int32_t *lmap) {
  if (m <= 0) return cudaSuccess;
  k_xi_scan_list<<<nblk(m, 256), 256, 0, st>>>(t, open, m, xi_crit, xi_norm, refine_on, flag, lmap);
  return cudaGetLastError();
}

cudaError_t launch_list_balance(const TreeView &t, const int32_t *open, int64_t m, uint32_t *flag,
                                uint32_t *err, cudaStream_t st, const int32_t *lmap) {
  if (m <= 0) return cudaSuccess;
  k_balance_list<<<stride_blocks(m, 128, 16), 128, 0, st>>>(t, open, m, flag, err, lmap);
  return cudaGetLastError();
}

cudaError_t launch_list_count(const TreeView &t, const int32_t *open, int64_t m,
                              const uint32_t *flag, int32_t *bcount, int64_t *boff,
                              int64_t *totals, cudaStream_t st) {
  const int64_t nb = scan_blocks(m);
  if (nb == 0) return cudaMemsetAsync(totals, 0, 3 * sizeof(int64_t), st);
  k_count3<<<(unsigned)nb, kScanBlock, 0, st>>>(t, open, m, flag, t.Lm, bcount, nb);
  k_scan_blocks3<<<3, 1024, 0, st>>>(bcount, nb, boff, totals);
  return cudaGetLastError();
}

cudaError_t launch_list_emit(const TreeView &t, const int32_t *open, int64_t m, uint32_t *flag,
                             const int64_t *boff, const int64_t *totals, int64_t n_old,
                             int32_t *next, cudaStream_t st, int32_t *lmap) {
  const int64_t nb = scan_blocks(m);
  if (nb == 0) return cudaSuccess;
  k_emit3<<<(unsigned)nb, kScanBlock, 0, st>>>(t, open, m, flag, t.Lm, boff, totals, nb, n_old, next, lmap);
  return cudaGetLastError();
}

cudaError_t launch_count_flags(const uint32_t *flag, int64_t n, int32_t *bcount, int64_t *boff,
                               int64_t *total, cudaStream_t st) {
  const int64_t nb = scan_blocks(n);
  if (nb == 0) return cudaMemsetAsync(total, 0, sizeof(int64_t), st);
  k_count<<<(unsigned)nb, kScanBlock, 0, st>>>(PredFlag{flag}, n, bcount);
  k_scan_blocks<<<1, 1024, 0, st>>>(bcount, nb, boff, total);
  return cudaGetLastError();
}

cudaError_t launch_scan_offsets(const int32_t *bcount, int64_t nb, int64_t *boff, int64_t *total,
                                cudaStream_t st) {
  if (nb == 0) return cudaMemsetAsync(total, 0, sizeof(int64_t), st);
  k_scan_blocks<<<1, 1024, 0, st>>>(bcount, nb, boff, total);
  return cudaGetLastError();
}


bool emit_out_scans(int all, int64_t n) { return !all && flux_blocks(n) > kFluxDirect; }

cudaError_t launch_emit_out(const TreeView &t, const OutView &o, int all, int64_t n,
                            const int32_t *chunk_leaves, const int32_t *block_leaves, int64_t *block_off,
                            int64_t *total, cudaStream_t st) {
  const int64_t nb = scan_blocks(n);
  if (nb == 0) return cudaSuccess;
  const bool scan = emit_out_scans(all, n);
  if (scan) {
    k_scan_blocks<<<1, 1024, 0, st>>>(block_leaves, flux_blocks(n), block_off, total);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return launch_pdl(k_emit_out, dim3((unsigned)nb), dim3(kScanBlock), 0, st, t, o, all, n, chunk_leaves,
                    block_leaves, (const int64_t *)(scan ? block_off : nullptr));
}

// Blocks of the device-count sweep kernels: a few per SM, looping over items.
static unsigned sweep_blocks(int per_sm) { return (unsigned)(sm_count() * per_sm); }

cudaError_t launch_open_init(SweepState *S, int64_t n, int32_t *list, uint32_t *flag, int64_t m,
                             uint32_t *counts, int64_t nb_cap, cudaStream_t st) {
  k_open_init<<<nblk(std::max<int64_t>(m, 1), 256), 256, 0, st>>>(S, n, list, flag, m, counts, nb_cap);
  return cudaGetLastError();
}

cudaError_t launch_sweep_scan_balance(const TreeView &t, int32_t *const open[2],
                                      const SweepState *S, int q, double xi_crit, int xi_norm,
                                      int refine_on, uint32_t *flag, uint32_t *counts,
                                      int64_t nb_cap, uint32_t *err, cudaStream_t st,
                                      const int32_t *lmap) {
  return launch_pdl(k_scan_balance_dev, dim3(sweep_blocks(8)), dim3(kScanBlock), 0, st, t,
                    (const int32_t *)open[q & 1], S, q, xi_crit, xi_norm, refine_on, flag, counts,
                    nb_cap, err, lmap);
}

cudaError_t launch_sweep_emit(const TreeView &t, int32_t *const open[2], SweepState *S, int q,
                              uint32_t *flag, uint32_t *counts, int64_t nb_cap,
                              const uint32_t *err, SweepReport *rep, uint32_t tag, cudaStream_t st,
                              int32_t *lmap) {
  return launch_pdl(k_emit3d, dim3(sweep_blocks(8)), dim3(kScanBlock), 0, st, t,
                    (const int32_t *)open[q & 1], open[(q + 1) & 1], S, q, flag, counts, nb_cap, err,
                    rep, tag, lmap);
}

int64_t flux_blocks(int64_t n) { return n <= 0 ? 0 : (n + kFluxPerBlock - 1) / kFluxPerBlock; }

cudaError_t launch_flux_partial(const FluxArgs &a, cudaStream_t st) {
  const int64_t nb = flux_blocks(a.n);
  if (nb == 0) return cudaSuccess;
  const unsigned rows = (unsigned)((a.n_bands + kFluxBands - 1) / kFluxBands) + 1;
  return launch_pdl(k_flux_partial, dim3((unsigned)nb, rows), dim3(256), 0, st, a);
}

cudaError_t launch_flux_final(const FluxArgs &a, cudaStream_t st) {
  return launch_pdl(k_flux_final, dim3((unsigned)(a.n_bands + 1)), dim3(256), 0, st, a, flux_blocks(a.n));
}

}  // namespace air
