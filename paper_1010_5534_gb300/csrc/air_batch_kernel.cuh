// air_batch_kernel.cuh -- the batched persistent kernel and its launch, as
// templates over the bands one thread carries; each width is compiled in a
// translation unit of its own (air_batch_<width>.cu). See air_batch.cu.
#pragma once
#include "air_handle.cuh"
#include "air_march.cuh"
#include "air_tree.cuh"

namespace air {

typedef cudaError_t (*BatchOccFn)(int *, size_t);

constexpr int kBatchBlock = 128;
constexpr int kBatchMaxViews = 256;
constexpr uint32_t kErrBalance = 1u, kErrTimeout = 2u, kErrCapacity = 4u;

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Grid barrier with a time limit. `expected` arrivals release it.
static __device__ bool grid_sync(BatchCtl *ctl, unsigned expected, long long timeout_ns) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    ok = 1;
    volatile unsigned *genp = &ctl->bar_gen;
    const unsigned gen = *genp;
    __threadfence();
    const unsigned arrived = atomicAdd(&ctl->bar_count, 1u) + 1u;
    if (arrived == expected) {
      atomicExch(&ctl->bar_count, 0u);
      __threadfence();
      atomicAdd(&ctl->bar_gen, 1u);
    } else {
      const unsigned long long t0 = global_ns();
      while (*genp == gen) {
        if ((long long)(global_ns() - t0) > timeout_ns) {
          atomicOr(&ctl->err, kErrTimeout);
          ok = 0;
          break;
        }
        __nanosleep(128);
      }
    }
    __threadfence();
  }
  __syncthreads();
  return ok != 0;
}

// Items [s0, s1) of one block, in rounds of blockDim. For every selected item
// k of view v: emit(k, v, run[v] + rank), rank = selected items of view v
// before k in the block's range. run[] (shared, V entries) advances per round.
template <class Pred, class Emit>
__device__ void block_emit_by_view(const Pred &pred, const int16_t *__restrict__ view, Emit &emit,
                                   int64_t s0, int64_t s1, int V, int64_t *run, int32_t *wcnt) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int64_t r0 = s0; r0 < s1; r0 += blockDim.x) {
    for (int x = threadIdx.x; x < nw * V; x += blockDim.x) wcnt[x] = 0;
    __syncthreads();
    const int64_t k = r0 + threadIdx.x;
    const bool sel = k < s1 && pred(k);
    const int v = sel ? (int)view[k] : -1;
    const unsigned m = __match_any_sync(0xffffffffu, v);
    const int rank_w = __popc(m & ((1u << lane) - 1u));
    if (sel && rank_w == 0) wcnt[warp * V + v] = __popc(m);
    __syncthreads();
    if (sel) {
      int64_t before = 0;
      for (int w = 0; w < warp; ++w) before += wcnt[w * V + v];
      emit(k, v, run[v] + before + rank_w);
    }
    __syncthreads();
    for (int vv = threadIdx.x; vv < V; vv += blockDim.x) {
      int64_t s = 0;
      for (int w = 0; w < nw; ++w) s += wcnt[w * V + vv];
      run[vv] += s;
    }
    __syncthreads();
  }
}

struct FlagPred {
  const uint32_t *flag;
  __device__ bool operator()(int64_t k) const { return flag[k] != 0; }
};

struct EmitChildrenV {
  TreeView t;
  int16_t *view;
  const int64_t *vbase;  // shared: first child slot of each view this sweep
  __device__ void operator()(int64_t k, int v, int64_t rank) {
    const int64_t c0 = vbase[v] + 4 * rank;
    const int L = t.lvl[k] + 1, i = t.pi[k], j = t.pj[k];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      t.lvl[c0 + c] = (int8_t)L;
      t.pi[c0 + c] = 2 * i + (c & 1);
      t.pj[c0 + c] = 2 * j + (c >> 1);
      t.child[c0 + c] = -1;
      view[c0 + c] = (int16_t)v;
    }
    t.child[k] = (int32_t)c0;
  }
};

// Table and constants of a band chunk of `width` (the wide form, NBT = 0) or NBT bands.
template <int NBT>
__host__ __device__ __forceinline__ size_t batch_tab_bytes(bool table, int n_tbins, int width) {
  if constexpr (NBT == 0) return wide_tab_bytes(table, n_tbins, width);
  else return chunk_bytes<NBT>(table, n_tbins);
}

// Shared memory of a block: the tables of `tabs` band chunks, the sums of the
// wide form, and the per-view counters.
template <int NBT>
static size_t batch_smem(const GridView &g, int V, int width, int tabs) {
  const size_t tab = tabs * batch_tab_bytes<NBT>(g.cell_fmt == kCellXq, g.n_tbins, width) +
                     (NBT == 0 ? wide_sum_bytes(width, kBatchBlock) : 0);
  return tab + 3 * sizeof(int64_t) * V + sizeof(int32_t) * V + sizeof(int32_t) * (kBatchBlock / 32) * V;
}

// DIR: 0 for any views, -2 when every view is inclined (trace_ray): without the
// column march of axis rays, which holds a chunk's band constants and partial
// sums in registers, a thread needs 124 registers instead of 168 at 8 bands.
// (Inclined views with 16 bands per thread take the wide form.)
constexpr int kBatchWideBlocks = 4;
template <int NBT, int DIR>
struct BatchBlocks {
  static constexpr int value = NBT == 0 ? kBatchWideBlocks : NBT <= 2 ? 5 : (NBT <= 4 ? 4 : (NBT <= 8 ? (DIR == 0 ? 3 : 4) : 2));
};

// Band chunks whose tables a block holds. All of them, filled once, where the
// form's resident blocks then still fit an SM's shared memory; else one at a
// time, filled again whenever the block's warps go on to the next chunk. (8
// inclined views, 255 table bins, every chunk held: 32 bands 10.5 ms with two
// blocks per SM, 64 bands 29.7 with one; one at a time 8.5 and 13.8. Mixed
// views 16.8 and 46.3, 13.7 and 25.4. 64 bins: 7.7 and 12.9, 13.7 and 25.7.
// Groups of as many tables as fit, one group at a time: 8.4 and 13.7, but 14.8
// and 27.7 for mixed views.)
constexpr size_t kSmShared = 228 * 1024, kBlockReserve = 1024;  // of an SM; taken per block
template <int NBT, int DIR>
static int batch_tables(const GridView &g, int V, int width) {
  const int chunks = NBT == 0 ? (g.n_bands + width - 1) / width : (g.n_bands + NBT - 1) / (NBT > 0 ? NBT : 1);
  auto blocks = [&](int tabs) {
    return std::min<size_t>(BatchBlocks<NBT, DIR>::value,
                            kSmShared / (batch_smem<NBT>(g, V, width, tabs) + kBlockReserve));
  };
  return blocks(chunks) >= blocks(1) ? chunks : 1;
}

// Where a traced ray's values go.
struct BatchOut {
  float *N, *I, *p;
  uint32_t *steps;
  uint8_t *maxlev;  // or NULL
  int64_t stride;
};

// Part `part` of band chunk `chunk` of the ray of pixel (L, i, j), to entry k.
// `all`: the part is the only one.
template <int NBT, bool AMR, int FMT, int DIR>
__device__ __forceinline__ void batch_trace(const BatchArgs &a, unsigned char *sm, const RayGeom &rg, int L,
                                            int i, int j, int chunk, int part, int parts, bool all,
                                            const BatchOut &o, int64_t k) {
  const GridView &g = a.g;
  if constexpr (NBT == 0) {
    const size_t tab = batch_tab_bytes<0>(FMT == kCellXq, g.n_tbins, a.width);
    int b0;
    const int c0 = chunk * a.width, slot = a.tabs > 1 ? chunk : 0;
    const WideCtx wc = wide_ctx<FMT>(sm + slot * tab, reinterpret_cast<float4 *>(sm + a.tabs * tab), a.width,
                                     min(a.width, g.n_bands - c0), part, parts, &b0);
    b0 += c0;
    if (wc.pairs <= 0) return;
    RTState<0> st;
    trace_wide<AMR, FMT>(st, g, rg, L, i, j, a.fp64_level, wc);
    if (b0 == 0) {
      o.N[k] = st.N;
      o.steps[k] = st.steps;
      if (o.maxlev) o.maxlev[k] = (uint8_t)st.maxlev;
    }
    float p = 0.f;
    for (int q = 0; q < wc.pairs; ++q) {
      const float4 s = wc.sums[q * blockDim.x];
      float *I = o.I + (int64_t)(b0 + 2 * q) * o.stride + k;
      I[0] = s.x;
      p += s.x;
      if (2 * q + 1 < wc.nbh) {
        I[o.stride] = s.z;
        p += s.z;
      }
    }
    if (all) o.p[k] = p;
  } else {
    const int b0 = chunk * NBT;
    const int slot = a.tabs > 1 ? chunk : 0;
    const BandCtx bc = chunk_ctx<NBT, FMT>(sm + slot * chunk_bytes<NBT>(FMT == kCellXq, g.n_tbins), g,
                                           min(NBT, g.n_bands - b0));
    BandRegs<NBT> br;
    band_regs<NBT, FMT>(br, bc);
    RTState<NBT> st;
    trace_ray<NBT, AMR, FMT, DIR>(st, g, rg, L, i, j, a.fp64_level, bc, br);
    if (chunk == 0) {
      o.N[k] = st.N;
      o.steps[k] = st.steps;
      if (o.maxlev) o.maxlev[k] = (uint8_t)st.maxlev;
    }
#pragma unroll
    for (int c = 0; c < NBT; ++c)
      if (c < bc.nbh) o.I[(int64_t)(b0 + c) * o.stride + k] = st.I[c];
    if (all) {
      float p = 0.f;
#pragma unroll
      for (int c = 0; c < NBT; ++c)
        if (c < bc.nbh) p += st.I[c];
      o.p[k] = p;
    }
  }
}

// Table and constants of chunk `chunk` at `sm`, by the block.
template <int NBT, int FMT>
__device__ __forceinline__ void batch_fill(const BatchArgs &a, unsigned char *sm, int chunk) {
  if constexpr (NBT == 0) wide_fill<FMT>(sm, a.g, chunk * a.width, a.width);
  else chunk_fill<NBT, FMT>(sm, a.g, chunk * NBT);
}

// The work of one phase: `items` items (rays x parts) of every band chunk, from
// the chunks' queues; a warp takes rpw at a time. body(chunk, item), lane by
// lane. With one table per block, the block goes from chunk to chunk together,
// beginning with the chunk whose table it holds (`held`; another one in every
// block at first, so the chunks of a phase of few rays are traced side by side)
// and leaving out chunks whose queues are empty by then. Every thread of the
// block calls this.
template <int NBT, int FMT, class Body>
__device__ __forceinline__ void batch_queue(const BatchArgs &a, unsigned char *sm, unsigned long long items,
                                            int rpw, int &held, const Body &body) {
  const int lane = threadIdx.x & 31, from = held;
  for (int i = 0; i < a.chunks; ++i) {
    const int chunk = from + i < a.chunks ? from + i : from + i - a.chunks;
    auto take = [&] {
      unsigned long long b = 0;
      if (lane == 0) b = atomicAdd(&a.ctl->q_head[chunk], (unsigned long long)rpw);
      return __shfl_sync(0xffffffffu, b, 0);
    };
    unsigned long long b = take();
    if (a.tabs < a.chunks) {
      if (!__syncthreads_or(b < items)) continue;
      if (chunk != held) {
        batch_fill<NBT, FMT>(a, sm, chunk);
        held = chunk;
        __syncthreads();
      }
    }
    for (; b < items; b = take()) {
      const unsigned long long it = lane < rpw ? b + lane : items;
      if (it < items) body(chunk, it);
    }
  }
}

template <int NBT, bool AMR, int FMT, int DIR>
__global__ void __launch_bounds__(kBatchBlock, BatchBlocks<NBT, DIR>::value) k_air_batch(BatchArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const GridView &g = a.g;
  const int V = a.V, nb = g.n_bands;
  const size_t tab = batch_tab_bytes<NBT>(FMT == kCellXq, g.n_tbins, a.width);
  int held = 0;  // where a block holds one table: its chunk
  if (a.tabs == a.chunks) {
    for (int c = 0; c < a.chunks; ++c) batch_fill<NBT, FMT>(a, smem_raw + c * tab, c);
  } else {
    held = (int)(blockIdx.x % (unsigned)a.chunks);
    batch_fill<NBT, FMT>(a, smem_raw, held);
  }
  const size_t tab_end = a.tabs * tab + (NBT == 0 ? wide_sum_bytes(a.width, kBatchBlock) : 0);
  int64_t *run = (int64_t *)(smem_raw + tab_end);
  int64_t *tot = run + V;
  int64_t *vbase = tot + V;
  int32_t *cnt = (int32_t *)(vbase + V);
  int32_t *wcnt = cnt + V;
  __shared__ int64_t s_total;
  __syncthreads();

  const TreeView t = a.t;
  const int n0 = t.n0;
  const int64_t nn0 = (int64_t)n0 * n0;
  const int64_t gtid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t gstride = (int64_t)gridDim.x * blockDim.x;
  const unsigned nblk = gridDim.x;

  // step i: the base image of every view, view-major, row-major within a view
  // (mode 2 continues from the base images a mode-1 launch traced)
  const int64_t nbase = (int64_t)V * nn0;
  if (a.mode != 2) {
    for (int64_t k = gtid; k < nbase; k += gstride) {
      const int v = (int)(k / nn0);
      const int64_t r = k - (int64_t)v * nn0;
      t.lvl[k] = 0;
      t.pi[k] = (int32_t)(r % n0);
      t.pj[k] = (int32_t)(r / n0);
      t.child[k] = -1;
      a.view[k] = (int16_t)v;
    }
    if (!grid_sync(a.ctl, nblk + (a.stall ? 1u : 0u), a.timeout_ns)) return;
  }

  int64_t first = a.mode == 2 ? nbase : 0, n = nbase;
  if (a.mode == 2 && a.P > 0) {
    // the proposal wave of every view: (ray, band chunk) items from the queue
    const int parts = NBT == 0 ? wide_parts(a.P * a.chunks, min(a.width, nb), a.fill) : 1;
    const BatchOut o{a.pN, a.pI, a.pp, a.psteps, nullptr, a.P};
    const int rpw = rays_per_warp(a.P, a.chunks * parts, (int64_t)nblk * (kBatchBlock / 32));
    batch_queue<NBT, FMT>(a, smem_raw, (unsigned long long)a.P * parts, rpw, held, [&](int chunk, unsigned long long it) {
      const int part = parts == 1 ? 0 : (int)(it / (unsigned long long)a.P);
      const int64_t q = (int64_t)(it - (unsigned long long)part * a.P);
      batch_trace<NBT, AMR, FMT, DIR>(a, smem_raw, a.geoms[a.pview[q]], a.plvl[q], a.ppi[q], a.ppj[q], chunk, part,
                                      parts, a.chunks * parts == 1, o, q);
    });
    // (the band sums of rays dealt to parts of one chunk: those of several
    // chunks are formed where the pixels take their values)
    if (a.chunks == 1 && parts > 1) {
      if (!grid_sync(a.ctl, nblk, a.timeout_ns)) return;
      for (int64_t k = gtid; k < a.P; k += gstride) {
        float s = 0.f;
        for (int q = 0; q < nb; ++q) s += a.pI[(int64_t)q * a.P + k];
        a.pp[k] = s;
      }
    }
    if (!grid_sync(a.ctl, nblk, a.timeout_ns)) return;
    if (blockIdx.x == 0 && threadIdx.x < a.chunks) a.ctl->q_head[threadIdx.x] = 0ull;
  }
  int sweep = 0;
  for (;; ++sweep) {
    // step ii: trace the rays added last sweep, all views and band chunks
    const int64_t cnt_r = n - first;
    const int parts = NBT == 0 ? wide_parts(cnt_r * a.chunks, min(a.width, nb), a.fill) : 1;
    const int shares = a.chunks * parts;
    const BatchOut o{t.N, t.I, t.p, t.steps, a.mode == 1 ? a.maxlev : nullptr, t.cap};
    const int rpw = rays_per_warp(cnt_r, shares, (int64_t)nblk * (kBatchBlock / 32));
    batch_queue<NBT, FMT>(a, smem_raw, (unsigned long long)cnt_r * parts, rpw, held, [&](int chunk, unsigned long long it) {
      const int part = parts == 1 ? 0 : (int)(it / (unsigned long long)cnt_r);
      const int64_t k = first + (int64_t)(it - (unsigned long long)part * cnt_r);
      const int v = a.view[k];
      if (a.mode == 2) {
        // the pixel's values from its view's proposal wave when the wave
        // traced it (the same trace, so the same bits); else trace it
        const int L = t.lvl[k], i = t.pi[k], j = t.pj[k];
        const int64_t pb = (int64_t)v * nn0 + (int64_t)(j >> L) * n0 + (i >> L);
        const int64_t q = prop_index(a.pdepth + 4 * pb, a.poff[pb], L, i, j);
        const int cp = chunk * parts + part;
        if (q >= 0) {
          if (cp == 0) {
            t.N[k] = a.pN[q];
            t.steps[k] = a.psteps[q];
          }
          const int b0 = (int)((int64_t)nb * cp / shares), b1 = (int)((int64_t)nb * (cp + 1) / shares);
          for (int c = b0; c < b1; ++c) t.I[(int64_t)c * t.cap + k] = a.pI[(int64_t)c * a.P + q];
          if (a.chunks == 1 && cp == 0) t.p[k] = a.pp[q];
          return;
        }
        if (cp == 0) atomicAdd(&a.ctl->fb_rays, 1ull);
      }
      batch_trace<NBT, AMR, FMT, DIR>(a, smem_raw, a.geoms[v], t.lvl[k], t.pi[k], t.pj[k], chunk, part, parts,
                                      shares == 1, o, k);
    });
    if (!grid_sync(a.ctl, nblk, a.timeout_ns)) return;
    if (blockIdx.x == 0 && threadIdx.x < a.chunks) a.ctl->q_head[threadIdx.x] = 0ull;  // next sweep's queues
    if (shares > 1) {
      for (int64_t k = first + gtid; k < n; k += gstride) {
        float s = 0.f;
        for (int q = 0; q < nb; ++q) s += t.I[(int64_t)q * t.cap + k];
        t.p[k] = s;
      }
      if (!grid_sync(a.ctl, nblk, a.timeout_ns)) return;
    }
    if (a.mode == 1) {
      // the base images are traced (and their band sums): the host computes
      // the features and the proposal, then launches mode 2
      if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.ctl->n_nodes = n;
        a.ctl->sweeps = 0;
      }
      return;
    }
    // step iii: scan, then balance
    for (int64_t k = gtid; k < n; k += gstride)
      a.flag[k] = xi_flag(t, NodeLookup{(int)(a.view[k] * nn0), nullptr}, k, a.xi_crit, a.xi_norm, a.refine_on);
    if (!grid_sync(a.ctl, nblk, a.timeout_ns)) return;
    for (int64_t k = gtid; k < n; k += gstride)
      if (a.flag[k]) balance_from(t, NodeLookup{(int)(a.view[k] * nn0), nullptr}, (int)k, a.flag, &a.ctl->err);
    if (!grid_sync(a.ctl, nblk, a.timeout_ns)) return;
    // step iv: per-view prefix sum over static node ranges
    const int64_t per = (n + nblk - 1) / nblk;
    const int64_t s0 = min(n, (int64_t)blockIdx.x * per), s1 = min(n, s0 + per);
    for (int v = threadIdx.x; v < V; v += blockDim.x) cnt[v] = 0;
    __syncthreads();
    for (int64_t k = s0 + threadIdx.x; k < s1; k += blockDim.x)
      if (a.flag[k]) atomicAdd(&cnt[a.view[k]], 1);
    __syncthreads();
    for (int v = threadIdx.x; v < V; v += blockDim.x) a.bcnt[(int64_t)blockIdx.x * V + v] = cnt[v];
    if (!grid_sync(a.ctl, nblk, a.timeout_ns)) return;
    for (int v = threadIdx.x; v < V; v += blockDim.x) {
      int64_t off = 0, all = 0;
      for (unsigned b2 = 0; b2 < nblk; ++b2) {
        const int64_t c = a.bcnt[(int64_t)b2 * V + v];
        if (b2 < blockIdx.x) off += c;
        all += c;
      }
      run[v] = off;
      tot[v] = all;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      int64_t acc = 0;
      for (int v = 0; v < V; ++v) {
        vbase[v] = n + 4 * acc;
        acc += tot[v];
      }
      s_total = acc;
    }
    __syncthreads();
    const int64_t total = s_total;
    if (total == 0) break;
    if (n + 4 * total > t.cap) {
      if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.ctl->need = n + 4 * total;
        atomicOr(&a.ctl->err, kErrCapacity);
      }
      break;
    }
    EmitChildrenV em{t, a.view, vbase};
    block_emit_by_view(FlagPred{a.flag}, a.view, em, s0, s1, V, run, wcnt);
    if (blockIdx.x == 0)
      for (int v = threadIdx.x; v < V; v += blockDim.x)
        if (tot[v] > 0) {
          a.refined[v] += tot[v];
          a.vsweeps[v] += 1;
        }
    if (!grid_sync(a.ctl, nblk, a.timeout_ns)) return;
    first = n;
    n += 4 * total;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    a.ctl->n_nodes = n;
    a.ctl->sweeps = sweep;
  }
}

// (One limit of dynamic shared memory for every launch, see kWideShared: the
// block's tables, constants and sums are below 114 KB by batch_tables, and 256
// views' counters take 11 KB.)
constexpr int kBatchShared = 200 * 1024;
template <int NBT, bool AMR, int FMT, int DIR>
static cudaError_t batch_occupancy(int *blocks_per_sm, size_t smem) {
  cudaError_t e = cudaFuncSetAttribute(k_air_batch<NBT, AMR, FMT, DIR>, cudaFuncAttributeMaxDynamicSharedMemorySize, kBatchShared);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_air_batch<NBT, AMR, FMT, DIR>, kBatchBlock, smem);
}

template <int NBT, bool AMR, int FMT, int DIR>
static cudaError_t batch_launch(const BatchArgs &a, int grid, size_t smem, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kBatchBlock);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_air_batch<NBT, AMR, FMT, DIR>, a);
}

template <int NBT, int FMT, int DIR>
static void batch_pick(const GridView &g, int V, int width, BatchOccFn *occ, BatchLaunchFn *launch, size_t *smem,
                       int *tabs) {
  const bool amr = g.kind == AIR_GRID_AMR;
  *tabs = batch_tables<NBT, DIR>(g, V, width);
  *smem = batch_smem<NBT>(g, V, width, *tabs);
  *occ = amr ? batch_occupancy<NBT, true, FMT, DIR> : batch_occupancy<NBT, false, FMT, DIR>;
  *launch = amr ? batch_launch<NBT, true, FMT, DIR> : batch_launch<NBT, false, FMT, DIR>;
}

// Occupancy and launch functions, shared memory and resident tables of the
// kernel for a grid and V views (inclined: all of them are) with NBT bands per
// thread (0: the wide form, `width` bands per chunk); false where there is no
// such form.
template <int NBT>
bool batch_fns(const GridView &g, int V, bool inclined, int width, BatchOccFn *occ, BatchLaunchFn *launch,
               size_t *smem, int *tabs) {
  if (g.cell_fmt == kCellLam) {
    // per-cell Lambda exists for one-band grids only
    if constexpr (NBT == 1) {
      if (inclined) batch_pick<1, kCellLam, -2>(g, V, width, occ, launch, smem, tabs);
      else batch_pick<1, kCellLam, 0>(g, V, width, occ, launch, smem, tabs);
      return true;
    }
    return false;
  }
  // inclined views with more than 8 bands per thread take the wide form
  constexpr int DIR = NBT == 0 ? -2 : 0;
  if constexpr (NBT >= 1 && NBT <= 8)
    if (inclined) {
      if (g.cell_fmt == kCellXq) batch_pick<NBT, kCellXq, -2>(g, V, width, occ, launch, smem, tabs);
      else batch_pick<NBT, kCellRho, -2>(g, V, width, occ, launch, smem, tabs);
      return true;
    }
  if (g.cell_fmt == kCellXq) batch_pick<NBT, kCellXq, DIR>(g, V, width, occ, launch, smem, tabs);
  else batch_pick<NBT, kCellRho, DIR>(g, V, width, occ, launch, smem, tabs);
  return true;
}

}  // namespace air
