// air_batch.cu -- batched adaptive images: many views of one grid (each view
// with all its energy bands) rendered by ONE cooperative persistent kernel.
// Parkin (2010), Section 2 steps i-vi, applied to every view at once.
//
// Inside the kernel, per sweep:
//   march   : a work queue of (ray, band chunk) items over the rays added in
//             the previous sweep, all views mixed; warps fetch up to 32 items
//             (rays_per_warp) at a time with one atomic, so rays of uneven
//             length, level, view and band balance across the whole GPU;
//   band sum: p = sum_b I_b when the bands were split over several threads;
//   scan    : Eq. 2 on every leaf below max_level (all views);
//   balance : 2:1 closure within each view's tree;
//   refine  : per-view prefix sum of the flags (static ranges of nodes per
//             block, per-view counts, per-view offsets), four children per
//             flagged leaf, emitted view by view so every view's nodes keep
//             the order of a single-view render.
// Phases are separated by a grid barrier of the library's own (an arrival
// counter and a generation word); every wait has a time limit after which the
// kernel records AIR_ERR_TIMEOUT and returns. The launch is cooperative, so
// all blocks are resident, and the host captures it in a CUDA graph.
#include <cstring>
#include <vector>

#include "air_batch_kernel.cuh"

namespace air {

// ---- output: per-view leaf compaction, band flux, step counts ---------------

struct LeafPred {
  const int32_t *child;
  int all;
  __device__ bool operator()(int64_t k) const { return all || child[k] < 0; }
};

// Per block of kScanItems nodes: selected nodes per view; ray-cell steps per view.
__global__ void __launch_bounds__(256) k_vcount(TreeView t, const int16_t *view, int all, int64_t n,
                                                int V, int32_t *bcnt,
                                                unsigned long long *vsteps) {
  extern __shared__ int32_t sm_cnt[];
  unsigned long long *sm_steps = (unsigned long long *)(sm_cnt + ((V + 1) & ~1));
  for (int v = threadIdx.x; v < V; v += blockDim.x) {
    sm_cnt[v] = 0;
    sm_steps[v] = 0ull;
  }
  __syncthreads();
  const int64_t s0 = (int64_t)blockIdx.x * kScanItems, s1 = min(n, s0 + kScanItems);
  for (int64_t r0 = s0; r0 < s1; r0 += blockDim.x) {
    // one addition per warp where its nodes are of one view (nodes of a view
    // lie together), else one per node
    const int64_t k = r0 + threadIdx.x;
    const bool in = k < s1;
    const int v = in ? (int)view[k] : -1;
    const bool sel = in && (all || t.child[k] < 0);
    const uint32_t st = in ? t.steps[k] : 0u;
    const int v0 = __shfl_sync(0xffffffffu, v, 0);
    const unsigned nsel = __popc(__ballot_sync(0xffffffffu, sel));
    if (__all_sync(0xffffffffu, v == v0 || !in)) {
      const unsigned lo = __reduce_add_sync(0xffffffffu, st & 0xffffu);
      const unsigned hi = __reduce_add_sync(0xffffffffu, st >> 16);
      if ((threadIdx.x & 31) == 0 && in) {
        if (nsel) atomicAdd(&sm_cnt[v0], (int)nsel);
        atomicAdd(&sm_steps[v0], ((unsigned long long)hi << 16) + lo);
      }
    } else if (in) {
      if (sel) atomicAdd(&sm_cnt[v], 1);
      atomicAdd(&sm_steps[v], (unsigned long long)st);
    }
  }
  __syncthreads();
  for (int v = threadIdx.x; v < V; v += blockDim.x) {
    bcnt[(int64_t)blockIdx.x * V + v] = sm_cnt[v];
    if (sm_steps[v]) atomicAdd(&vsteps[v], sm_steps[v]);
  }
}

// One block per view: exclusive scan of that view's per-block counts.
__global__ void __launch_bounds__(256) k_vscan(const int32_t *bcnt, int64_t nblocks, int V,
                                               int64_t *boff) {
  __shared__ int64_t part[256];
  const int v = blockIdx.x;
  const int64_t per = (nblocks + 255) / 256;
  const int64_t a = threadIdx.x * per, b = min(nblocks, a + per);
  int64_t s = 0;
  for (int64_t x = a; x < b; ++x) s += bcnt[x * V + v];
  part[threadIdx.x] = s;
  __syncthreads();
  for (int off = 1; off < 256; off <<= 1) {
    const int64_t u = threadIdx.x >= off ? part[threadIdx.x - off] : 0;
    __syncthreads();
    part[threadIdx.x] += u;
    __syncthreads();
  }
  int64_t run = part[threadIdx.x] - s;
  for (int64_t x = a; x < b; ++x) {
    boff[x * V + v] = run;
    run += bcnt[x * V + v];
  }
}

struct EmitOutV {
  TreeView t;
  const OutView *outs;    // [V] (global)
  __device__ void operator()(int64_t k, int v, int64_t r) {
    const OutView &o = outs[v];
    if (o.level) o.level[r] = t.lvl[k];
    if (o.i) o.i[r] = t.pi[k];
    if (o.j) o.j[r] = t.pj[k];
    if (o.is_leaf) o.is_leaf[r] = t.child[k] < 0;
    if (o.N) o.N[r] = t.N[k];
    if (o.p) o.p[r] = t.p[k];
    if (o.I) {
#pragma unroll 4
      for (int b = 0; b < o.n_bands; ++b) o.I[(int64_t)b * o.stride + r] = t.I[(int64_t)b * t.cap + k];
    }
  }
};

__global__ void __launch_bounds__(256) k_vemit(TreeView t, const int16_t *view, int all, int64_t n,
                                               int V, const int64_t *boff, const OutView *outs) {
  extern __shared__ __align__(16) unsigned char sm[];
  int64_t *run = (int64_t *)sm;
  int32_t *wcnt = (int32_t *)(run + V);
  for (int v = threadIdx.x; v < V; v += blockDim.x) run[v] = boff[(int64_t)blockIdx.x * V + v];
  __syncthreads();
  const int64_t s0 = (int64_t)blockIdx.x * kScanItems, s1 = min(n, s0 + kScanItems);
  EmitOutV e{t, outs};
  block_emit_by_view(LeafPred{t.child, all}, view, e, s0, s1, V, run, wcnt);
}

// Band flux of every view, every addition in FP64. A block takes 2048 nodes and
// kFluxBands bands (blockIdx.y). Nodes of a view lie together, so a warp's strip
// of 32 nodes mostly belongs to one view: its lanes sum on until the view
// changes, and the block adds its warps' sums to the view's flux at the end.
// (An FP64 atomic in shared memory per leaf and band, in the kernel above,
// took most of the 2 ms that the output of 8 views x 16 bands cost.)
constexpr int kVfluxRounds = 8;
__global__ void __launch_bounds__(256) k_vflux(TreeView t, const int16_t *view, int64_t n,
                                               int n_bands, const RayGeom *geoms, double *vflux) {
  __shared__ double sums[kFluxBands][8];
  __shared__ int views[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int b0 = blockIdx.y * kFluxBands, nb = min(kFluxBands, n_bands - b0);
  const int64_t start = (int64_t)blockIdx.x * (256 * kVfluxRounds) + threadIdx.x;
  double acc[kFluxBands];
  int cur = -1;
#pragma unroll
  for (int q = 0; q < kFluxBands; ++q) acc[q] = 0.0;
  auto area = [&](int v) { return geoms[v].pix0 * geoms[v].pix0; };
  for (int r = 0; r < kVfluxRounds; ++r) {
    const int64_t k = start + (int64_t)r * 256;
    const bool in = k < n;
    const int v = in ? (int)view[k] : -1;
    const bool leaf = in && t.child[k] < 0;
    const int L = leaf ? t.lvl[k] : 0;
    const int v0 = __shfl_sync(0xffffffffu, v, 0);
    if (v0 < 0) break;  // past the end
    if (__all_sync(0xffffffffu, v == v0 || !in)) {
      if (v0 != cur) {
        if (cur >= 0) {
          const double s = flux_warp_sum(acc);
          if ((lane & 7) == 0 && (lane >> 3) < nb) atomicAdd(&vflux[(int64_t)cur * n_bands + b0 + (lane >> 3)], s * area(cur));
#pragma unroll
          for (int q = 0; q < kFluxBands; ++q) acc[q] = 0.0;
        }
        cur = v0;
      }
#pragma unroll
      for (int q = 0; q < kFluxBands; ++q)
        if (leaf && q < nb) {
          const float I = t.I[(int64_t)(b0 + q) * t.cap + k];
          // (an FP64 conversion costs as much as an addition: normal numbers
          // are widened by integer operations)
          const bool normal = fabsf(I) >= 0x1p-126f && fabsf(I) <= FLT_MAX;
          acc[q] = fma(normal ? widen(I) : (double)I, pow4_neg(L), acc[q]);
        }
    } else if (leaf) {
      for (int q = 0; q < nb; ++q)
        atomicAdd(&vflux[(int64_t)v * n_bands + b0 + q],
                  (double)t.I[(int64_t)(b0 + q) * t.cap + k] * pow4_neg(L) * area(v));
    }
  }
  const double s4 = flux_warp_sum(acc);
  if ((lane & 7) == 0) sums[lane >> 3][warp] = s4;
  if (lane == 0) views[warp] = cur;
  __syncthreads();
  if (threadIdx.x < nb) {
    const int q = threadIdx.x;
    for (int w = 0; w < 8;) {  // runs of warps that ended on the same view
      const int v = views[w];
      double s = 0.0;
      for (; w < 8 && views[w] == v; ++w) s += sums[q][w];
      if (v >= 0) atomicAdd(&vflux[(int64_t)v * n_bands + b0 + q], s * area(v));
    }
  }
}

// ---- host ---------------------------------------------------------------------

#define CU_TRY(x)                                    \
  do {                                               \
    cudaError_t e_ = (x);                            \
    if (e_ != cudaSuccess) return cuda_fail(e_, #x); \
  } while (0)

// Compiled in air_batch_<NBT>.cu.
extern template bool batch_fns<0>(const GridView &, int, bool, int, BatchOccFn *, BatchLaunchFn *, size_t *, int *);
extern template bool batch_fns<1>(const GridView &, int, bool, int, BatchOccFn *, BatchLaunchFn *, size_t *, int *);
extern template bool batch_fns<2>(const GridView &, int, bool, int, BatchOccFn *, BatchLaunchFn *, size_t *, int *);
extern template bool batch_fns<4>(const GridView &, int, bool, int, BatchOccFn *, BatchLaunchFn *, size_t *, int *);
extern template bool batch_fns<8>(const GridView &, int, bool, int, BatchOccFn *, BatchLaunchFn *, size_t *, int *);
extern template bool batch_fns<16>(const GridView &, int, bool, int, BatchOccFn *, BatchLaunchFn *, size_t *, int *);

static bool batch_form(int nbt, const GridView &g, int V, bool inclined, int width, BatchOccFn *occ,
                       BatchLaunchFn *launch, size_t *smem, int *tabs) {
  if (width) return batch_fns<0>(g, V, true, width, occ, launch, smem, tabs);
  if (nbt == 1) return batch_fns<1>(g, V, inclined, width, occ, launch, smem, tabs);
  if (nbt == 2) return batch_fns<2>(g, V, inclined, width, occ, launch, smem, tabs);
  if (nbt == 4) return batch_fns<4>(g, V, inclined, width, occ, launch, smem, tabs);
  if (nbt == 8) return batch_fns<8>(g, V, inclined, width, occ, launch, smem, tabs);
  if (nbt == 16) return batch_fns<16>(g, V, inclined, width, occ, launch, smem, tabs);
  return false;
}

// Bands per thread of batched renders when the tuning leaves it open: the
// template width that holds every band, up to 8 (8 inclined views of 16 bands:
// 16.1 ms at 8, 20.0 ms at 16, where two blocks fit an SM).
static int default_batch_bands_per_thread(int nb) {
  if (nb <= 1) return 1;
  if (nb <= 2) return 2;
  if (nb <= 4) return 4;
  return 8;
}

// Node count for the next attempt of a batch that outgrew its arrays at
// `need` nodes (more sweeps may follow): twice that, as far as half of the
// free device memory allows, and at least a sixteenth above it.
static int64_t batch_regrow(air_grid *g, int64_t need, int64_t bound) {
  const double per_node = 31.0 + 4.0 * g->gv.n_bands;
  size_t fr = 0, tot = 0;
  int64_t roomy = 2 * need;
  if (cudaMemGetInfo(&fr, &tot) == cudaSuccess) {
    const int64_t held = g->ws.cap;  // freed when the arrays are replaced
    const int64_t fit = (int64_t)(0.5 * (double)fr / per_node) + held;
    roomy = std::min<int64_t>(roomy, fit);
  } else {
    cudaGetLastError();
  }
  return std::min<int64_t>(bound, std::max<int64_t>(need + need / 16, roomy));
}

air_status render_batch(air_grid *g, const air_view *views, int32_t V, const air_params *pr,
                        const air_batch_opts *opts, air_image *outs, air_mlp *mlp,
                        const air_learned_opts *lopts, air_learned_stats *stats) {
  g->raster.ok = false;  // the workspace tree is about to change
  if (!views || !outs || !pr) return set_error(AIR_ERR_ARG, "views, params and outs must not be NULL");
  if (V < 1 || V > kBatchMaxViews) return set_error(AIR_ERR_ARG, "n_views must be in [1, %d]", kBatchMaxViews);
  const int n0 = pr->base_res, Lm = pr->max_level;
  if (n0 < 1 || Lm < 0 || Lm >= kMaxLevels || ((int64_t)n0 << Lm) > (1 << 20))
    return set_error(AIR_ERR_ARG, "need base_res >= 1, 0 <= max_level < %d, base_res << max_level <= 2^20", kMaxLevels);
  if (!(pr->xi_crit >= 0.0) || pr->xi_crit > 1e300) return set_error(AIR_ERR_ARG, "xi_crit must be finite and >= 0");
  if (pr->xi_norm != 0 && pr->xi_norm != 1) return set_error(AIR_ERR_ARG, "xi_norm must be 0 or 1");
  if (pr->refine_on < 0 || pr->refine_on > 2) return set_error(AIR_ERR_ARG, "refine_on must be 0, 1 or 2");
  if (pr->include_interior != 0 && pr->include_interior != 1) return set_error(AIR_ERR_ARG, "include_interior must be 0 or 1");
  air_batch_opts op{};
  op.bands_per_thread = 0;
  op.use_graph = 1;
  op.wait_timeout_ms = 2000.0;
  op.test_stall_barrier = 0;
  if (opts) op = *opts;
  if (!(op.wait_timeout_ms > 0.0)) op.wait_timeout_ms = 2000.0;
  const int nb = g->gv.n_bands;
  for (int v = 0; v < V; ++v) {
    air_status s = check_image(&outs[v]);
    if (s) return s;
  }
  std::vector<RayGeom> geoms(V);
  for (int v = 0; v < V; ++v) {
    Camera cam;
    air_status s = make_camera(&views[v], cam);
    if (s) return s;
    geoms[v] = make_geom(g->gv, cam, n0);
  }
  bool inclined = true;  // no view along a grid axis
  for (const RayGeom &r : geoms) inclined = inclined && (r.Dhi[0] != 0.f) + (r.Dhi[1] != 0.f) + (r.Dhi[2] != 0.f) > 1;
  const bool set = op.bands_per_thread > 0 || g->tune.batch_bands_per_thread > 0;  // by the caller
  int nbt = op.bands_per_thread > 0 ? op.bands_per_thread
            : (g->tune.batch_bands_per_thread > 0 ? g->tune.batch_bands_per_thread : default_batch_bands_per_thread(nb));
  if (g->gv.cell_fmt == kCellLam && nbt > 0) nbt = 1;  // one band
  BatchOccFn occ;
  BatchLaunchFn launch;
  size_t smem = 0;
  int tabs = 0;
  // inclined views with more than 8 bands (per thread, where the caller has set
  // that): the wide form, whose chunks hold as many bands as fit
  const int width = !inclined ? 0 : (set ? (nbt == 16 ? 16 : 0) : (nb > 8 ? wide_width(g->gv, kBatchBlock) : 0));
  if (!batch_form(nbt, g->gv, V, inclined, width, &occ, &launch, &smem, &tabs))
    return set_error(AIR_ERR_ARG, "bands_per_thread must be 1, 2, 4, 8 or 16");
  g->last.valid = false;  // the batch reuses the single-view workspace
  air_status s = init_scalars(g->ws);
  if (s) return s;
  Workspace &w = g->ws;
  BatchWork &bw = g->batch;
  cudaStream_t st = g->stream;
  const int64_t nbase = (int64_t)V * n0 * n0;
  int64_t bound = 0;
  for (int l = 0; l <= Lm; ++l) bound += ((int64_t)n0 << l) * ((int64_t)n0 << l);
  bound *= V;
  if (bound > INT32_MAX) bound = INT32_MAX;
  int per_sm = 0;
  int dev = 0, sms = 0;
  CU_TRY(cudaGetDevice(&dev));
  CU_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  CU_TRY(occ(&per_sm, smem));
  if (per_sm < 1) return set_error(AIR_ERR_CUDA, "batched kernel cannot be resident (smem %zu B)", smem);
  if (g->tune.batch_blocks_per_sm > 0 && g->tune.batch_blocks_per_sm < per_sm) per_sm = g->tune.batch_blocks_per_sm;
  const int grid = per_sm * sms;
  // device-side state
  CU_TRY(ensure((void **)&bw.geoms, &bw.geoms_b, sizeof(RayGeom) * V));
  CU_TRY(ensure((void **)&bw.ctl, &bw.ctl_b, sizeof(BatchCtl)));
  CU_TRY(ensure((void **)&bw.bcnt, &bw.bcnt_b, sizeof(int32_t) * (size_t)std::max<int64_t>(grid, scan_blocks(bound)) * V));
  CU_TRY(ensure((void **)&bw.refined, &bw.refined_b, sizeof(int64_t) * V));
  CU_TRY(ensure((void **)&bw.vsweeps, &bw.vsweeps_b, sizeof(int32_t) * V));
  CU_TRY(ensure((void **)&bw.vsteps, &bw.vsteps_b, sizeof(unsigned long long) * V));
  CU_TRY(ensure((void **)&bw.vflux, &bw.vflux_b, sizeof(double) * V * nb));
  CU_TRY(ensure((void **)&bw.outs, &bw.outs_b, sizeof(OutView) * V));
  if (!bw.h_ctl) CU_TRY(cudaMallocHost((void **)&bw.h_ctl, sizeof(BatchCtl)));
  if (bw.h_geoms_b < sizeof(RayGeom) * V) {
    if (bw.h_geoms) cudaFreeHost(bw.h_geoms);
    bw.h_geoms = nullptr;
    bw.h_geoms_b = 0;
    CU_TRY(cudaMallocHost(&bw.h_geoms, sizeof(RayGeom) * kBatchMaxViews));
    bw.h_geoms_b = sizeof(RayGeom) * kBatchMaxViews;
  }
  std::memcpy(bw.h_geoms, geoms.data(), sizeof(RayGeom) * V);
  int64_t want = std::max<int64_t>(std::min<int64_t>(bound, 4 * nbase), w.cap);
  bool done = false;
  for (int attempt = 0; attempt < 8 && !done; ++attempt) {
    // a batch that outgrew the node arrays is rendered again with arrays of
    // the size it needed (and a sixteenth more), not the usual doubling
    if ((s = ensure_nodes(g, want, 0, bound, true, attempt > 0))) return s;
    TreeView t = w.tree(n0, Lm);
    BatchArgs a{};
    a.g = g->gv;
    a.geoms = bw.geoms;
    a.V = V;
    a.width = width;
    a.tabs = tabs;
    a.fill = width && !set ? (int64_t)grid * kBatchBlock * 2 : 0;
    a.chunks = width ? (nb + width - 1) / width : (nb + nbt - 1) / nbt;
    a.fp64_level = pr->fp64_level < 0 ? 3 : pr->fp64_level;
    a.xi_norm = pr->xi_norm;
    a.refine_on = pr->refine_on;
    a.stall = op.test_stall_barrier ? 1 : 0;
    a.xi_crit = pr->xi_crit;
    a.t = t;
    a.view = w.view;
    a.flag = w.flag;
    a.ctl = bw.ctl;
    a.bcnt = bw.bcnt;
    a.refined = bw.refined;
    a.vsweeps = bw.vsweeps;
    a.timeout_ns = (long long)(op.wait_timeout_ms * 1e6);
    CU_TRY(cudaMemcpyAsync(bw.geoms, bw.h_geoms, sizeof(RayGeom) * V, cudaMemcpyHostToDevice, st));
    g->prof.used = 0;
    if (mlp) {
      // learned proposal: the base images (mode 1), the network's proposal
      // for every view, then every proposal wave and the sweeps (mode 2)
      LearnWork &lw = g->learn;
      const double q = (lopts && lopts->quantile > 0.0 && lopts->quantile <= 1.0) ? lopts->quantile : 0.8;
      CU_TRY(ensure((void **)&lw.maxlev, &lw.maxlev_b, (size_t)nbase));
      a.mode = 1;
      a.maxlev = lw.maxlev;
      for (int phase = 1; phase <= 2; ++phase) {
        if (phase == 2) {
          int64_t P = 0;
          if ((s = batch_proposal(g, V, pr, mlp, q, lw.maxlev, &P))) return s;
          a.mode = 2;
          a.maxlev = nullptr;
          a.pdepth = lw.depth;
          a.poff = lw.off;
          a.plvl = lw.plvl;
          a.ppi = lw.ppi;
          a.ppj = lw.ppj;
          a.pview = lw.pview;
          a.P = P;
          a.pN = lw.pN;
          a.pI = lw.pI;
          a.pp = lw.pp;
          a.psteps = lw.psteps;
          if (stats) {
            std::memset(stats, 0, sizeof(*stats));
            stats->proposed_rays = P;
          }
        }
        CU_TRY(prof_open(g, AIR_PHASE_BATCH, 1));
        CU_TRY(cudaMemsetAsync(bw.ctl, 0, sizeof(BatchCtl), st));
        if (phase == 1) {
          CU_TRY(cudaMemsetAsync(bw.refined, 0, sizeof(int64_t) * V, st));
          CU_TRY(cudaMemsetAsync(bw.vsweeps, 0, sizeof(int32_t) * V, st));
        }
        CU_TRY(launch(a, grid, smem, st));
        CU_TRY(prof_close(g));
        CU_TRY(cudaMemcpyAsync(bw.h_ctl, bw.ctl, sizeof(BatchCtl), cudaMemcpyDeviceToHost, st));
        CU_TRY(cudaStreamSynchronize(st));
        if (bw.h_ctl->err & kErrTimeout)
          return set_error(AIR_ERR_TIMEOUT, "batched kernel: a grid barrier wait exceeded %.0f ms", op.wait_timeout_ms);
        if (bw.h_ctl->err & kErrBalance) return set_error(AIR_ERR_NUMERIC, "balance closure overflowed its stack");
        if (bw.h_ctl->err & kErrCapacity) break;
      }
      const BatchCtl c = *bw.h_ctl;
      if (c.err & kErrCapacity) {
        if (c.need > bound) return set_error(AIR_ERR_NUMERIC, "quadtree exceeds its bound");
        want = batch_regrow(g, c.need, bound);
        continue;
      }
      if (stats) stats->fallback_rays = (int64_t)c.fb_rays;
      done = true;
      continue;
    }
    // the graph holds: reset of the control words, the cooperative launch
    const bool same = bw.exec && !std::memcmp(&bw.key, &a, sizeof(BatchArgs)) && bw.key_grid == grid &&
                      bw.key_smem == smem && bw.key_launch == launch;
    CU_TRY(prof_open(g, AIR_PHASE_BATCH, 1));
    if (op.use_graph) {
      if (!same) {
        if (bw.exec) {
          cudaGraphExecDestroy(bw.exec);
          bw.exec = nullptr;
        }
        // capture on a private stream (the caller's may be the legacy default
        // stream, which cannot be captured); the graph then runs on the caller's
        if (!bw.cap_stream) CU_TRY(cudaStreamCreateWithFlags(&bw.cap_stream, cudaStreamNonBlocking));
        cudaStream_t cs = bw.cap_stream;
        cudaGraph_t graph;
        CU_TRY(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
        cudaError_t e1 = cudaMemsetAsync(bw.ctl, 0, sizeof(BatchCtl), cs);
        cudaError_t e2 = cudaMemsetAsync(bw.refined, 0, sizeof(int64_t) * V, cs);
        cudaError_t e3 = cudaMemsetAsync(bw.vsweeps, 0, sizeof(int32_t) * V, cs);
        cudaError_t e4 = launch(a, grid, smem, cs);
        cudaError_t e5 = cudaStreamEndCapture(cs, &graph);
        if (e1 || e2 || e3 || e4 || e5) {
          cudaGetLastError();
          return set_error(AIR_ERR_CUDA, "graph capture of the batched launch failed: %s",
                           cudaGetErrorString(e4 ? e4 : (e5 ? e5 : (e1 ? e1 : (e2 ? e2 : e3)))));
        }
        cudaError_t e6 = cudaGraphInstantiate(&bw.exec, graph, 0);
        cudaGraphDestroy(graph);
        if (e6 != cudaSuccess) return cuda_fail(e6, "cudaGraphInstantiate");
        bw.key = a;
        bw.key_grid = grid;
        bw.key_smem = smem;
        bw.key_launch = launch;
      }
      CU_TRY(cudaGraphLaunch(bw.exec, st));
    } else {
      CU_TRY(cudaMemsetAsync(bw.ctl, 0, sizeof(BatchCtl), st));
      CU_TRY(cudaMemsetAsync(bw.refined, 0, sizeof(int64_t) * V, st));
      CU_TRY(cudaMemsetAsync(bw.vsweeps, 0, sizeof(int32_t) * V, st));
      CU_TRY(launch(a, grid, smem, st));
    }
    CU_TRY(prof_close(g));
    CU_TRY(cudaMemcpyAsync(bw.h_ctl, bw.ctl, sizeof(BatchCtl), cudaMemcpyDeviceToHost, st));
    CU_TRY(cudaStreamSynchronize(st));
    const BatchCtl c = *bw.h_ctl;
    if (c.err & kErrTimeout) return set_error(AIR_ERR_TIMEOUT, "batched kernel: a grid barrier wait exceeded %.0f ms", op.wait_timeout_ms);
    if (c.err & kErrBalance) return set_error(AIR_ERR_NUMERIC, "balance closure overflowed its stack");
    if (c.err & kErrCapacity) {
      if (c.need > bound) return set_error(AIR_ERR_NUMERIC, "quadtree exceeds its bound");
      want = batch_regrow(g, c.need, bound);
      continue;
    }
    done = true;
  }
  if (!done) return set_error(AIR_ERR_CAPACITY, "batched quadtree did not fit after regrowing");
  const int64_t n = bw.h_ctl->n_nodes;
  std::vector<int64_t> refined(V);
  std::vector<int32_t> vsw(V);
  CU_TRY(cudaMemcpy(refined.data(), bw.refined, sizeof(int64_t) * V, cudaMemcpyDeviceToHost));
  CU_TRY(cudaMemcpy(vsw.data(), bw.vsweeps, sizeof(int32_t) * V, cudaMemcpyDeviceToHost));
  if (mlp && stats) {
    int64_t traced = 0;  // nodes beyond the base images: from the wave or traced after it
    for (int v = 0; v < V; ++v) traced += 4 * refined[v];
    stats->used_rays = traced - stats->fallback_rays;
    stats->wasted_rays = stats->proposed_rays - stats->used_rays;
    int32_t mx = 0;
    for (int v = 0; v < V; ++v) mx = std::max(mx, vsw[v]);
    stats->sweeps = mx;
    stats->waves = 2;  // the base images, then the proposal waves and sweeps in one launch
  }
  const int all = pr->include_interior;
  // sizes and capacities
  std::vector<int64_t> n_out(V);
  bool short_cap = false;
  for (int v = 0; v < V; ++v) {
    const int64_t leaves = (int64_t)n0 * n0 + 3 * refined[v];
    const int64_t rays = (int64_t)n0 * n0 + 4 * refined[v];
    n_out[v] = all ? rays : leaves;
    outs[v].n_out = n_out[v];
    outs[v].n_leaves = leaves;
    outs[v].n_rays = rays;
    outs[v].n_sweeps = vsw[v];
    outs[v].n_steps = 0;
    if (outs[v].capacity < n_out[v]) short_cap = true;
  }
  if (short_cap) return set_error(AIR_ERR_CAPACITY, "an output image's capacity is smaller than its pixel count (n_out set per view)");
  // output views: caller device arrays, or staging slices for host memory
  std::vector<OutView> ov(V);
  int64_t stage = 0;
  for (int v = 0; v < V; ++v)
    if (outs[v].mem == AIR_HOST) stage += std::max<int64_t>(n_out[v], 1);
  if (stage > 0) {
    CU_TRY(ensure((void **)&w.o_level, &w.o_level_b, 4 * stage));
    CU_TRY(ensure((void **)&w.o_i, &w.o_i_b, 4 * stage));
    CU_TRY(ensure((void **)&w.o_j, &w.o_j_b, 4 * stage));
    CU_TRY(ensure((void **)&w.o_leaf, &w.o_leaf_b, stage));
    CU_TRY(ensure((void **)&w.o_N, &w.o_N_b, 4 * stage));
    CU_TRY(ensure((void **)&w.o_p, &w.o_p_b, 4 * stage));
    CU_TRY(ensure((void **)&w.o_I, &w.o_I_b, 4 * stage * nb));
  }
  int64_t so = 0;
  for (int v = 0; v < V; ++v) {
    const air_image &im = outs[v];
    OutView &o = ov[v];
    o.n_bands = nb;
    if (im.mem == AIR_DEVICE) {
      o.level = im.level; o.i = im.i; o.j = im.j; o.is_leaf = im.is_leaf;
      o.N = im.coldens; o.p = im.p; o.I = im.intensity;
      o.stride = im.capacity;
    } else {
      const int64_t m = std::max<int64_t>(n_out[v], 1);
      o.level = im.level ? w.o_level + so : nullptr;
      o.i = im.i ? w.o_i + so : nullptr;
      o.j = im.j ? w.o_j + so : nullptr;
      o.is_leaf = im.is_leaf ? w.o_leaf + so : nullptr;
      o.N = im.coldens ? w.o_N + so : nullptr;
      o.p = im.p ? w.o_p + so : nullptr;
      o.I = im.intensity ? w.o_I + so * nb : nullptr;
      o.stride = m;
      so += m;
    }
  }
  CU_TRY(cudaMemcpyAsync(bw.outs, ov.data(), sizeof(OutView) * V, cudaMemcpyHostToDevice, st));
  CU_TRY(cudaMemsetAsync(bw.vsteps, 0, sizeof(unsigned long long) * V, st));
  CU_TRY(cudaMemsetAsync(bw.vflux, 0, sizeof(double) * V * nb, st));
  TreeView t = w.tree(n0, Lm);
  const int64_t nblocks = scan_blocks(n);
  CU_TRY(prof_open(g, AIR_PHASE_OUTPUT, 4));
  if (nblocks > 0) {
    const size_t sm1 = sizeof(int32_t) * ((V + 1) & ~1) + sizeof(unsigned long long) * V;
    k_vcount<<<(unsigned)nblocks, 256, sm1, st>>>(t, w.view, all, n, V, bw.bcnt, bw.vsteps);
    CU_TRY(cudaGetLastError());
    CU_TRY(ensure((void **)&bw.boff, &bw.boff_b, sizeof(int64_t) * nblocks * V));
    k_vscan<<<V, 256, 0, st>>>(bw.bcnt, nblocks, V, bw.boff);
    CU_TRY(cudaGetLastError());
    const size_t sm3 = sizeof(int64_t) * V + sizeof(int32_t) * 8 * V;
    k_vemit<<<(unsigned)nblocks, 256, sm3, st>>>(t, w.view, all, n, V, bw.boff, bw.outs);
    CU_TRY(cudaGetLastError());
    k_vflux<<<dim3((unsigned)((n + 256 * kVfluxRounds - 1) / (256 * kVfluxRounds)),
                   (unsigned)((nb + kFluxBands - 1) / kFluxBands)),
              256, 0, st>>>(t, w.view, n, nb, bw.geoms, bw.vflux);
    CU_TRY(cudaGetLastError());
  }
  CU_TRY(prof_close(g));
  // copies out
  std::vector<double> vflux((size_t)V * nb);
  std::vector<unsigned long long> vsteps(V);
  for (int v = 0; v < V; ++v) {
    const air_image &im = outs[v];
    const OutView &o = ov[v];
    const int64_t m = n_out[v];
    if (im.mem == AIR_HOST && m > 0) {
      if (im.level) CU_TRY(cudaMemcpyAsync(im.level, o.level, 4 * m, cudaMemcpyDeviceToHost, st));
      if (im.i) CU_TRY(cudaMemcpyAsync(im.i, o.i, 4 * m, cudaMemcpyDeviceToHost, st));
      if (im.j) CU_TRY(cudaMemcpyAsync(im.j, o.j, 4 * m, cudaMemcpyDeviceToHost, st));
      if (im.is_leaf) CU_TRY(cudaMemcpyAsync(im.is_leaf, o.is_leaf, m, cudaMemcpyDeviceToHost, st));
      if (im.coldens) CU_TRY(cudaMemcpyAsync(im.coldens, o.N, 4 * m, cudaMemcpyDeviceToHost, st));
      if (im.p) CU_TRY(cudaMemcpyAsync(im.p, o.p, 4 * m, cudaMemcpyDeviceToHost, st));
      if (im.intensity)
        for (int b = 0; b < nb; ++b)
          CU_TRY(cudaMemcpyAsync(im.intensity + (size_t)b * im.capacity, o.I + (size_t)b * o.stride, 4 * m,
                                 cudaMemcpyDeviceToHost, st));
    }
    if (im.band_flux && im.mem == AIR_DEVICE)
      CU_TRY(cudaMemcpyAsync(im.band_flux, bw.vflux + (size_t)v * nb, sizeof(double) * nb, cudaMemcpyDeviceToDevice, st));
  }
  CU_TRY(cudaMemcpyAsync(vflux.data(), bw.vflux, sizeof(double) * V * nb, cudaMemcpyDeviceToHost, st));
  CU_TRY(cudaMemcpyAsync(vsteps.data(), bw.vsteps, sizeof(unsigned long long) * V, cudaMemcpyDeviceToHost, st));
  CU_TRY(cudaStreamSynchronize(st));
  for (int v = 0; v < V; ++v) {
    if (outs[v].band_flux && outs[v].mem == AIR_HOST)
      std::memcpy(outs[v].band_flux, vflux.data() + (size_t)v * nb, sizeof(double) * nb);
    outs[v].n_steps = (int64_t)vsteps[v];
  }
  CU_TRY(prof_resolve(g));
  g->last.valid = false;
  return AIR_OK;
}

void free_batch(air_grid *g) {
  BatchWork &bw = g->batch;
  if (bw.exec) cudaGraphExecDestroy(bw.exec);
  bw.exec = nullptr;
  if (bw.cap_stream) cudaStreamDestroy(bw.cap_stream);
  void *ps[] = {bw.geoms, bw.ctl, bw.bcnt, bw.refined, bw.vsweeps, bw.vsteps, bw.vflux, bw.outs, bw.boff};
  for (void *p : ps)
    if (p) cudaFree(p);
  if (bw.h_ctl) cudaFreeHost(bw.h_ctl);
  if (bw.h_geoms) cudaFreeHost(bw.h_geoms);
  bw = BatchWork{};
}

}  // namespace air

extern "C" air_status air_render_batch(air_grid *g, const air_view *views, int32_t n_views,
                                       const air_params *params, const air_batch_opts *opts,
                                       air_image *outs) {
  air::set_error(AIR_OK, "");
  if (!g) return air::set_error(AIR_ERR_ARG, "grid is NULL");
  return air::render_batch(g, views, n_views, params, opts, outs);
}

extern "C" air_status air_render_batch_learned(air_grid *g, const air_view *views, int32_t n_views,
                                               const air_params *params, const air_batch_opts *opts,
                                               air_mlp *mlp, const air_learned_opts *lopts,
                                               air_image *outs, air_learned_stats *stats) {
  air::set_error(AIR_OK, "");
  if (!g) return air::set_error(AIR_ERR_ARG, "grid is NULL");
  if (!mlp) return air::set_error(AIR_ERR_ARG, "mlp is NULL");
  if (opts && opts->test_stall_barrier) return air::set_error(AIR_ERR_ARG, "test_stall_barrier is for air_render_batch");
  return air::render_batch(g, views, n_views, params, opts, outs, mlp, lopts, stats);
}
