// air_refine.cuh -- image quadtree layout and the refinement launchers.
#pragma once
#include "air_internal.cuh"

namespace air {

constexpr int kScanBlock = 256;
constexpr int kScanRounds = 2;
constexpr int kScanItems = kScanBlock * kScanRounds;
constexpr int kBalanceStack = 8 * kMaxLevels;

// Offset of level l's map in the level maps of a single-view tree (levels
// 1 .. Lm - 1, each a dense (n0 2^l)^2 array of node indices); the maps of
// levels below Lm take level_map_offset(n0, Lm) entries.
__host__ __device__ inline int64_t level_map_offset(int n0, int l) {
  // sum over 1 <= l' < l of (n0 2^l')^2 = n0^2 (4^l - 4) / 3
  return l <= 1 ? 0 : (int64_t)n0 * n0 * ((((int64_t)1 << (2 * l)) - 4) / 3);
}

// Scan chunks (of kScanItems) covering n items.
__host__ __device__ inline int64_t scan_chunks(int64_t n) { return (n + kScanItems - 1) / kScanItems; }

// Node arrays of the image quadtree (capacity `cap`).
struct TreeView {
  int n0, Lm;
  int64_t cap;
  int8_t *lvl;
  int32_t *pi, *pj;
  int32_t *child;   // first child index, -1 for a leaf
  float *N;         // column density
  float *I;         // [n_bands][cap]
  float *p;         // band-summed intensity
  uint32_t *steps;
};

// Output arrays (device memory), entry r of `stride`.
struct OutView {
  int32_t *level, *i, *j;
  uint8_t *is_leaf;
  float *N, *p, *I;
  int64_t stride;
  int n_bands;
};

struct FluxArgs {
  int64_t n;             // nodes or pixels
  const int32_t *child;  // NULL: every entry is a leaf
  const int8_t *lvl;     // NULL: level 0
  const float *I;        // [n_bands][stride]
  int64_t stride;
  const uint32_t *steps;
  int n_bands;
  double area0;          // pixel area at level 0
  double *partial;       // [blocks][n_bands + 1]
  // leaves counted on the way (NULL: not): per scan chunk of kScanItems nodes,
  // and per block of kFluxPerBlock nodes
  int32_t *chunk_leaves, *block_leaves;
  // where the sums go: the flux to device memory (may be NULL), and to
  // page-locked memory, [n_bands], with the step count behind it
  double *flux, *host;
};
// Nodes of a flux block: 8192, 32 per thread. (2048: the FP64 sums at each
// block's end took longer than its loads; 70 us instead of 44 for 7.7 M nodes
// of one band.)
constexpr int64_t kFluxPerBlock = 8192;
constexpr int kFluxChunks = kFluxPerBlock / kScanItems;
// Flux blocks whose leaf counts every block of k_emit_out adds up for itself (up
// to four loads per thread); above, one launch forms their prefix sums first.
constexpr int64_t kFluxDirect = 1024;

// Device-resident bookkeeping of the sweep loop when the counts stay on the
// device (render_adaptive without a read-back per sweep). Sweep q starts from
// slot q & 3; its emit kernel knows what the sweep adds and writes the next
// slot, which the march of the new pixels reads beside the first (so no kernel
// waits for a last block to move the state on). Once a slot is `done`, later
// kernels return at once and the next slots are copies of it, so sweeps queued
// past the end do nothing. A slot is written again four sweeps later, when
// every kernel that reads it has ended.
struct SweepSlot {
  long long n;          // traced nodes when the sweep starts
  long long m;          // length of its open-leaf list
  long long n_refined;  // refined nodes so far
  int sweeps;           // sweeps so far that refined something
  int done;             // nothing is left to scan, or the sweep before flagged nothing
  unsigned long long ray_ctr[kMaxBands];  // march work counters, one per band chunk
  // with a learned proposal: pixels of this sweep that it missed
  unsigned long long missed;
};
struct SweepState {
  SweepSlot slot[4];
  // with a learned proposal: pixels it missed, and the sweeps that had any
  unsigned long long fb_total;
  int fb_waves;
};

// What the host sees of it: page-locked memory, of which the emit kernel of
// sweep q writes entry q & 3 (`progress` last: the render's tag in the high
// word, q + 1 in the low one), so the host follows the loop without a copy or
// an event in the stream. It reads an entry before it queues the sweep that
// will write it again.
struct SweepReport {
  long long n, n_refined;
  int sweeps, done;
  unsigned int err;  // the balance's error word
  unsigned long long progress;
};

// Programmatic dependent launch: a kernel of the sweep chain waits here for
// the kernel before it (launched with cudaLaunchAttributeProgrammaticStream-
// Serialization, the wait returns once that kernel has completed and its
// memory is visible; launched without it, the wait returns at once).
// From then on the kernel after it may be scheduled too: its blocks come up
// beside this kernel's last ones and wait here in their turn, so a launch
// costs no gap. (Without the second instruction the next kernel was scheduled
// only when this one had ended.)
// So the kernel before may write while this one already runs: what it writes is
// read by ordinary loads, through pointers without `const __restrict__`. Those
// make read-only loads, which are defined for data that nothing writes during
// the kernel and which the wait does not have to order.
__device__ __forceinline__ void wait_prior_grid() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Launch with programmatic stream serialization: the kernel may be scheduled
// while the one before it in the stream is finishing, and waits for it in
// wait_prior_grid(), so the launch latency between the short kernels of a
// sweep overlaps the previous kernel's tail.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                              cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// ---- band flux (shared by the single-view and the batched output) ----------
constexpr int kFluxBands = 4;  // bands a block sums side by side

__device__ __forceinline__ double pow4_neg(int L) {
  return __longlong_as_double((long long)(1023 - 2 * L) << 52);
}

// A thread's leaves are summed as an unevaluated pair of FP32 numbers
// (Knuth's two-sum: hi + lo carries the sum of 32 terms to 2^-38 relative or
// better) of I 4^-L, an exact scaling while the product stays a normal number;
// the rare smaller terms, and those so large that their sum could leave the
// FP32 range, go to an FP64 sum. FP64 work per thread, not per leaf (FP64
// issues at 1/64 of the FP32 rate here); between threads the sums are FP64.
__device__ __forceinline__ void flux_add(float I, int L, float &hi, float &lo, double &rest) {
  const float x = __fmul_rn(I, __int_as_float((127 - 2 * L) << 23));
  const float m = fabsf(x);
  if ((m >= 0x1p-126f && m <= 0x1p120f) || x == 0.f) {
    const float t = __fadd_rn(hi, x);
    const float bv = __fsub_rn(t, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(t, bv)), __fsub_rn(x, bv)));
    hi = t;
  } else {
    rest = fma((double)I, pow4_neg(L), rest);
  }
}

// The warp's FP64 sums of v[0 .. kFluxBands): the eight lanes from 8 q on return
// the sum of v[q]. Lanes first trade away the bands they will not hold, so four
// bands take six FP64 additions per warp (a butterfly for each takes twenty).
// No shared memory: with 8 KB of it the flux kernel, launched as a dependent,
// changed the SMs' split of L1 and shared memory behind the march, and a fixed
// image of 200^2 pixels took 67 us instead of 52.
__device__ __forceinline__ double flux_warp_sum(const double (&v)[kFluxBands]) {
  static_assert(kFluxBands == 4, "eight lanes per band");
  const bool hi = threadIdx.x & 16, odd = threadIdx.x & 8;
  const double a = (hi ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, hi ? v[0] : v[2], 16);
  const double b = (hi ? v[3] : v[1]) + __shfl_xor_sync(0xffffffffu, hi ? v[1] : v[3], 16);
  double s = (odd ? b : a) + __shfl_xor_sync(0xffffffffu, odd ? a : b, 8);
  for (int off = 4; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  return s;
}

cudaError_t launch_init_base(const TreeView &t, cudaStream_t st);
int64_t scan_blocks(int64_t n);
cudaError_t launch_count_flags(const uint32_t *flag, int64_t n, int32_t *bcount, int64_t *boff,
                               int64_t *total, cudaStream_t st);
// chunk_leaves, block_leaves: from launch_flux_partial (unused with `all`);
// block_off, total: room for the prefix sums of block_leaves and their sum, used
// where emit_out_scans (a launch of its own).
bool emit_out_scans(int all, int64_t n);
cudaError_t launch_emit_out(const TreeView &t, const OutView &o, int all, int64_t n,
                            const int32_t *chunk_leaves, const int32_t *block_leaves, int64_t *block_off,
                            int64_t *total, cudaStream_t st);
// Exclusive scan of nb per-block counts (one block) -> boff, total.
cudaError_t launch_scan_offsets(const int32_t *bcount, int64_t nb, int64_t *boff, int64_t *total,
                                cudaStream_t st);
// Open-leaf list (leaves below the top level, ascending): steps iii-iv over it.
cudaError_t launch_list_init(int32_t *list, int64_t m, cudaStream_t st);
// lmap: level maps of a single-view tree (see air_tree.cuh), or NULL to find
// stencil neighbours by descent through the child links.
cudaError_t launch_list_scan(const TreeView &t, const int32_t *open, int64_t m, double xi_crit,
                             int xi_norm, int refine_on, uint32_t *flag, cudaStream_t st,
                             const int32_t *lmap = nullptr);
cudaError_t launch_list_balance(const TreeView &t, const int32_t *open, int64_t m, uint32_t *flag,
                                uint32_t *err, cudaStream_t st, const int32_t *lmap = nullptr);
// totals[0] flagged, [1] kept, [2] flagged with children below the top level;
// bcount / boff hold 3 x scan_blocks(m) entries.
cudaError_t launch_list_count(const TreeView &t, const int32_t *open, int64_t m,
                              const uint32_t *flag, int32_t *bcount, int64_t *boff,
                              int64_t *totals, cudaStream_t st);
// Children of the flagged entries at n_old + 4 * rank; the next list into `next`.
cudaError_t launch_list_emit(const TreeView &t, const int32_t *open, int64_t m, uint32_t *flag,
                             const int64_t *boff, const int64_t *totals, int64_t n_old,
                             int32_t *next, cudaStream_t st, int32_t *lmap = nullptr);
// The same steps with every count read from the device: sweep q of the loop
// (SweepState S). The current list is open[q & 1], the next one
// open[(q + 1) & 1]. Grids are sized for the GPU, not for the count, and loop
// over the items. counts: 4 x nb_cap chunk counts, nb_cap = scan_blocks of the
// largest list.
// The state, the first list (the m base pixels), its flag words and the counts.
cudaError_t launch_open_init(SweepState *S, int64_t n, int32_t *list, uint32_t *flag, int64_t m,
                             uint32_t *counts, int64_t nb_cap, cudaStream_t st);
// Scan and balance fused; flagged leaves counted per chunk.
cudaError_t launch_sweep_scan_balance(const TreeView &t, int32_t *const open[2],
                                      const SweepState *S, int q, double xi_crit, int xi_norm,
                                      int refine_on, uint32_t *flag, uint32_t *counts,
                                      int64_t nb_cap, uint32_t *err, cudaStream_t st,
                                      const int32_t *lmap);
// Children, the next list, the level maps, the next slot and the report.
cudaError_t launch_sweep_emit(const TreeView &t, int32_t *const open[2], SweepState *S, int q,
                              uint32_t *flag, uint32_t *counts, int64_t nb_cap,
                              const uint32_t *err, SweepReport *rep, uint32_t tag, cudaStream_t st,
                              int32_t *lmap);
int64_t flux_blocks(int64_t n);
cudaError_t launch_flux_partial(const FluxArgs &a, cudaStream_t st);
cudaError_t launch_flux_final(const FluxArgs &a, cudaStream_t st);

}  // namespace air
