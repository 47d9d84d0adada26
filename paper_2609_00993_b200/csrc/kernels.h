// Internal launcher interface between the C-ABI layer (ctx.cu) and the kernels.
// Every launcher enqueues on `stream`, never synchronises, and returns the CUDA error of the launch.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace moe {

// Raises a kernel's dynamic shared-memory limit once per kernel, device and size, so that steady-state launches
// make no driver calls besides the launch itself (which also keeps them legal while a stream is being captured).
// The first time it also asks for the largest shared-memory carve-out, which the GEMM kernels need: an SM that one of the
// small kernels left with more L1 has to drain before it can be divided anew (one-token V3-shaped decode 133.6 us a step
// with it, 134.2 without).
cudaError_t ensure_dynamic_smem_impl(const void* kern, size_t bytes);
template <typename Kernel>
inline cudaError_t ensure_dynamic_smem(Kernel kern, size_t bytes) {
  return ensure_dynamic_smem_impl(reinterpret_cast<const void*>(kern), bytes);
}

// Programmatic dependent launch: the kernels of the library are launched with "programmatic stream serialization
// allowed" (the GEMMs for small problems only, see kGemmOverlapMaxRows), so their CTAs may become resident and run their
// prologue (barrier set-up, tensor-memory allocation, tensor-map prefetch) while the previous kernel of the stream is
// still draining; pdl_wait() then blocks until that kernel has completed and its writes are visible.
// Rules.  A thread calls pdl_wait() before it first touches global memory that an unfinished kernel may write (or, for its
// own writes, read), and pdl_launch_dependents() right after that wait, never before it.  A kernel therefore starts when
// everything before its predecessor has completed, and may read that -- but nothing of its predecessor -- before it waits
// (offsets_settled below, and the tile counters, of which launches in a row use different pairs).
// The one exception is a quantisation launched with release_early: it releases before it waits.  The kernel behind it (or
// behind several of them in a row) may start while the kernel BEFORE the quantisation is still running, so that before its
// wait it may read only what is older than that one: everything before it has completed, because it releases by the rule.
// A kernel that is launched behind such a quantisation must be held against that.
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl_clusters(bool allow_overlap, int cluster_y, void (*kern)(KArgs...), dim3 grid, dim3 block,
                                       size_t smem, cudaStream_t stream, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  int n = 0;
  if (allow_overlap) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (cluster_y > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = attr[n].val.clusterDim.z = 1;
    attr[n++].val.clusterDim.y = (unsigned)cluster_y;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(bool allow_overlap, void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem,
                              cudaStream_t stream, Args&&... args) {
  return launch_pdl_clusters(allow_overlap, 1, kern, grid, block, smem, stream, static_cast<KArgs>(args)...);
}
// The GEMM kernels take the overlap only for problems of up to this many rows: a step of a few hundred microseconds gains
// 7 % from it (six launch latencies and prologues hidden), while a limit of 32768 rows or none at all changes nothing on the
// weight-streaming workloads and costs 3-6 % on the tensor-bound one (the small kernels keep it at every size).
#ifndef MOE_GEMM_OVERLAP_MAX_ROWS
#define MOE_GEMM_OVERLAP_MAX_ROWS 8192
#endif
constexpr int64_t kGemmOverlapMaxRows = MOE_GEMM_OVERLAP_MAX_ROWS;
#endif

// Device status codes (same values as moe_status in the public header).
constexpr int kStOk = 0;
constexpr int kStTimeout = 6;
constexpr int kStBadIndex = 7;

// ---- a1 route ------------------------------------------------------------------------------
cudaError_t launch_route(const float* logits, const float* bias, int T, int E, int k, float scale, int32_t* idx,
                         float* w, cudaStream_t stream, int* n_launches);

// ---- a2-a4 layout --------------------------------------------------------------------------
// Scratch of the two-launch path: one row of E counts per chunk.  Sized for chunks of 256 slots, which is also the
// documented limit of moe_dispatch_layout_static (the kernels use 1024 and more: rules.h).
constexpr int kLayoutChunk = 256;
inline size_t layout_scratch_ints(int64_t n_slots, int E) {
  int64_t chunks = (n_slots + kLayoutChunk - 1) / kLayoutChunk;
  return (size_t)(chunks > 0 ? chunks : 1) * (size_t)E;
}
cudaError_t launch_layout(const int32_t* topk_idx, int64_t n_slots, int E, int32_t* counts, int32_t* offsets,
                          int32_t* perm, int32_t* inv_perm, int32_t* scratch, int* status, cudaStream_t stream,
                          int* n_launches);

// ---- a1-a5 of a few tokens in one launch (the results of the three stages) -------------------
// x_perm nullptr: no rows move.  Only where small_dispatch_fits (512 experts: 16 keys per lane).  The n_zero words at `zero`
// are set to zero (the counters of the step's next launch).
constexpr int kSmallDispatchMaxTokens = 64, kSmallDispatchMaxSlots = 1024;
bool small_dispatch_fits(int T, int E, int k);
cudaError_t launch_small_dispatch(const float* logits, const float* bias, int T, int E, int k, float scale, int32_t* idx,
                                  float* w, int32_t* counts, int32_t* offsets, int32_t* perm, int32_t* inv_perm,
                                  const void* x, void* x_perm, int H, int* zero, int n_zero, cudaStream_t stream,
                                  int* n_launches);

// ---- a5 permute, a9 combine ----------------------------------------------------------------
// wait_limit_ns: time limit of the kernels' bounded waits (0 = the default of 2 s).
cudaError_t launch_permute(const void* x, const int32_t* inv_perm, void* x_perm, int T, int k, int H, int* status,
                           cudaStream_t stream, int* n_launches, unsigned long long wait_limit_ns = 0);
// Columns [c_begin, c_end) of the rows (c_end < 0: all; multiples of 8).  settled: inv_perm and topk_w were final before the
// previous kernel of the stream started, so the kernel may read its first ones before it waits.
cudaError_t launch_combine(const void* y_perm, const void* y_shared, const int32_t* inv_perm, const float* topk_w,
                           void* out, int T, int k, int H, int* status, cudaStream_t stream, int* n_launches,
                           unsigned long long wait_limit_ns = 0, int c_begin = 0, int c_end = -1, bool settled = false);

// Tensor maps of one launch of the swap-AB kernels (host memory, opaque outside swap_ab.cuh).  A context keeps one plan per
// buffer set and pass; a launch whose operands (addresses and shapes) are the plan's re-encodes nothing.  (Looking 34
// maps up per launch in a locked table costs 3.4 us of host time, in steps that take the GPU 20.)
struct StreamPlan;
StreamPlan* stream_plan_create();
void stream_plan_destroy(StreamPlan* plan);
int64_t stream_plan_encoded(const StreamPlan* plan);  // maps encoded since the plan was created

// ---- a6-a8 grouped GEMM --------------------------------------------------------------------
// One grouped GEMM pass:  out[r, :] = epilogue( A[r, :] . W[e]^T )  for r in expert e's segment.
//   gated:     W[e] is [2*n_feat, K]; out[r,i] = silu(A.W[e,i]) * (A.W[e,n_feat+i]),  i < n_feat
//   not gated: W[e] is [n_feat, K];   out[r,c] = A.W[e,c]
// offsets == nullptr means a single group of `fixed_rows` rows (the shared expert).
struct GemmProblem {
  const void* A;           // bf16 [rows_cap, K]
  const void* W;           // bf16 [E, (gated?2:1)*n_feat, K]
  void* out;               // bf16 [rows_cap, n_feat]
  const int32_t* offsets;  // [E+1] device, or nullptr
  int32_t fixed_rows;      // rows when offsets == nullptr
  int64_t rows_cap;        // rows addressable in A / out (capacity of the buffers)
  int64_t rows_bound;      // upper bound on the rows actually routed this call (T*k or T)
  int32_t E;               // experts in W and offsets
  int32_t n_feat;
  int32_t K;
  bool gated;
  int32_t e_begin = 0;     // this launch covers experts [e_begin, e_end) only (a prefill segment);
  int32_t e_end = -1;      // e_end < 0 means E
  int32_t f_begin = 0;     // ... and output features [f_begin, f_end) only (f_begin a multiple of 256; f_end < 0 means
  int32_t f_end = -1;      // n_feat); a dense group in the same launch then has the same n_feat and range
  // Row gather (bf16 gated pass of the large-M kernel, and of the small-M kernel above kGemmOverlapMaxRows rows): when gather_src
  // is set, A is not read; row p of the operand is gather_src[perm[p] / top_k, :] instead (gather_src is bf16 [T, K], perm is
  // [rows_bound]).
  const void* gather_src = nullptr;
  const int32_t* perm = nullptr;
  int32_t top_k = 1;
  // FP8 variant (tensor-core path only): A and W hold E4M3 codes; the result is scaled by
  // row_scale[row] * w_scale[expert, weight row] (w_scale: [E, (gated?2:1)*n_feat]) before the epilogue's maths.
  bool fp8 = false;
  const float* row_scale = nullptr;
  const float* w_scale = nullptr;
  // Bounded waits of the tensor-core kernels: time limit in nanoseconds (0 = the default of 2 s), and the
  // failure-detection hook (the TMA producer issues nothing, so every consumer wait runs into the limit).
  unsigned long long wait_limit_ns = 0;
  bool debug_stall = false;
  // Swap-AB kernels: two words of device memory, {next tile, CTAs (pairs) that take no more}, zero before the launch; the
  // launch's CTAs take their tiles from the first (an atomic counter over the size-ordered tile list) and the last one that
  // finds none left puts both back to zero.  Consecutive launches of a stream must use different pairs: with the launch overlap the
  // next kernel's CTAs take tiles while this one's are still finishing.
  int* tile_counters = nullptr;
  // Preemption at tile granularity (small-M kernel only; both null = off).  Before it takes a tile a CTA reads
  // *yield_req; when it is non-zero the CTA finishes the tiles it has taken, adds one to *stopped and exits, and the
  // tile counter is left where it is: launching the same problem again with the same tile_counters goes on with the
  // tiles not yet taken.
  const int* yield_req = nullptr;
  int* stopped = nullptr;
  // Every launch of a pass that may be stopped and launched again sets this (also a launch without yield_req that
  // finishes such a pass): all its tiles come from the counter, none is dealt statically.
  bool resumable = false;
  // Small-M kernel: `offsets` was final before the previous kernel of the stream started (behind a quantisation that
  // releases early: before the kernel in front of that one started), so the kernel may read it (and fetch weights) before
  // it waits; only the rows of A (and the FP8 row scales) wait.
  bool offsets_settled = false;
  // Upper bound on the rows of any one group (a token reaches an expert at most once, so T), or 0 if unknown.  With
  // at most 16, every non-empty group is one tile of the same cost and the small-M kernel skips ordering them.
  int32_t max_group_rows = 0;
  StreamPlan* plan = nullptr;  // swap-AB kernels: the launch's tensor maps
};

// A dense group (the shared expert) that rides in the same launch as a grouped problem: its tiles are added
// to the tile list, so a pass that would fill only a few CTAs by itself shares the persistent grid.
struct GemmDenseGroup {
  const void* A;    // bf16 [rows, K]
  const void* W;    // bf16 [(gated?2:1)*n_feat, K]
  void* out;        // bf16 [rows, n_feat]
  int32_t rows;
  int32_t n_feat;
  int32_t K;
  const float* row_scale = nullptr;  // FP8 variant: [rows]
  const float* w_scale = nullptr;    // FP8 variant: [(gated?2:1)*n_feat]
};

// ---- a6-a9 of a few tokens in one launch (step_ffn.cu) ---------------------------------------
// bf16; behind launch_small_dispatch, which zeroed the counters.
constexpr int kStepMaxTokens = 64;
struct StepFfn {
  int E = 0, T = 0, k = 0, H = 0, I = 0, Is = 0;  // Is = 0: no shared expert
  int64_t rows_cap = 0;                           // rows of x and act
  const void *w1 = nullptr, *w2 = nullptr, *w1_sh = nullptr, *w2_sh = nullptr;  // gated and down weights, the shared expert's
  const void *x = nullptr, *x_sh = nullptr;       // routed rows, token rows
  void *act = nullptr, *act_sh = nullptr, *y = nullptr, *y_sh = nullptr, *out = nullptr;
  const int32_t *offsets = nullptr, *inv_perm = nullptr;
  const float* topk_w = nullptr;
  int* counters = nullptr;  // step_ffn_counters words
  int* status = nullptr;
  unsigned long long wait_limit_ns = 0;
  bool debug_stall = false;
};
struct StepPlan;  // the launch's tensor maps, kept per buffer set
StepPlan* step_plan_create();
void step_plan_destroy(StepPlan* plan);
int64_t step_plan_encoded(const StepPlan* plan);
int step_ffn_counters(int E, int H);
cudaError_t launch_step_ffn(const StepFfn& f, StepPlan* plan, int max_ctas, cudaStream_t stream, int* n_launches);

// FP8 variant: per-row dynamic quantisation of bf16 rows [rows, n] -> E4M3 codes [rows, n] + scale [rows]
// (n a multiple of 16, at most 8192).  A second set of rows of the same length may ride in the launch.
// release_early: the next kernel of the stream may start although neither this launch nor the one before it has finished
// (rules above).  For the quantisation between the two passes: the down pass reads only weights and the offsets, which are
// older than the gated pass, before it waits, so its weights are on their way when the codes are there (V3-shaped FP8
// decode, one token 85.8 us a step without, 84.3 with).
cudaError_t launch_quantize_rows(const void* x, int64_t rows, int n, void* q, float* scale, bool release_early,
                                 cudaStream_t stream, int* n_launches, const void* x2 = nullptr, int64_t rows2 = 0,
                                 void* q2 = nullptr, float* scale2 = nullptr);
// The same for T token rows, whose codes and scales also go to their k places in the dispatch: row inv_perm[t * k + j] of
// q_perm / scale_perm (negative: dropped).  q and scale (token order) may be nullptr.
cudaError_t launch_quantize_move(const void* x, int T, int n, void* q, float* scale, const int32_t* inv_perm, int k,
                                 void* q_perm, float* scale_perm, cudaStream_t stream, int* n_launches);

cudaError_t launch_gemm_validation(const GemmProblem& p, cudaStream_t stream, int* n_launches);

// Tensor-core path (tcgen05 + TMEM + TMA), large-M variant: 128 tokens fill the MMA M dimension.  `max_ctas`
// caps the persistent grid.  Returns cudaErrorNotSupported for shapes it does not handle.
// `dense` (optional) is computed in the same launch with the same `gated` epilogue.
cudaError_t launch_gemm_tc(const GemmProblem& p, const GemmDenseGroup* dense, int max_ctas, int* status,
                           cudaStream_t stream, int* n_launches);
// Weight-streaming variant (swap-AB with the MMA N following each expert's row count, up to 256 tokens per tile,
// operands in a byte ring): the variant for experts of up to a few hundred rows, where the step is bound by the
// bytes the SMs ingest.  Same contract as launch_gemm_tc; row gather in bf16 gated passes above kGemmOverlapMaxRows rows.
cudaError_t launch_gemm_stream(const GemmProblem& p, const GemmDenseGroup* dense, int max_ctas, int* status,
                               cudaStream_t stream, int* n_launches);
// Two-CTA variant (swap-AB, a tile multiplied by a pair of SMs): needs clusters of two CTAs, that is whole pairs of free
// SMs.  Same contract as launch_gemm_tc; no row gather, no preemption.
cudaError_t launch_gemm_pair(const GemmProblem& p, const GemmDenseGroup* dense, int max_ctas, int* status,
                             cudaStream_t stream, int* n_launches);
// One-time driver entry-point lookup for tensor-map encoding; returns false (with a reason) if unavailable.
bool gemm_tc_init(const char** why);

}  // namespace moe
