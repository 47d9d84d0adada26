// Stages a2-a4: per-expert counts, exclusive scan, stable token-to-expert permutation.
//
// The permutation must be bit-exact and run-to-run identical, so no slot is claimed with a global
// atomic.  The flat slots are cut into chunks, one per CTA, and a chunk into 32 runs, one per warp; a warp walks its run
// 32 slots at a time and ranks equal experts inside a step with __match_any_sync, which keeps ascending slot order.
// What a CTA needs beyond its own chunk -- how many slots of each expert lie in earlier chunks, and in all -- it finds out
// by itself, so that no kernel only scans:
//   up to kRecountMaxSlots slots   one launch: every CTA counts the other chunks too (a few slots per thread);
//   more                           a launch that counts each chunk, then the same kernel reading those counts.
// The arithmetic is nothing; what it costs is launches, dependent round trips and the slots one SM can walk.  Back to
// back in a CUDA graph: 512 slots of 256 experts 3.2 us, 5600 5.9, 12248 of 128 6.8, 32768 of 512 8.5, 65536 of 128 7.9,
// 262144 of 256 12.2.  (Recounting up to 32768 slots instead of 16384: 0.3 us less at 20000, 0.5 more at 32000.)
// How the slots are cut into chunks: rules.h.
#include <mutex>

#include "kernels.h"
#include "routing.cuh"
#include "rules.h"

namespace moe {
namespace {

constexpr int kWarps = 32;                // warps (= runs) per CTA
constexpr int kThreads = 32 * kWarps;
constexpr int64_t kRecountMaxSlots = 16384;  // see above
constexpr int kBatch = 8;                 // loads issued together (latency hiding)

// Counts the slots [f0, f1) into hist[0..E) with all threads of the CTA (integer adds commute: the count does not
// depend on their order).
__device__ __forceinline__ void count_slots(const int32_t* __restrict__ topk_idx, int64_t f0, int64_t f1, int E, int* hist,
                                            int* status) {
  for (int64_t base = f0; base < f1; base += (int64_t)kThreads * kBatch) {
    int ev[kBatch];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int64_t f = base + u * kThreads + threadIdx.x;
      ev[u] = (f < f1) ? __ldg(topk_idx + f) : -2;
    }
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      if (base + u * kThreads + threadIdx.x >= f1) continue;
      if (ev[u] >= 0 && ev[u] < E) atomicAdd(&hist[ev[u]], 1);
      else flag_status(status, kStBadIndex);
    }
  }
}

// chunk_counts[chunk][e] of the CTA's chunk.
__global__ void __launch_bounds__(kThreads)
layout_count_kernel(const int32_t* __restrict__ topk_idx, int64_t n_slots, int E, int chunk,
                    int32_t* __restrict__ chunk_counts, int* status) {
  extern __shared__ int sh[];
  for (int e = threadIdx.x; e < E; e += kThreads) sh[e] = 0;
  pdl_wait();
  pdl_launch_dependents();
  __syncthreads();
  const int64_t f0 = (int64_t)blockIdx.x * chunk;
  count_slots(topk_idx, f0, min(f0 + chunk, n_slots), E, sh, status);
  __syncthreads();
  for (int e = threadIdx.x; e < E; e += kThreads) chunk_counts[(size_t)blockIdx.x * E + e] = sh[e];
}

// base[e] += counts of the chunks before this CTA's, total[e] += those of the chunks behind it.  A thread takes V
// consecutive experts and every parts-th chunk, kBatch chunks' loads in flight.
template <int V>
__device__ __forceinline__ void sum_chunks(const int32_t* __restrict__ chunk_counts, int E, int* base, int* total) {
  const int EV = E / V, parts = max(1, kThreads / EV), n_chunks = (int)gridDim.x, me = (int)blockIdx.x;
  for (int i = threadIdx.x; i < parts * EV; i += kThreads) {
    const int part = i / EV, e = (i - part * EV) * V;
    int before[V] = {}, after[V] = {};
    for (int q = part; q < n_chunks; q += parts * kBatch) {
      int v[kBatch][V];
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        const int c = q + u * parts;
        const int32_t* src = chunk_counts + (size_t)c * E + e;
        if constexpr (V == 4) {
          const int4 w = c < n_chunks ? *reinterpret_cast<const int4*>(src) : make_int4(0, 0, 0, 0);
          v[u][0] = w.x; v[u][1] = w.y; v[u][2] = w.z; v[u][3] = w.w;
        } else {
          v[u][0] = c < n_chunks ? *src : 0;
        }
      }
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        const int c = q + u * parts;
#pragma unroll
        for (int x = 0; x < V; ++x) {
          if (c < me) before[x] += v[u][x];
          else if (c > me) after[x] += v[u][x];
        }
      }
    }
#pragma unroll
    for (int x = 0; x < V; ++x) {
      if (before[x]) atomicAdd(&base[e + x], before[x]);
      if (after[x]) atomicAdd(&total[e + x], after[x]);
    }
  }
}

// Places the CTA's chunk; CTA 0 also stores counts and offsets.  chunk_counts: every chunk's counts, or nullptr: the
// CTA counts the other chunks itself.
// shared memory: hist[kWarps][E] | base[E] | total[E] | offsets_sh[E+1] | warp_sums[33]
__global__ void __launch_bounds__(kThreads)
layout_place_kernel(const int32_t* __restrict__ topk_idx, int64_t n_slots, int E, int chunk,
                    const int32_t* __restrict__ chunk_counts, int32_t* __restrict__ counts, int32_t* __restrict__ offsets,
                    int32_t* __restrict__ perm, int32_t* __restrict__ inv_perm, int* status) {
  extern __shared__ int sh[];
  int* hist = sh;                 // per warp: counts of its run, then their prefix over the warps before it
  int* base = hist + kWarps * E;  // slots of earlier chunks, then the destination of the chunk's first slot
  int* total = base + E;
  int* offsets_sh = total + E;
  int* warp_sums = offsets_sh + (E + 1);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned lt_mask = (1u << lane) - 1u;
  for (int i = threadIdx.x; i < (kWarps + 2) * E; i += kThreads) sh[i] = 0;
  pdl_wait();
  pdl_launch_dependents();
  const int64_t c0 = (int64_t)blockIdx.x * chunk, c1 = min(c0 + chunk, n_slots);
  const int run = chunk / kWarps;  // a multiple of 32
  const int64_t f0 = min(c0 + (int64_t)warp * run, c1), f1 = min(f0 + run, c1);
  int* mine = hist + warp * E;
  const bool one_step = run == 32;
  // one step: the warp's index and its rank among the step's equals stay in registers
  int e1 = -1, rank1 = 0;
  if (one_step) {
    if (f0 + lane < f1) e1 = __ldg(topk_idx + f0 + lane);
    const bool valid = e1 >= 0 && e1 < E;
    if (f0 + lane < f1 && !valid) flag_status(status, kStBadIndex);
    if (!valid) e1 = -1;
    const unsigned peers = __match_any_sync(0xffffffffu, valid ? e1 : E);  // (the slower, the more values there are)
    rank1 = __popc(peers & lt_mask);
    __syncthreads();  // the counters are zero
    if (valid && rank1 == 0) mine[e1] = __popc(peers);
  } else {
    __syncthreads();
    for (int64_t b = f0; b < f1; b += 32 * kBatch) {
      int ev[kBatch];
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        const int64_t f = b + 32 * u + lane;
        ev[u] = (f < f1) ? __ldg(topk_idx + f) : -2;
      }
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        if (b + 32 * u + lane >= f1) continue;
        if (ev[u] >= 0 && ev[u] < E) atomicAdd(&mine[ev[u]], 1);
        else flag_status(status, kStBadIndex);
      }
    }
  }
  if (gridDim.x > 1) {
    if (chunk_counts == nullptr) {
      count_slots(topk_idx, 0, c0, E, base, nullptr);
      count_slots(topk_idx, c1, n_slots, E, total, nullptr);
    } else if (E % 4 == 0) {
      sum_chunks<4>(chunk_counts, E, base, total);
    } else {
      sum_chunks<1>(chunk_counts, E, base, total);
    }
  }
  __syncthreads();
  // per expert: exclusive prefix over the warps' runs, and the total over all chunks
  for (int e = threadIdx.x; e < E; e += kThreads) {
    const int sum = prefix_over_warps(hist, E, e);
    total[e] += base[e] + sum;  // later chunks, earlier ones, this one
    if (blockIdx.x == 0) counts[e] = total[e];
  }
  __syncthreads();
  block_exclusive_scan(total, E, blockIdx.x == 0 ? offsets : nullptr, offsets_sh, warp_sums);
  for (int e = threadIdx.x; e < E; e += kThreads) base[e] += offsets_sh[e];
  __syncthreads();
  if (one_step) {
    if (f0 + lane < f1) {
      const int p = e1 >= 0 ? base[e1] + mine[e1] + rank1 : -1;
      inv_perm[f0 + lane] = p;
      if (p >= 0) perm[p] = (int32_t)(f0 + lane);
    }
    return;
  }
  for (int64_t b = f0; b < f1; b += 32 * kBatch) {
    int ev[kBatch];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int64_t f = b + 32 * u + lane;
      ev[u] = (f < f1) ? __ldg(topk_idx + f) : -1;
    }
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      if (b + 32 * u >= f1) break;  // uniform across the warp
      const int64_t f = b + 32 * u + lane;
      const int e = ev[u];
      const bool valid = e >= 0 && e < E;
      const unsigned peers = __match_any_sync(0xffffffffu, valid ? e : E);
      int p = -1;
      if (valid) p = base[e] + mine[e] + __popc(peers & lt_mask);
      __syncwarp();
      if (valid && (peers & lt_mask) == 0u) mine[e] += __popc(peers);  // the lowest lane of a group advances it
      __syncwarp();
      if (f < f1) {
        inv_perm[f] = p;
        if (valid) perm[p] = (int32_t)f;
      }
    }
  }
}

__global__ void layout_empty_kernel(int E, int32_t* __restrict__ counts, int32_t* __restrict__ offsets) {
  pdl_wait();
  pdl_launch_dependents();
  for (int e = threadIdx.x; e <= E; e += blockDim.x) {
    if (e < E) counts[e] = 0;
    offsets[e] = 0;
  }
}

}  // namespace

cudaError_t launch_layout(const int32_t* topk_idx, int64_t n_slots, int E, int32_t* counts, int32_t* offsets,
                          int32_t* perm, int32_t* inv_perm, int32_t* scratch, int* status, cudaStream_t stream,
                          int* n_launches) {
  cudaError_t err;
  if (n_slots <= 0) {
    err = launch_pdl(true, layout_empty_kernel, dim3(1), dim3(256), 0, stream, E, counts, offsets);
    if (err == cudaSuccess && n_launches) *n_launches += 1;
    return err;
  }
  const int64_t chunk = layout_chunk_slots(n_slots, E);
  const int n_chunks = (int)((n_slots + chunk - 1) / chunk);
  int n = 1;
  const int32_t* chunk_counts = nullptr;
  if (n_slots > kRecountMaxSlots) {
    if ((err = ensure_dynamic_smem(layout_count_kernel, (size_t)E * sizeof(int))) != cudaSuccess) return err;
    if ((err = launch_pdl(true, layout_count_kernel, dim3(n_chunks), dim3(kThreads), (size_t)E * sizeof(int), stream, topk_idx,
                          n_slots, E, (int)chunk, scratch, status)) != cudaSuccess) return err;
    chunk_counts = scratch;
    ++n;
  }
  const size_t smem = ((size_t)(kWarps + 3) * E + 1 + 33) * sizeof(int);
  if ((err = ensure_dynamic_smem(layout_place_kernel, smem)) != cudaSuccess) return err;
  err = launch_pdl(true, layout_place_kernel, dim3(n_chunks), dim3(kThreads), smem, stream, topk_idx, n_slots, E, (int)chunk,
                   chunk_counts, counts, offsets, perm, inv_perm, status);
  if (err == cudaSuccess && n_launches) *n_launches += n;
  return err;
}

}  // namespace moe

// ------------------------------------------------------------------------------------------------
// Dispatch layout for callers that cannot allocate.
//
// Some hosts of this library are not allowed to obtain device memory at the point where they need a
// layout: code that lives inside another framework's memory pool and must not disturb it, or a runtime
// that has handed all device memory to its own allocator and has no cudaMalloc left to call.  They cannot give a context a workspace either.  For
// them the chunk histograms of the multi-CTA path live in this fixed array instead.  It is part of the
// loaded module, so every GPU that loads the library holds these 256 KiB until the process exits.
#include "../../include/moe_pd.h"

namespace {

constexpr int kStaticScratchInts = 64 * 1024;  // 256 KiB: up to ceil(N/256) * E = 65536 histogram cells
static __device__ __align__(256) int32_t g_static_layout_scratch[kStaticScratchInts];

constexpr int kMaxDevices = 64;
std::mutex g_static_mutex;
int32_t* g_static_scratch_addr[kMaxDevices] = {};  // device address of the array, per device ordinal

}  // namespace

extern "C" moe_status moe_dispatch_layout_static(const int32_t* topk_idx, int32_t T, int32_t top_k,
                                                 int32_t n_experts, int32_t* counts, int32_t* offsets,
                                                 int32_t* perm, int32_t* inv_perm, void* cuda_stream) {
  if (T < 0 || top_k < 1 || n_experts < 1 || n_experts > 1024) return MOE_ERR_INVALID_ARG;
  if (!counts || !offsets || (T > 0 && (!topk_idx || !perm || !inv_perm))) return MOE_ERR_INVALID_ARG;
  const int64_t n_slots = (int64_t)T * top_k;
  if (n_slots > ((int64_t)1 << 30)) return MOE_ERR_CAPACITY;
  if (moe::layout_scratch_ints(n_slots, n_experts) > (size_t)kStaticScratchInts) return MOE_ERR_CAPACITY;

  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return MOE_ERR_CUDA;
  int32_t* scratch = nullptr;
  {
    // Set-up, once per device, with that device current: in host code the array's name is only a
    // stand-in for the symbol, so ask the runtime for the address the kernels must be given.
    std::lock_guard<std::mutex> lock(g_static_mutex);
    if (g_static_scratch_addr[dev] == nullptr) {
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, g_static_layout_scratch) != cudaSuccess || p == nullptr) {
        (void)cudaGetLastError();
        return MOE_ERR_CUDA;
      }
      g_static_scratch_addr[dev] = static_cast<int32_t*>(p);
    }
    scratch = g_static_scratch_addr[dev];
  }
  // Nothing in the scratch has to start at zero: the count kernel writes every cell that the place kernel reads
  // afterwards, so what the previous call left behind is never seen.
  cudaError_t e = moe::launch_layout(topk_idx, n_slots, n_experts, counts, offsets, perm, inv_perm, scratch,
                                     /*status=*/nullptr, static_cast<cudaStream_t>(cuda_stream), nullptr);
  if (e != cudaSuccess) {
    (void)cudaGetLastError();
    return MOE_ERR_CUDA;
  }
  return MOE_OK;
}
