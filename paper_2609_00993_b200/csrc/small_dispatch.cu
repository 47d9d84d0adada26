// Stages a1-a5 of up to 64 tokens in one launch: routing, layout and row movement.
// At this size each of the three is latency -- a launch, a round trip to memory, a few scans -- and the gated pass waits for
// them in a row.  Here every CTA has the routing of all tokens itself: it routes them, a warp each, with the logits out of
// L2, or from 17 tokens on a cluster shares the work and hands the expert indices round through distributed shared memory.
// It then finds the positions of its own token's slots by counting (no scan, no round trip), and copies its piece of that
// token's row, which it has loaded meanwhile.
// Whole steps, this launch | the three, us: 8 experts, 2 of them, 256 features: 1 token 21.1 | 24.1, 16 21.6 | 24.6, 64
// 22.6 | 24.5; 128 experts, 8 of them, 2048 features: 1 token 34.9 | 36.8, 16 133.2 | 135.4, 37 180.8 | 182.2, 64 199.4 |
// 200.9; 512 experts, 8 of them: 1 token 31.2 | 33.4, 32 82.0 | 85.1.
// (In one CTA, two tokens a warp at 64: 23.9 | 24.5 and 201.3 | 200.9.  128 tokens over a cluster: 23.9 | 25.2 with 8
// experts but 207.6 | 206.1 with 128, so 64 is the limit.)
// Beside another phase without SM budgets the clusters of 8 start as soon as the three launches did: decode steps of 64
// tokens beside back-to-back V3-shaped prefill of 4096 take 3.35 ms on average, 3.55 in a build that makes three launches.
#include "kernels.h"
#include "routing.cuh"

namespace moe {
namespace {

constexpr int kMaxThreads = 512, kMaxExperts = 512;

// How many of the n indices s[] (padded to a multiple of 4 with INT_MAX) are below e, and how many of the first `limit`
// equal it.
__device__ __forceinline__ int2 count_alone(const int* s, int n, int e, int limit) {
  int below = 0, equal = 0;
  for (int g = 0; g < n; g += 4) {
    const int4 v = *reinterpret_cast<const int4*>(s + g);
    below += (v.x < e) + (v.y < e) + (v.z < e) + (v.w < e);
    equal += (v.x == e && g < limit) + (v.y == e && g + 1 < limit) + (v.z == e && g + 2 < limit) + (v.w == e && g + 3 < limit);
  }
  return make_int2(below, equal);
}
// ... by a warp.
__device__ __forceinline__ int2 count_together(const int* s, int n, int e, int limit) {
  int below = 0, equal = 0;
  for (int g = threadIdx.x & 31; g < n; g += 32) {
    const int v = s[g];
    below += v < e;
    equal += v == e && g < limit;
  }
  __syncwarp();
  return make_int2((int)__reduce_add_sync(0xffffffffu, (unsigned)below), (int)__reduce_add_sync(0xffffffffu, (unsigned)equal));
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
// Stores v at the same place of CTA `rank` of the cluster.
__device__ __forceinline__ void store_in_cta(int* p, int rank, int v) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

// grid (pieces of a row, T rounded up to whole clusters of n_ranks CTAs).  VPT, VEC: as in the routing kernel.
// x_perm == nullptr: no rows move.  CTA r of a cluster routes the tokens r * warps + warp for all of them.
// The first cluster of a row's first piece writes the routing; the CTAs of first pieces write the positions of their own
// token's slots and the counts and offsets of their share of the experts.
template <int VPT, bool VEC>
__global__ void __launch_bounds__(kMaxThreads)
small_dispatch_kernel(const float* __restrict__ logits, const float* __restrict__ bias, int T, int E, int k, float scale,
                      int32_t* __restrict__ idx, float* __restrict__ w, int32_t* __restrict__ counts,
                      int32_t* __restrict__ offsets, int32_t* __restrict__ perm, int32_t* __restrict__ inv_perm,
                      const uint4* __restrict__ x, uint4* __restrict__ x_perm, int row_vecs, int n_ranks, int* __restrict__ zero,
                      int n_zero) {
  __shared__ unsigned long long s_cand[kMaxThreads / 32][32];
  __shared__ int s_sel[kMaxThreads / 32][32];
  __shared__ __align__(16) int s_idx[kSmallDispatchMaxSlots + 4];
  __shared__ int s_pos[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5, n = T * k;
  const int t = blockIdx.y, col = blockIdx.x * blockDim.x + threadIdx.x;
  const int rank = n_ranks > 1 ? t % n_ranks : 0;
  if (n_ranks > 1) cluster_arrive();  // this CTA has started
  pdl_wait();
  pdl_launch_dependents();
  uint4 piece;
  const bool moves = x_perm != nullptr && t < T && col < row_vecs;
  if (moves) piece = x[(size_t)t * row_vecs + col];
  if (blockIdx.x == 0)
    for (int i = t * (int)blockDim.x + (int)threadIdx.x; i < n_zero; i += (int)(gridDim.y * blockDim.x)) zero[i] = 0;
  const int q = rank * n_warps + warp;
  int e = 0;
  if (q < T) {
    const float weight = route_token<VPT, VEC>(logits + (size_t)q * E, bias, E, k, scale, s_cand[warp], s_sel[warp], e);
    if (lane < k && blockIdx.x == 0 && t == rank) {
      idx[q * k + lane] = e;
      w[q * k + lane] = weight;
    }
  }
  if (n_ranks > 1) {
    cluster_wait();
    if (q < T && lane < k)
      for (int r = 0; r < n_ranks; ++r) store_in_cta(&s_idx[q * k + lane], r, e);
    if (threadIdx.x < 4) s_idx[n + threadIdx.x] = 0x7fffffff;
    cluster_arrive();
    cluster_wait();
  } else {
    if (q < T && lane < k) s_idx[q * k + lane] = e;
    if (threadIdx.x < 4) s_idx[n + threadIdx.x] = 0x7fffffff;
    __syncthreads();
  }
  if (t >= T) return;
  for (int j = warp; j < k; j += n_warps) {
    const int f = t * k + j;
    const int2 c = count_together(s_idx, n, s_idx[f], f);
    if (lane == 0) s_pos[j] = c.x + c.y;
  }
  if (blockIdx.x == 0) {
    const int share = (E + T - 1) / T, e0 = t * share, e1 = min(e0 + share, E);
    // a warp's count of one expert takes as long as a thread's of 32 indices (8 experts of 40 slots a warp instead: +1 us)
    if (n <= 32 * ((share + n_warps - 1) / n_warps)) {
      for (int i = e0 + (int)threadIdx.x; i < e1; i += (int)blockDim.x) {
        const int2 c = count_alone(s_idx, n, i, n);
        offsets[i] = c.x;
        counts[i] = c.y;
      }
    } else {
      for (int i = e0 + warp; i < e1; i += n_warps) {
        const int2 c = count_together(s_idx, n, i, n);
        if (lane == 0) {
          offsets[i] = c.x;
          counts[i] = c.y;
        }
      }
    }
    if (t == 0 && threadIdx.x == 0) offsets[E] = n;
  }
  __syncthreads();
  if (moves)
    for (int j = 0; j < k; ++j) x_perm[(size_t)s_pos[j] * row_vecs + col] = piece;
  if (blockIdx.x == 0 && threadIdx.x < k) {
    const int p = s_pos[threadIdx.x], f = t * k + (int)threadIdx.x;
    inv_perm[f] = p;
    perm[p] = f;
  }
}

}  // namespace

bool small_dispatch_fits(int T, int E, int k) {
  return T >= 1 && T <= kSmallDispatchMaxTokens && T * k <= kSmallDispatchMaxSlots && E <= kMaxExperts;
}

cudaError_t launch_small_dispatch(const float* logits, const float* bias, int T, int E, int k, float scale, int32_t* idx,
                                  float* w, int32_t* counts, int32_t* offsets, int32_t* perm, int32_t* inv_perm,
                                  const void* x, void* x_perm, int H, int* zero, int n_zero, cudaStream_t stream,
                                  int* n_launches) {
  const bool vec = routes_in_vectors(logits, bias, E);
  const int per_lane = (E + 31) / 32, row_vecs = H / 8;
  // A warp per token.  More warps in a CTA than 16 are in one another's way (32 tokens in one CTA of 1024 threads instead of
  // two of 512: level with 8 experts, 0.2 us more with 128); a cluster costs 0.5 to 1 us by itself (16 tokens in two CTAs
  // of 256 threads instead of one of 512: 22.6 against 21.6 us, 134.1 against 133.2).  From 33 tokens on eight CTAs of 256
  // threads and four of 512 are level.
  const int n_ranks = T <= 16 ? 1 : T <= 32 ? 2 : 8, threads = T <= 8 || T > 32 ? 256 : 512;
  const dim3 grid(x_perm ? (row_vecs + threads - 1) / threads : 1, (T + n_ranks - 1) / n_ranks * n_ranks);
  auto go = [&](auto kern) {
    const cudaError_t err = ensure_dynamic_smem(kern, 0);
    if (err != cudaSuccess) return err;
    return launch_pdl_clusters(true, n_ranks, kern, grid, dim3(threads), 0, stream, logits, bias, T, E, k, scale, idx, w, counts,
                               offsets, perm, inv_perm, static_cast<const uint4*>(x), static_cast<uint4*>(x_perm), row_vecs,
                               n_ranks, zero, n_zero);
  };
  cudaError_t err;
  if (per_lane <= 1) err = go(small_dispatch_kernel<1, false>);
  else if (per_lane <= 2) err = go(small_dispatch_kernel<2, false>);
  else if (per_lane <= 4) err = vec ? go(small_dispatch_kernel<4, true>) : go(small_dispatch_kernel<4, false>);
  else if (per_lane <= 8) err = vec ? go(small_dispatch_kernel<8, true>) : go(small_dispatch_kernel<8, false>);
  else err = vec ? go(small_dispatch_kernel<16, true>) : go(small_dispatch_kernel<16, false>);
  if (err == cudaSuccess && n_launches) *n_launches += 1;
  return err;
}

}  // namespace moe
