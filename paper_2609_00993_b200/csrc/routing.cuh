// Device code that the routing, the layout and the kernel that does both for a small batch have in common.
#pragma once
#include "kernels.h"

namespace moe {

// Monotone map from a finite float to an unsigned integer (larger float <=> larger integer), so that the
// warp arg-max can use the integer redux instructions.  -0.0 has been folded into +0.0 before the call,
// which keeps the IEEE tie between the two zeros.
__device__ __forceinline__ unsigned ordered_bits(float v) {
  const unsigned u = __float_as_uint(v);
  return u ^ ((unsigned)((int)u >> 31) | 0x80000000u);  // negative: all bits flipped; else the sign bit set
}

// Whether rows of E logits (and the bias) can be read 16 bytes per lane.
inline bool routes_in_vectors(const float* logits, const float* bias, int E) {
  return (E % 128 == 0) && ((reinterpret_cast<uintptr_t>(logits) & 15u) == 0) &&
         (bias == nullptr || (reinterpret_cast<uintptr_t>(bias) & 15u) == 0);
}

// Routes one token with one warp (row: its E logits).  VPT: keys per lane (power of two >= ceil(E/32)).  VEC: lanes own
// runs of 4 consecutive experts.  s_cand, s_sel: 32 words each of the warp's own shared memory.  Lane j < k returns the
// weight of the j-th selected expert and its index in `expert`.
template <int VPT, bool VEC>
__device__ __forceinline__ float route_token(const float* __restrict__ row, const float* __restrict__ bias, int E, int k,
                                             float scale, unsigned long long* s_cand, int* s_sel,
                                             int& expert) {
  const int lane = threadIdx.x & 31;
  // expert owned by this lane's i-th register; increasing in i so that "first wins" keeps the lower index
  auto expert_of = [&](int i) -> int { return VEC ? 128 * (i >> 2) + 4 * lane + (i & 3) : 32 * i + lane; };

  unsigned key[VPT];  // ordered_bits(logit + bias)
  if constexpr (VEC) {
#pragma unroll
    for (int q = 0; q < VPT / 4; ++q) {
      const int e0 = 128 * q + 4 * lane;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (e0 < E) {
        v = *reinterpret_cast<const float4*>(row + e0);
        if (bias != nullptr) {
          const float4 b = *reinterpret_cast<const float4*>(bias + e0);
          v.x = __fadd_rn(v.x, b.x); v.y = __fadd_rn(v.y, b.y); v.z = __fadd_rn(v.z, b.z); v.w = __fadd_rn(v.w, b.w);
        }
      }
      key[4 * q + 0] = ordered_bits(v.x + 0.0f); key[4 * q + 1] = ordered_bits(v.y + 0.0f);
      key[4 * q + 2] = ordered_bits(v.z + 0.0f); key[4 * q + 3] = ordered_bits(v.w + 0.0f);
    }
  } else {
#pragma unroll
    for (int i = 0; i < VPT; ++i) {
      const int e = 32 * i + lane;
      float v = 0.f;
      if (e < E) {
        v = row[e];
        if (bias != nullptr) v = __fadd_rn(v, bias[e]);
      }
      key[i] = ordered_bits(v + 0.0f);
    }
  }

  // ---- selection.  Fast path: the k-th largest of the 32 lane maxima is a threshold that at least k keys reach
  // (the maxima of k different lanes); the keys that reach it -- typically k to 2k of them -- are the only
  // candidates, and each is ranked exactly against the others (key descending, expert index ascending).  When
  // ties put more than 32 keys at or above the threshold the k-round warp arg-max below takes over.
  int my_e = 0;  // lane j (< k) ends up holding the j-th selected expert
  unsigned lmax = 0u;  // 0 is below the image of every float
#pragma unroll
  for (int i = 0; i < VPT; ++i)
    if (expert_of(i) < E) lmax = max(lmax, key[i]);
  unsigned tau = 0u, cur = lmax;
  for (int j = 0; j < k; ++j) {
    tau = __reduce_max_sync(0xffffffffu, cur);
    const unsigned holders = __ballot_sync(0xffffffffu, cur == tau);
    if (lane == __ffs(holders) - 1) cur = 0u;  // remove one holder per round
  }
  // One pass compacts the candidates into the warp's list (any order) as (key image << 32 | ~expert index) -- a
  // larger entry comes earlier in (key descending, expert index ascending) -- and counts them; places beyond the
  // list's 32 are not written.
  unsigned lt_mask;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(lt_mask));
  int n_cand = 0;
#pragma unroll
  for (int i = 0; i < VPT; ++i) {
    const bool c = expert_of(i) < E && key[i] >= tau;
    const unsigned b = __ballot_sync(0xffffffffu, c);
    const int pos = n_cand + __popc(b & lt_mask);
    if (c && pos < 32) s_cand[pos] = ((unsigned long long)key[i] << 32) | (unsigned)(0x7fffffff - expert_of(i));
    n_cand += __popc(b);
  }
  if (n_cand <= 32) {
    // rank each candidate against all
    __syncwarp();
    if (lane < n_cand) {
      const unsigned long long pc = s_cand[lane];
      int rank = 0;
      for (int q = 0; q < n_cand; ++q) rank += s_cand[q] > pc ? 1 : 0;
      if (rank < k) s_sel[rank] = 0x7fffffff - (int)(unsigned)(pc & 0xffffffffull);
    }
    __syncwarp();
    if (lane < k) my_e = s_sel[lane];
  } else {
    unsigned taken = 0u;  // bit i: this lane's i-th key is already selected
    for (int j = 0; j < k; ++j) {
      unsigned bv = 0u;
      int be = 0x7fffffff;
      bool has = false;
#pragma unroll
      for (int i = 0; i < VPT; ++i) {
        const int e = expert_of(i);
        const bool avail = (e < E) && !((taken >> i) & 1u);
        if (avail && (!has || key[i] > bv)) {
          bv = key[i]; be = e; has = true;
        }
      }
      // warp arg-max on (key descending, expert index ascending): largest key, then the lowest index holding it
      const unsigned top = __reduce_max_sync(0xffffffffu, has ? bv : 0u);
      const int win = (int)__reduce_min_sync(0xffffffffu, (unsigned)((has && bv == top) ? be : 0x7fffffff));
      const int owner = VEC ? ((win & 127) >> 2) : (win & 31);
      const int slot = VEC ? (4 * (win >> 7) + (win & 3)) : (win >> 5);
      if (lane == owner) taken |= (1u << slot);
      if (lane == j) my_e = win;
    }
  }

  const bool active = lane < k;
  const float l = active ? row[my_e] : -INFINITY;
  float m = l;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
  const float p = active ? expf(l - m) : 0.f;
  float s = 0.f;
  for (int j = 0; j < k; ++j) s += __shfl_sync(0xffffffffu, p, j);  // summed in j order
  expert = my_e;
  return scale * p / s;
}

__device__ __forceinline__ void flag_status(int* status, int code) {
  if (status != nullptr) atomicCAS(status, kStOk, code);
}

// Block-wide exclusive scan of counts[0..E) -> offsets[0..E]; E <= 1024, blockDim.x a multiple of 32 and >= E...
// handled in rounds of blockDim.x so that any E works.  `warp_sums` is 33 ints of shared scratch.
__device__ __forceinline__ void block_exclusive_scan(const int* counts_sh, int E, int32_t* __restrict__ offsets_out, int* offsets_sh,
                                     int* warp_sums) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  int carry = 0;
  for (int base = 0; base < E; base += blockDim.x) {
    const int e = base + threadIdx.x;
    const int v = (e < E) ? counts_sh[e] : 0;
    int incl = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int n = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += n;
    }
    if (lane == 31) warp_sums[warp] = incl;
    __syncthreads();
    if (warp == 0) {
      int ws = (lane < nwarps) ? warp_sums[lane] : 0;
      int wincl = ws;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const int n = __shfl_up_sync(0xffffffffu, wincl, off);
        if (lane >= off) wincl += n;
      }
      if (lane < nwarps) warp_sums[lane] = wincl - ws;  // exclusive prefix of the warp totals
      if (lane == 31) warp_sums[32] = wincl;            // total of this round
    }
    __syncthreads();
    const int excl = carry + warp_sums[warp] + incl - v;
    if (e < E) {
      offsets_sh[e] = excl;
      if (offsets_out != nullptr) offsets_out[e] = excl;
    }
    carry += warp_sums[32];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    offsets_sh[E] = carry;
    if (offsets_out != nullptr) offsets_out[E] = carry;
  }
  __syncthreads();
}

// Exclusive prefix of the 32 warps' counts hist[warp][e], in place; returns their sum.
__device__ __forceinline__ int prefix_over_warps(int* hist, int E, int e) {
  int sum = 0;
#pragma unroll
  for (int w0 = 0; w0 < 32; w0 += 16) {  // 16 reads in flight
    int v[16];
#pragma unroll
    for (int w = 0; w < 16; ++w) v[w] = hist[(w0 + w) * E + e];
#pragma unroll
    for (int w = 0; w < 16; ++w) {
      hist[(w0 + w) * E + e] = sum;
      sum += v[w];
    }
  }
  return sum;
}

}  // namespace moe
