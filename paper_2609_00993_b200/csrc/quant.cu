// FP8 precision variant: per-row dynamic quantisation of bf16 activation rows to E4M3.
//
//   amax  = max(max_i |v_i|, 2^-100)       scale = amax / 448,  inv = 448 / amax
//   code_i = e4m3(v_i * inv)               round to nearest even, saturating at +-448
//
// The codes are integers decided by floating point, so every operation that decides them is spelled out in
// IEEE fp32 (__fdiv_rn once per row, __fmul_rn per element, cvt.rn.satfinite) and nothing is contracted or
// approximated.
// One warp (rows of up to 2048 elements) or one CTA of 128 threads (up to 8192) per row; the row stays in
// registers between the two passes, so it is read once: 2 n bytes in, n + 4 bytes out per row.  The kernel is compiled
// for the number of 16-element pieces a thread holds (1..4): what bounds it on short rows is instructions, and with four
// pieces for every row a quarter to three quarters of them handled pieces that are not there.
// The quantised row may go to several places: MOVE writes it to its k destination rows of the dispatch (k n bytes) and,
// when the shared expert needs it, in token order too -- from registers, so that no second kernel reads it back.
// Bound by HBM on long steps: hidden 2560, 512 experts, T = 20000 moves x in 93 us (164 with eight 8-element vectors a
// thread for every row and a row movement of its own) and quantises the activation in 79 (125); Qwen3-shaped layer,
// T = 6007 25.1 (37.8) and 22.9 (35.0).
#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include "kernels.h"

namespace moe {
namespace {

constexpr int kQuantThreads = 128;
constexpr int kQuantMaxPieces = 4;  // 16-element pieces per thread

__device__ __forceinline__ float bf16_bits_to_f32(uint32_t bits16) { return __uint_as_float(bits16 << 16); }

__device__ __forceinline__ uint32_t e4m3x2(float lo, float hi) {
  return (uint32_t)__nv_cvt_float2_to_fp8x2(make_float2(lo, hi), __NV_SATFINITE, __NV_E4M3);  // lo in bits 0-7
}

// two bf16 pairs -> four codes
__device__ __forceinline__ uint32_t quantize4(uint32_t w0, uint32_t w1, float inv) {
  return e4m3x2(__fmul_rn(bf16_bits_to_f32(w0 & 0xffffu), inv), __fmul_rn(__uint_as_float(w0 & 0xffff0000u), inv)) |
         (e4m3x2(__fmul_rn(bf16_bits_to_f32(w1 & 0xffffu), inv), __fmul_rn(__uint_as_float(w1 & 0xffff0000u), inv)) << 16);
}

// ROW_WARPS = 4: one CTA per row.  ROW_WARPS = 1: one warp per row, four rows per CTA and no CTA-wide barrier.
// n_pieces: 16-element pieces of a row.  MOVE: row's codes also go to rows inv_perm[row * k + j], j < k, of q_perm
// (negative: dropped), its scale to the same places of scale_perm; q / scale may then be nullptr.
// A second set of rows of the same length (x2, rows2 of them -> q2, scale2) may ride in the launch, behind the first: the
// shared expert's activation in a launch of its own costs 4 us a step (V3-shaped FP8 decode, one token 90.0 against 85.8 us).
template <int ROW_WARPS, int NP, bool MOVE>
__global__ void __launch_bounds__(kQuantThreads)
quantize_rows_kernel(const uint4* __restrict__ x, long long rows, int n_pieces, uint4* __restrict__ q,
                     float* __restrict__ scale, const int32_t* __restrict__ inv_perm, int k, uint4* __restrict__ q_perm,
                     float* __restrict__ scale_perm, const uint4* __restrict__ x2, long long rows2, uint4* __restrict__ q2,
                     float* __restrict__ scale2, bool release_early) {
  __shared__ uint32_t warp_max[kQuantThreads / 32];
  if (release_early) pdl_launch_dependents();  // (see launch_quantize_rows)
  pdl_wait();
  if (!release_early) pdl_launch_dependents();
  constexpr int kRowThreads = 32 * ROW_WARPS;
  const int tid = ROW_WARPS == 1 ? (int)(threadIdx.x & 31) : (int)threadIdx.x;
  long long row = ROW_WARPS == 1 ? (long long)blockIdx.x * (kQuantThreads / 32) + (threadIdx.x >> 5)
                                 : (long long)blockIdx.x;
  if (!MOVE && row >= rows) {
    row -= rows;
    rows = rows2;
    x = x2;
    q = q2;
    scale = scale2;
  }
  if (ROW_WARPS == 1 && row >= rows) return;  // whole warps leave; there is no barrier on this path
  const uint4* xr = x + row * n_pieces * 2;
  int dst = -1;  // MOVE: lane j of every warp holds destination j
  if (MOVE && (int)(threadIdx.x & 31) < k) dst = __ldg(inv_perm + row * k + (threadIdx.x & 31));
  uint4 v[NP][2];
#pragma unroll
  for (int j = 0; j < NP; ++j) {
    const int i = tid + j * kRowThreads;
    v[j][0] = v[j][1] = make_uint4(0u, 0u, 0u, 0u);
    if (i < n_pieces) {
      v[j][0] = xr[2 * i];
      v[j][1] = xr[2 * i + 1];
    }
  }
  // largest |bf16| as a bit pattern, two at a time: for finite values the integer order is the value order
  uint32_t m2 = 0;
#pragma unroll
  for (int j = 0; j < NP; ++j)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      m2 = __vmaxu2(m2, v[j][h].x & 0x7fff7fffu);
      m2 = __vmaxu2(m2, v[j][h].y & 0x7fff7fffu);
      m2 = __vmaxu2(m2, v[j][h].z & 0x7fff7fffu);
      m2 = __vmaxu2(m2, v[j][h].w & 0x7fff7fffu);
    }
  uint32_t m = __reduce_max_sync(0xffffffffu, max(m2 & 0xffffu, m2 >> 16));
  if (ROW_WARPS > 1) {
    if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = m;
    __syncthreads();
    m = max(max(warp_max[0], warp_max[1]), max(warp_max[2], warp_max[3]));
  }
  const float amax = fmaxf(bf16_bits_to_f32(m), 0x1p-100f);
  const float inv = __fdiv_rn(448.f, amax);
  const float sc = __fdiv_rn(amax, 448.f);
  if (tid == 0 && scale != nullptr) scale[row] = sc;
#pragma unroll
  for (int j = 0; j < NP; ++j)
    v[j][0] = make_uint4(quantize4(v[j][0].x, v[j][0].y, inv), quantize4(v[j][0].z, v[j][0].w, inv),
                         quantize4(v[j][1].x, v[j][1].y, inv), quantize4(v[j][1].z, v[j][1].w, inv));
  auto store = [&](uint4* to) {
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      const int i = tid + j * kRowThreads;
      if (i < n_pieces) to[i] = v[j][0];
    }
  };
  if (q != nullptr) store(q + row * n_pieces);
  if (MOVE) {
    if (tid < k && dst >= 0) scale_perm[dst] = sc;
    for (int j = 0; j < k; ++j) {
      const int d = __shfl_sync(0xffffffffu, dst, j);
      if (d >= 0) store(q_perm + (size_t)d * n_pieces);
    }
  }
}

}  // namespace

namespace {

template <bool MOVE>
cudaError_t launch(const void* x, int64_t rows, int n, void* q, float* scale, const int32_t* inv_perm, int k, void* q_perm,
                   float* scale_perm, const void* x2, int64_t rows2, void* q2, float* scale2, bool release_early,
                   cudaStream_t stream, int* n_launches) {
  if (rows <= 0) return cudaSuccess;
  if (n <= 0 || n % 16 != 0 || n > 16 * kQuantThreads * kQuantMaxPieces || rows + rows2 > 0x7fffffffLL || k > 32)
    return cudaErrorNotSupported;
  const int pieces = n / 16;
  const bool warp_row = pieces <= 32 * kQuantMaxPieces;
  const int np = warp_row ? (pieces + 31) / 32 : (pieces + kQuantThreads - 1) / kQuantThreads;
  const int64_t all = rows + rows2;
  const unsigned blocks = (unsigned)(warp_row ? (all + kQuantThreads / 32 - 1) / (kQuantThreads / 32) : all);
  auto go = [&](auto kern) -> cudaError_t {
    cudaError_t e = ensure_dynamic_smem(kern, 0);
    if (e != cudaSuccess) return e;
    return launch_pdl(true, kern, dim3(blocks), dim3(kQuantThreads), 0, stream, static_cast<const uint4*>(x), (long long)rows,
                      pieces, static_cast<uint4*>(q), scale, inv_perm, k, static_cast<uint4*>(q_perm), scale_perm,
                      static_cast<const uint4*>(x2), (long long)rows2, static_cast<uint4*>(q2), scale2, release_early);
  };
  cudaError_t err;
  if (warp_row)
    err = np == 1 ? go(quantize_rows_kernel<1, 1, MOVE>) : np == 2 ? go(quantize_rows_kernel<1, 2, MOVE>)
        : np == 3 ? go(quantize_rows_kernel<1, 3, MOVE>) : go(quantize_rows_kernel<1, 4, MOVE>);
  else  // more than 2048 elements: two pieces per thread at least
    err = np == 2 ? go(quantize_rows_kernel<4, 2, MOVE>) : np == 3 ? go(quantize_rows_kernel<4, 3, MOVE>)
                                                         : go(quantize_rows_kernel<4, 4, MOVE>);
  if (err == cudaSuccess && n_launches) *n_launches += 1;
  return err;
}

}  // namespace

cudaError_t launch_quantize_rows(const void* x, int64_t rows, int n, void* q, float* scale, bool release_early,
                                 cudaStream_t stream, int* n_launches, const void* x2, int64_t rows2, void* q2,
                                 float* scale2) {
  return launch<false>(x, rows, n, q, scale, nullptr, 0, nullptr, nullptr, x2, rows2, q2, scale2, release_early, stream,
                       n_launches);
}

cudaError_t launch_quantize_move(const void* x, int T, int n, void* q, float* scale, const int32_t* inv_perm, int k,
                                 void* q_perm, float* scale_perm, cudaStream_t stream, int* n_launches) {
  return launch<true>(x, T, n, q, scale, inv_perm, k, q_perm, scale_perm, nullptr, 0, nullptr, nullptr, false, stream,
                      n_launches);
}

}  // namespace moe
