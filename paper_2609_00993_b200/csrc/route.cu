// Stage a1: top-k routing over given router logits.  One warp per token; each lane keeps
// ceil(E/32) selection keys in registers (128-bit loads when E is a multiple of 128) as order-preserving integer
// images.  Selection: k warp maxima over the lanes' own maxima give a threshold that at least k keys reach; the few
// keys that reach it are compacted into a per-warp list and each is ranked exactly against the others (key
// descending, expert index ascending).  Only when ties put more than 32 keys at the threshold do k rounds of a
// warp arg-max over all keys run instead (redux.sync: a max over the key images, then a min over the expert
// indices that hold it).  The routed weights are a max-subtracted softmax over the k selected
// unbiased logits, summed in selection order.
#include "kernels.h"
#include "routing.cuh"

namespace moe {
namespace {

constexpr int kWarpsPerBlock = 8;

// VPT: keys per lane (power of two >= ceil(E/32)).  VEC: lanes own runs of 4 consecutive experts.
template <int VPT, bool VEC>
__global__ void __launch_bounds__(kWarpsPerBlock * 32)
route_kernel(const float* __restrict__ logits, const float* __restrict__ bias, int T, int E, int k, float scale,
             int32_t* __restrict__ idx, float* __restrict__ w) {
  pdl_wait();
  pdl_launch_dependents();
  const int lane = threadIdx.x & 31;
  const int t = blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5);
  if (t >= T) return;
  __shared__ unsigned long long s_cand[kWarpsPerBlock][32];
  __shared__ int s_sel[kWarpsPerBlock][32];
  const int wib = threadIdx.x >> 5;
  int e;
  const float weight = route_token<VPT, VEC>(logits + (size_t)t * E, bias, E, k, scale, s_cand[wib], s_sel[wib], e);
  if (lane < k) {
    idx[(size_t)t * k + lane] = e;
    w[(size_t)t * k + lane] = weight;
  }
}

template <int VPT>
cudaError_t launch_vpt(bool vec, const float* logits, const float* bias, int T, int E, int k, float scale,
                       int32_t* idx, float* w, cudaStream_t stream) {
  const int blocks = (T + kWarpsPerBlock - 1) / kWarpsPerBlock;
  cudaError_t err = cudaSuccess;
  if constexpr (VPT >= 4) {
    if (vec) {
      if ((err = ensure_dynamic_smem(route_kernel<VPT, true>, 0)) != cudaSuccess) return err;
      return launch_pdl(true, route_kernel<VPT, true>, dim3(blocks), dim3(kWarpsPerBlock * 32), 0, stream, logits, bias, T, E, k,
                        scale, idx, w);
    }
  }
  if ((err = ensure_dynamic_smem(route_kernel<VPT, false>, 0)) != cudaSuccess) return err;
  return launch_pdl(true, route_kernel<VPT, false>, dim3(blocks), dim3(kWarpsPerBlock * 32), 0, stream, logits, bias, T, E, k, scale,
                    idx, w);
}

}  // namespace

cudaError_t launch_route(const float* logits, const float* bias, int T, int E, int k, float scale, int32_t* idx,
                         float* w, cudaStream_t stream, int* n_launches) {
  if (T <= 0) return cudaSuccess;
  const int per_lane = (E + 31) / 32;
  const bool vec = routes_in_vectors(logits, bias, E);
  cudaError_t err;
  if (per_lane <= 1) err = launch_vpt<1>(false, logits, bias, T, E, k, scale, idx, w, stream);
  else if (per_lane <= 2) err = launch_vpt<2>(false, logits, bias, T, E, k, scale, idx, w, stream);
  else if (per_lane <= 4) err = launch_vpt<4>(vec, logits, bias, T, E, k, scale, idx, w, stream);
  else if (per_lane <= 8) err = launch_vpt<8>(vec, logits, bias, T, E, k, scale, idx, w, stream);
  else if (per_lane <= 16) err = launch_vpt<16>(vec, logits, bias, T, E, k, scale, idx, w, stream);
  else err = launch_vpt<32>(vec, logits, bias, T, E, k, scale, idx, w, stream);
  if (err == cudaSuccess && n_launches) *n_launches += 1;
  return err;
}

}  // namespace moe
