// Stages a6-a9 of a whole bf16 step of up to 64 tokens in one launch (sm_100a): gated pass, down pass and combine, the weights
// streamed through the tensor cores as in gemm_stream.cu.
//
// A step of a few tokens is a chain of launches that each wait for the one before to end and then for their first copies, and
// its passes have fewer tiles than there are SMs.  Here the tiles of both passes are one list, taken from a counter:
//   tile       (group, feature tile): 128 weight rows fill the MMA M dimension -- gated pass 64 features, 16 gate rows and the
//              16 matching up rows in turn -- and the group's rows, at most 64, are N.  A group is an expert with rows, or
//              the shared expert.  Half the tile of gemm_stream.cu, because what an SM takes in (about 70 GB/s) is what bounds a
//              pass of fewer tiles than SMs: eight experts of 768 features are 48 of its tiles.
//   order      every gated tile comes before every down tile.  A CTA that takes a down tile fetches the tile's weights as far
//              as its ring goes, while its rows wait until the group's gated tiles have all been stored (a counter per group):
//              the weights keep streaming over the seam between the passes.  Whoever holds a tile that is waited for is
//              running and waits for nobody, so this needs no co-residency of the CTAs.
//   combine    (feature tile, 16 tokens) tiles come last: they wait until every group has stored the feature tile.
// The counters are zeroed by the launch that dispatches the step's tokens (small_dispatch.cu).
//
// Bound by HBM where there are tiles enough; else by the chain dispatch 3 us, list and first operands 3, gated tile 2 (0.17 us a
// k-block of four MMAs), its stores seen by another SM 1.5, rows 1.5, down tile 2.5, stores seen 1.5, combine 1 (tiny layer).  Whole
// steps against three launches: rules.h.  With FP8 the quantisation between the passes needs two more trips through L2 inside the
// kernel, and tiles of half the k-blocks: 2048 / 768 x 128, 9 tokens 67.8 us against 61.5 with launches, so it is not taken there.
//
// Warp roles (480 threads): warps 0-7 epilogue (two per TMEM lane group), warp 8 takes the tiles and fetches the weights, warp 9
// issues the MMAs and owns the TMEM, warps 10-13 do what follows a stored tile, warp 14 fetches the rows.  The weights have a
// warp of their own because the stream may not stop for rows that are not there yet, and because a loop that fetches both takes 600
// clocks a k-block, all the time there is at 7 TB/s (64 tokens of the V3-shaped layer 2164 us with one warp, 2105 with two).
// Every wait is bounded: on expiry the kernel records a timeout in the status word, raises a CTA-wide abort flag, lets copies in
// flight land, frees its TMEM and returns.
#include <cuda.h>
#include <cuda_bf16.h>

#include <cstring>
#include <new>

#include "combine.cuh"
#include "kernels.h"
#include "tc_common.cuh"

namespace moe {
namespace {

using namespace tc;

constexpr int kEpilogueWarps = 8;
constexpr int kProducerWarp = kEpilogueWarps;
constexpr int kMmaWarp = kEpilogueWarps + 1;
constexpr int kFinishWarp0 = kEpilogueWarps + 2, kFinishWarps = 4;
constexpr int kRowWarp = kFinishWarp0 + kFinishWarps;
constexpr int kWarps = kRowWarp + 1, kThreads = 32 * kWarps;
constexpr int kMaxGroups = 513;  // 512 experts (small_dispatch_fits) and the shared one
// A k-block takes one slot of the ring, its rows behind its weights, or, with more than 16 rows, a second one for them.
constexpr int kSmallRows = 16;
constexpr int kSlotBytes = kWBoxBytes + kSmallRows * 128;
constexpr int kSlots = 11;
static_assert(kStepMaxTokens * 128 <= kSlotBytes && kSlotBytes % 1024 == 0, "");
constexpr int kAccs = 4;
constexpr uint32_t kAccCols = kStepMaxTokens, kTmemCols = kAccs * kAccCols;
constexpr int kStagingBytes = 1024;  // epilogue, per warp: 16 tokens x 32 features
constexpr int kQ = 4;
// k-blocks before a tile's last at which the next tile's number is asked for (8 and 10 are level on long passes, 10 loses 1 % with 128
// experts, 24 tokens), and k-blocks that are multiplied in one go
constexpr int kTakeAhead = 4, kBatch = 4;
constexpr int kGatedFeat = 64, kDownFeat = 128;  // output features of a tile
constexpr int kCombineTokens = 4 * kFinishWarps;  // tokens of a combine tile: half a warp to two of them
constexpr int kRowMaps = kStepMaxTokens / 16;

struct StepParams {
  const int32_t* offsets;  // [E+1]
  int32_t E, T, k, H, I, Is;  // Is = 0: no shared expert
  __nv_bfloat16 *act, *act_sh, *y, *y_sh, *out;
  const int32_t* inv_perm;
  const float* topk_w;
  // next tile | groups ready | gated tiles stored of each group [E+1] | down tiles stored of each feature tile
  int* ctr;
  int* status;
  unsigned long long wait_limit_ns;
  int32_t inject_producer_stall;
};

struct StepMaps {
  CUtensorMap w1, w2, w1_sh, w2_sh;    // weights: gated, down; of the shared expert
  CUtensorMap x[kRowMaps], a[kRowMaps];  // routed rows of either pass, in boxes of 16, 32, 48, 64 rows
  CUtensorMap x_sh, a_sh;              // the shared expert's: every token's
};

// A tile as the producer hands it to the other roles
enum TileKind { kGated = 0, kDown = 1, kCombine = 2 };
struct __align__(16) Tile {
  int group;  // (combine: the block of tokens); -1: no more
  int kind, ft, unused;
};

__device__ __forceinline__ int load_relaxed(const int* p) {
  int v;
  asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void fence_async_proxy() { asm volatile("fence.proxy.async;" ::: "memory"); }

// A wait for a counter in device memory, by a whole warp; what was counted is visible then.  `all` (or nullptr) is looked at in
// the same round trip.
__device__ __forceinline__ bool wait_count(const int* counter, int want, const int* all, int& all_seen, volatile int* abort_flag,
                                           unsigned long long limit) {
  unsigned long long t0 = 0;
  for (uint32_t polls = 0;; ++polls) {
    const int v = load_relaxed(counter);
    if (all != nullptr) all_seen = load_relaxed(all);
    if (__all_sync(0xffffffffu, v >= want)) break;
    if ((polls & 63u) != 63u) continue;
    const unsigned long long now = global_ns();
    if (t0 == 0) t0 = now;
    if (!__all_sync(0xffffffffu, *abort_flag == 0 && now - t0 <= limit)) return false;
  }
  __threadfence();
  return true;
}

// Eight columns, vector v of a row, of the tokens t0 and t0 + kCombineTokens / 2 (as far as there are): K of their rows at a time,
// so that as many loads are in flight.  Ascending j, then the shared row, as in combine_kernel.
template <int K>
__device__ __forceinline__ void combine_columns(const StepParams& p, const int* s_pos, const float* s_weight, unsigned v, int t0) {
  const uint4* const y = reinterpret_cast<const uint4*>(p.y) + v;
  const unsigned row_vecs = (unsigned)p.H / 8u;  // (at most 1024 rows)
  int tok[2];
  float sum[2][8];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    tok[i] = min(t0 + i * (kCombineTokens / 2), p.T - 1);  // (one that is not there: the last one that is)
#pragma unroll
    for (int c = 0; c < 8; ++c) sum[i][c] = 0.f;
  }
#pragma unroll 1
  for (int j0 = 0; j0 < p.k; j0 += K) {
    uint4 r[2][K];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < K; ++j) r[i][j] = __ldcg(y + (unsigned)s_pos[tok[i] * p.k + min(j0 + j, p.k - 1)] * row_vecs);
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < K; ++j)
        if (j0 + j < p.k) fma_bf16x8(sum[i], r[i][j], s_weight[tok[i] * p.k + j0 + j]);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    if (t0 + i * (kCombineTokens / 2) >= p.T) break;
    if (p.Is > 0) fma_bf16x8(sum[i], __ldcg(reinterpret_cast<const uint4*>(p.y_sh) + v + (unsigned)tok[i] * row_vecs), 1.0f);
    reinterpret_cast<uint4*>(p.out)[v + (unsigned)tok[i] * row_vecs] = bf16x8(sum[i]);
  }
}

__global__ void __launch_bounds__(kThreads, 1)
step_ffn_kernel(const __grid_constant__ StepMaps maps, const __grid_constant__ StepParams p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bars[2 * kSlots + 2 * kAccs + 3 * kQ];
  __shared__ Tile tq[kQ];
  __shared__ int g_expert[kMaxGroups], g_row0[kMaxGroups], g_rows[kMaxGroups];  // groups; expert -1: the shared one
  __shared__ int s_pos[kSmallDispatchMaxSlots];    // inv_perm
  __shared__ float s_weight[kSmallDispatchMaxSlots];  // topk_w
  __shared__ int word_sum[32];
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int abort_word;
  __shared__ volatile int rows_found;  // tiles whose rows have been found to be there; all there will ever be: INT_MAX
  volatile int* const abort_flag = &abort_word;
  const uint32_t raw_addr = smem_u32(smem_raw);
  const uint32_t base_addr = (raw_addr + 1023u) & ~1023u;
  uint8_t* const staging = smem_raw + (base_addr - raw_addr) + kSlots * kSlotBytes;
  const uint32_t bar_full = smem_u32(bars);
  const uint32_t bar_empty = bar_full + 8u * kSlots;
  const uint32_t bar_tfull = bar_empty + 8u * kSlots;
  const uint32_t bar_tempty = bar_tfull + 8u * kAccs;
  const uint32_t bar_tqfull = bar_tempty + 8u * kAccs;
  const uint32_t bar_tqempty = bar_tqfull + 8u * kQ;
  const uint32_t bar_stored = bar_tqempty + 8u * kQ;  // every epilogue warp has stored its part of the entry's tile
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned long long limit = p.wait_limit_ns;

  // ---- set-up
  if (threadIdx.x == 32 * kProducerWarp) {
    for (uint32_t s = 0; s < kSlots; ++s) {
      mbar_init(bar_full + 8u * s, 1);
      mbar_init(bar_empty + 8u * s, 1);
    }
    for (uint32_t a = 0; a < kAccs; ++a) {
      mbar_init(bar_tfull + 8u * a, 1);
      mbar_init(bar_tempty + 8u * a, kEpilogueWarps);
    }
    for (uint32_t q = 0; q < kQ; ++q) {
      mbar_init(bar_tqfull + 8u * q, 1);
      mbar_init(bar_tqempty + 8u * q, 2 + kEpilogueWarps + kFinishWarps);
      mbar_init(bar_stored + 8u * q, kEpilogueWarps);
    }
    abort_word = 0;
    rows_found = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == kMmaWarp) tmem_alloc(smem_u32(&tmem_slot), kTmemCols);
  // the maps, while the launch in front is still running
  if (warp == kRowWarp && lane < (int)(sizeof(StepMaps) / sizeof(CUtensorMap)))
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<const CUtensorMap*>(&maps) + lane) : "memory");
  pdl_wait();
  pdl_launch_dependents();
  int* const tile_ctr = p.ctr;
  int* const groups_ready = p.ctr + 1;
  int* const ready = p.ctr + 2;
  const int n_shared = p.Is > 0 ? 1 : 0;
  // the first tile's number is on its way while the list is built
  int taken = 0;
  if (warp == kProducerWarp && lane == 0) taken = atomicAdd(tile_ctr, 1);
  // ---- the groups: the shared expert, then the experts that have rows
  for (int i = threadIdx.x; i < p.T * p.k; i += kThreads) {
    s_pos[i] = __ldcg(p.inv_perm + i);
    s_weight[i] = __ldcg(p.topk_w + i);
  }
  const int n_words = (p.E + 31) >> 5;
  int e_mine[2], beg[2], cnt[2];  // at most 16 words of 32 experts on 15 warps
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int word = warp + i * kWarps, e = 32 * word + lane;
    e_mine[i] = e;
    beg[i] = cnt[i] = 0;
    if (word < n_words) {
      if (e < p.E) {
        beg[i] = __ldcg(p.offsets + e);
        cnt[i] = min(__ldcg(p.offsets + e + 1) - beg[i], p.T);  // (a token reaches an expert once)
      }
      const unsigned some = __ballot_sync(0xffffffffu, cnt[i] > 0);
      if (lane == 0) word_sum[word] = __popc(some);
    }
  }
  if (threadIdx.x == 0 && n_shared) {
    g_expert[0] = -1;
    g_row0[0] = 0;
    g_rows[0] = p.T;
  }
  __syncthreads();
  int n_groups;
  {
    int incl = lane < n_words ? word_sum[lane] : 0;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int n = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += n;
    }
    n_groups = n_shared + __shfl_sync(0xffffffffu, incl, 31);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int word = warp + i * kWarps;
      const unsigned some = __ballot_sync(0xffffffffu, cnt[i] > 0);
      const int before = word > 0 ? __shfl_sync(0xffffffffu, incl, min(word - 1, 31)) : 0;
      if (cnt[i] > 0) {
        const int at = n_shared + before + __popc(some & ((1u << lane) - 1u));
        g_expert[at] = e_mine[i];
        g_row0[at] = beg[i];
        g_rows[at] = cnt[i];
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_slot;
  const int n_ft1 = p.I / kGatedFeat, n_ft1_sh = p.Is / kGatedFeat, n_ft2 = (p.H + kDownFeat - 1) / kDownFeat;
  const int gated_tiles = n_ft1_sh + (n_groups - n_shared) * n_ft1, total_tiles = gated_tiles + n_groups * n_ft2;
  int* const down_done = ready + p.E + 1;
  const int all_tiles = total_tiles + n_ft2 * ((p.T + kCombineTokens - 1) / kCombineTokens);
  auto give_up = [&]() {
    abort_word = 1;
    atomicCAS(p.status, kStOk, kStTimeout);
  };

  if (warp == kProducerWarp) {
    // ================================================================= tiles and weights
    if (!p.inject_producer_stall) {
      RingCursor ring;
      uint32_t tcount = 0;
      bool ok = true, seen = true;  // seen: the next slot was seen to be free
      for (;;) {
        const int tile = __shfl_sync(0xffffffffu, taken, 0);
        Tile t{-1, 0, 0, 0};
        if (tile < n_ft1_sh) {
          t = {0, kGated, tile, 0};
        } else if (tile < gated_tiles) {
          const int g = (tile - n_ft1_sh) / n_ft1;
          t = {n_shared + g, kGated, tile - n_ft1_sh - g * n_ft1, 0};
        } else if (tile < total_tiles) {
          const int g = (tile - gated_tiles) / n_ft2;
          t = {g, kDown, tile - gated_tiles - g * n_ft2, 0};
        } else if (tile < all_tiles) {
          const int block = (tile - total_tiles) / n_ft2;
          t = {block, kCombine, tile - total_tiles - block * n_ft2, 0};
        }
        const uint32_t q = tcount % kQ;
        if (!mbar_wait_warp(bar_tqempty + 8u * q, ((tcount / kQ) & 1u) ^ 1u, abort_flag, limit)) { ok = false; break; }
        if (elect_one()) {
          tq[q] = t;
          mbar_arrive(bar_tqfull + 8u * q);
        }
        ++tcount;
        if (t.group < 0) break;
        if (t.kind == kCombine) {
          // Nothing to fetch; the next one is taken when this one is done, so that they spread over the CTAs, and none if there is
          // one for every CTA.
          if (all_tiles - total_tiles <= (int)gridDim.x) {
            taken = all_tiles;
            continue;
          }
          if (!mbar_wait_warp(bar_tqempty + 8u * q, ((tcount - 1) / kQ) & 1u, abort_flag, limit)) { ok = false; break; }
          taken = lane == 0 ? atomicAdd(tile_ctr, 1) : 0;
          continue;
        }
        const bool down = t.kind == kDown, sh = g_expert[t.group] < 0;
        const uint32_t n = (uint32_t)((g_rows[t.group] + 15) & ~15), bytes = (uint32_t)kWBoxBytes + n * 128u;
        const bool apart = n > (uint32_t)kSmallRows;
        const CUtensorMap* const mw = down ? (sh ? &maps.w2_sh : &maps.w2) : (sh ? &maps.w1_sh : &maps.w1);
        const int w_e = sh ? 0 : g_expert[t.group], K = down ? (sh ? p.Is : p.I) : p.H;
        const int num_kb = (K + kBlockK - 1) / kBlockK, f0 = t.ft * (down ? kDownFeat : kGatedFeat / 16);
        // The counter is read some k-blocks before the tile's last copy, so that its round trip hides behind those -- but not
        // while this down tile may still have to wait for its rows, so that no CTA holds a second one while others have none.
        const bool all_found = __shfl_sync(0xffffffffu, rows_found, 0) == 0x7fffffff;
        const int take_kb = down && !all_found ? num_kb : max(0, num_kb - kTakeAhead);
        for (int kb = 0, k0 = 0; kb < num_kb; ++kb, k0 += kBlockK) {
          if (kb == take_kb) taken = lane == 0 ? atomicAdd(tile_ctr, 1) : 0;
          if (!seen && !mbar_wait_warp(bar_empty + 8u * ring.stage, ring.phase ^ 1u, abort_flag, limit)) { ok = false; break; }
          const uint32_t full = bar_full + 8u * ring.stage, st = base_addr + ring.stage * (uint32_t)kSlotBytes;
          uint32_t full_x = 0;
          ring.advance(kSlots);
          if (apart) {
            if (!mbar_wait_warp(bar_empty + 8u * ring.stage, ring.phase ^ 1u, abort_flag, limit)) { ok = false; break; }
            full_x = bar_full + 8u * ring.stage;
            ring.advance(kSlots);
          }
          const bool next = mbar_test(bar_empty + 8u * ring.stage, ring.phase ^ 1u);  // the answer arrives behind the copy
          if (elect_one()) {
            mbar_expect_tx(full, bytes);  // the rows' bytes too, which may even be there already
            if (down) tma_load_3d(st, mw, full, k0, f0, w_e);
            else tma_load_5d(st, mw, full, k0, 0, 0, f0, w_e);
            if (apart) mbar_arrive(full_x);  // (the k-block completes on its first slot's barrier; this keeps the second's in step)
          }
          seen = __all_sync(0xffffffffu, next);
        }
        if (!ok) break;
        if (take_kb == num_kb) {
          unsigned long long t0 = 0;
          for (uint32_t polls = 0; !__all_sync(0xffffffffu, rows_found >= (int)tcount); ++polls) {
            __nanosleep(32);
            if ((polls & 255u) != 255u) continue;
            const unsigned long long now = global_ns();
            if (t0 == 0) t0 = now;
            if (!__all_sync(0xffffffffu, *abort_flag == 0 && now - t0 <= limit)) { ok = false; break; }
          }
          if (!ok) break;
          taken = lane == 0 ? atomicAdd(tile_ctr, 1) : 0;
        }
      }
      if (!ok && lane == 0) give_up();
    }
  } else if (warp == kRowWarp) {
    // ================================================================= rows
    if (!p.inject_producer_stall) {
      RingCursor ring;
      uint32_t tcount = 0;
      bool ok = true, all_there = false;
      for (;;) {
        const uint32_t q = tcount % kQ;
        if (!mbar_wait_warp(bar_tqfull + 8u * q, (tcount / kQ) & 1u, abort_flag, limit)) { ok = false; break; }
        const Tile t = tq[q];
        __syncwarp();
        ++tcount;
        if (t.group < 0) break;
        if (t.kind == kCombine) {
          if (lane == 0) mbar_arrive(bar_tqempty + 8u * q);
          continue;
        }
        const int expert = g_expert[t.group], rows = g_rows[t.group];
        const bool down = t.kind == kDown, sh = expert < 0;
        const uint32_t n = (uint32_t)((rows + 15) & ~15);
        const bool apart = n > (uint32_t)kSmallRows;
        const int row0 = g_row0[t.group];
        const CUtensorMap* const mx = down ? (sh ? &maps.a_sh : maps.a + ((n >> 4) - 1u)) : (sh ? &maps.x_sh : maps.x + ((n >> 4) - 1u));
        const int K = down ? (sh ? p.Is : p.I) : p.H, num_kb = (K + kBlockK - 1) / kBlockK;
        if (down && !all_there) {
          // the group's gated tiles are stored, or every group's are
          int n_ready = 0;
          if (!wait_count(ready + t.group, sh ? n_ft1_sh : n_ft1, groups_ready, n_ready, abort_flag, limit)) { ok = false; break; }
          all_there = __all_sync(0xffffffffu, n_ready == n_groups);
          fence_async_proxy();  // threads of other SMs stored the rows
          if (lane == 0) rows_found = all_there ? 0x7fffffff : (int)tcount;
        }
        for (int kb = 0, k0 = 0; kb < num_kb; ++kb, k0 += kBlockK) {
          const uint32_t full = bar_full + 8u * ring.stage;
          if (!mbar_wait_warp(bar_empty + 8u * ring.stage, ring.phase ^ 1u, abort_flag, limit)) { ok = false; break; }
          uint32_t st = base_addr + ring.stage * (uint32_t)kSlotBytes + (uint32_t)kWBoxBytes;
          ring.advance(kSlots);
          if (apart) {
            if (!mbar_wait_warp(bar_empty + 8u * ring.stage, ring.phase ^ 1u, abort_flag, limit)) { ok = false; break; }
            st = base_addr + ring.stage * (uint32_t)kSlotBytes;
            ring.advance(kSlots);
          }
          if (elect_one()) tma_load_2d(st, mx, full, k0, row0);
        }
        if (!ok) break;
        if (lane == 0) mbar_arrive(bar_tqempty + 8u * q);
      }
      if (!ok && lane == 0) give_up();
    }
  } else if (warp == kMmaWarp) {
    // ================================================================= MMA issuer
    RingCursor ring, acc;
    uint32_t tcount = 0;
    bool ok = true;
    const uint32_t desc_hi = (uint32_t)(umma_smem_desc(0) >> 32);
    const uint32_t lo_base = (uint32_t)umma_smem_desc(base_addr);
    for (;;) {
      const uint32_t q = tcount % kQ;
      if (!mbar_wait_warp(bar_tqfull + 8u * q, (tcount / kQ) & 1u, abort_flag, limit)) { ok = false; break; }
      const Tile t = tq[q];
      __syncwarp();
      if (elect_one()) mbar_arrive(bar_tqempty + 8u * q);
      ++tcount;
      if (t.group < 0) break;
      if (t.kind == kCombine) continue;
      const uint32_t n = (uint32_t)((g_rows[t.group] + 15) & ~15);
      const int K = t.kind == kDown ? (g_expert[t.group] < 0 ? p.Is : p.I) : p.H, num_kb = (K + kBlockK - 1) / kBlockK;
      if (!mbar_wait_warp(bar_tempty + 8u * acc.stage, acc.phase ^ 1u, abort_flag, limit)) { ok = false; break; }
      tc_fence_after();
      const uint32_t d = tmem_base + acc.stage * kAccCols;
      const bool apart = n > (uint32_t)kSmallRows;
      const uint32_t idesc = umma_idesc(128, n);
      // Up to four k-blocks that are there are issued in one go: behind a wait for rows a ring of them is, and a turn of this loop
      // takes longer than their MMAs.
      for (int kb = 0; kb < num_kb;) {
        if (!mbar_wait_warp(bar_full + 8u * ring.stage, ring.phase, abort_flag, limit)) { ok = false; break; }
        RingCursor at = ring;
        bool there[kBatch];
        there[0] = true;
#pragma unroll
        for (int i = 1; i < kBatch; ++i) {
          at.advance(kSlots);
          if (apart) at.advance(kSlots);
          there[i] = kb + i < num_kb && mbar_test(bar_full + 8u * at.stage, at.phase);
        }
        int m = 1;
#pragma unroll
        for (int i = 1; i < kBatch; ++i)
          if (m == i && __all_sync(0xffffffffu, there[i])) m = i + 1;
        tc_fence_after();
        const bool one = elect_one();
#pragma unroll 1
        for (int i = 0; i < m; ++i) {
          const uint32_t empty = bar_empty + 8u * ring.stage;
          const uint32_t lo_w = lo_base + ring.stage * ((uint32_t)kSlotBytes >> 4);
          uint32_t lo_x = lo_w + ((uint32_t)kWBoxBytes >> 4), empty_x = 0;
          ring.advance(kSlots);
          if (apart) {
            lo_x = lo_base + ring.stage * ((uint32_t)kSlotBytes >> 4);
            empty_x = bar_empty + 8u * ring.stage;
            ring.advance(kSlots);
          }
          if (one) {
#pragma unroll
            for (int kk = 0; kk < kBlockK / kUmmaK; ++kk) {
              const uint32_t adv = (uint32_t)((kk * kUmmaK * 2) >> 4);  // +32 bytes per MMA, in 16-byte units
              const uint32_t more = ((kb + i) | kk) != 0 ? 1u : 0u;
              umma_bf16_lo(d, lo_w + adv, lo_x + adv, desc_hi, idesc, more);
            }
            umma_commit(empty);
            if (apart) umma_commit(empty_x);
          }
        }
        kb += m;
      }
      if (!ok) break;
      if (elect_one()) umma_commit(bar_tfull + 8u * acc.stage);
      acc.advance(kAccs);
    }
    if (!ok && lane == 0) give_up();
  } else if (warp < kEpilogueWarps) {
    // ================================================================= epilogue (warps 0-7)
    // Fragments and stmatrix as in gemm_stream.cu and gemm_pair.cu; warps w and w + 4 share a lane group and take alternate
    // chunks of 16 tokens.  Down tile: 32 features a warp; gated: 16 (lanes 0-15 gate, 16-31 up).
    RingCursor acc;
    uint32_t tcount = 0;
    bool ok = true;
    const int lg = warp & 3;
    const int c_first = 16 * (warp >> 2), c_step = 32;
    // staging: tokens of 64 bytes (gated 32), the 16-byte pieces XOR-swizzled by pairs (fours) of tokens
    uint8_t* const stg = staging + warp * kStagingBytes;
    auto piece = [](bool down, int tok, int i) {
      return down ? tok * 64 + ((i ^ ((tok >> 1) & 3)) << 4) : tok * 32 + ((i ^ ((tok >> 2) & 1)) << 4);
    };
    const int st_tok = (lane & 7) + 8 * (lane >> 4), st_piece = (lane >> 3) & 1;  // stmatrix: this lane's row of 8 features
    for (;;) {
      const uint32_t q = tcount % kQ;
      if (!mbar_wait_warp(bar_tqfull + 8u * q, (tcount / kQ) & 1u, abort_flag, limit)) { ok = false; break; }
      const Tile t = tq[q];
      ++tcount;
      if (t.group < 0) break;
      if (t.kind == kCombine) {
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(bar_stored + 8u * q);
          mbar_arrive(bar_tqempty + 8u * q);
        }
        continue;
      }
      const bool down = t.kind == kDown;
      const int expert = g_expert[t.group], row0 = g_row0[t.group], rows = g_rows[t.group];
      const bool sh = expert < 0;
      const int n_feat = down ? p.H : sh ? p.Is : p.I;
      __nv_bfloat16* const out = down ? (sh ? p.y_sh : p.y) : (sh ? p.act_sh : p.act);
      const int f0 = t.ft * (down ? kDownFeat : kGatedFeat) + lg * (down ? 32 : 16);  // this warp's first feature
      if (!mbar_wait_warp(bar_tfull + 8u * acc.stage, acc.phase, abort_flag, limit)) { ok = false; break; }
      tc_fence_after();
      const uint32_t d = tmem_base + acc.stage * kAccCols + ((uint32_t)(lg * 32) << 16);
#pragma unroll 1
      for (int c = c_first; c < rows; c += c_step) {
        uint32_t r[2][8];  // [lanes 0-15, 16-31][fragments of 16 tokens]
#pragma unroll
        for (int k = 0; k < 2; ++k) tmem_ld_frag(d + ((uint32_t)(16 * k) << 16) + (uint32_t)c, r[k]);
        tmem_ld_wait();
        uint64_t v[2][4];  // pairs of neighbouring tokens
#pragma unroll
        for (int k = 0; k < 2; ++k)
#pragma unroll
          for (int i = 0; i < 4; ++i) v[k][i] = f32x2(__uint_as_float(r[k][2 * i]), __uint_as_float(r[k][2 * i + 1]));
        uint32_t o[2][4];
        if (down) {
#pragma unroll
          for (int k = 0; k < 2; ++k)
#pragma unroll
            for (int i = 0; i < 4; ++i) o[k][i] = pack_bf16(v[k][i]);
          stmatrix_trans(smem_u32(stg) + (uint32_t)piece(true, st_tok, st_piece), o[0]);
          stmatrix_trans(smem_u32(stg) + (uint32_t)piece(true, st_tok, st_piece + 2), o[1]);
          __syncwarp();
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int tok = (lane >> 2) + 8 * i, f = f0 + 8 * (lane & 3);
            const uint4 u = *reinterpret_cast<const uint4*>(stg + piece(true, tok, lane & 3));
            if (c + tok < rows && f < n_feat) *reinterpret_cast<uint4*>(out + (size_t)(row0 + c + tok) * n_feat + f) = u;
          }
        } else {
#pragma unroll
          for (int i = 0; i < 4; ++i) o[0][i] = pack_bf16(silu_mul2(v[0][i], v[1][i]));
          stmatrix_trans(smem_u32(stg) + (uint32_t)piece(false, st_tok, st_piece), o[0]);
          __syncwarp();
          const int tok = lane >> 1, f = f0 + 8 * (lane & 1);
          const uint4 u = *reinterpret_cast<const uint4*>(stg + piece(false, tok, lane & 1));
          if (c + tok < rows && f < n_feat) *reinterpret_cast<uint4*>(out + (size_t)(row0 + c + tok) * n_feat + f) = u;
        }
        __syncwarp();  // read: the staging may be written again
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(bar_tempty + 8u * acc.stage);
        mbar_arrive(bar_stored + 8u * q);
        mbar_arrive(bar_tqempty + 8u * q);
      }
      acc.advance(kAccs);
    }
    if (!ok && lane == 0) give_up();
  } else {
    // ================================================================= finishing warps (10-13)
    // What follows a tile that is stored: the first of these warps tells whoever waits for it, beside the epilogue, because the
    // fence takes a microsecond.  And the combine tiles.
    uint32_t tcount = 0;
    bool ok = true;
    const int f = warp - kFinishWarp0;
    for (;;) {
      const uint32_t q = tcount % kQ, par = (tcount / kQ) & 1u;
      if (!mbar_wait_warp(bar_tqfull + 8u * q, par, abort_flag, limit)) { ok = false; break; }
      const Tile t = tq[q];
      if (t.group < 0) break;
      if (!mbar_wait_warp(bar_stored + 8u * q, par, abort_flag, limit)) { ok = false; break; }
      ++tcount;
      if (t.kind == kCombine) {
        // when every group's rows have these columns: half a warp to a token, a thread to eight columns
        int unused;
        if (!wait_count(down_done + t.ft, n_groups, nullptr, unused, abort_flag, limit)) { ok = false; break; }
        const int v = t.ft * (kDownFeat / 8) + (lane & 15), t0 = t.group * kCombineTokens + 2 * f + (lane >> 4);
        if (8 * v < p.H && t0 < p.T) {
          if (p.k <= 2) combine_columns<2>(p, s_pos, s_weight, v, t0);
          else if (p.k <= 4) combine_columns<4>(p, s_pos, s_weight, v, t0);
          else combine_columns<8>(p, s_pos, s_weight, v, t0);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_tqempty + 8u * q);
        continue;
      }
      if (lane == 0) {
        mbar_arrive(bar_tqempty + 8u * q);
        if (f == 0) {
          __threadfence();
          if (t.kind == kDown) {
            atomicAdd(down_done + t.ft, 1);
          } else if (atomicAdd(ready + t.group, 1) == (g_expert[t.group] < 0 ? n_ft1_sh : n_ft1) - 1) {
            __threadfence();
            atomicAdd(groups_ready, 1);
          }
        }
      }
      __syncwarp();
    }
    if (!ok && lane == 0) give_up();
  }

  // ---- teardown
  tc_fence_before();
  __syncthreads();
  if (abort_word) {
    // give copies still in flight time to land in this CTA's shared memory before it is released
    for (int i = 0; i < 64; ++i) __nanosleep(1000);
    __syncthreads();
  }
  if (warp == kMmaWarp) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kTmemCols);
  }
}

}  // namespace

// The maps of a context's steps, encoded again where an operand's address or shape is another.
struct StepPlan {
  StepMaps maps;
  StepFfn had;
  bool valid = false;
  int64_t encoded = 0;
};

StepPlan* step_plan_create() {
  StepPlan* p = new (std::nothrow) StepPlan();
  if (p != nullptr) memset(&p->maps, 0, sizeof p->maps);
  return p;
}
void step_plan_destroy(StepPlan* plan) { delete plan; }
int64_t step_plan_encoded(const StepPlan* plan) { return plan->encoded; }

int step_ffn_counters(int E, int H) { return 2 + (E + 1) + (H + kDownFeat - 1) / kDownFeat; }

static bool encode_step_maps(StepPlan& plan, const StepFfn& f) {
  const StepFfn had = plan.had;
  const bool kept = plan.valid;
  plan.valid = false;  // a failure half way leaves no valid maps
  const bool shared = f.Is > 0;
  auto gated = [&](CUtensorMap* m, const void* w, uint64_t K, uint64_t n_feat, uint64_t groups) {
    ++plan.encoded;
    const uint64_t dims[5] = {K, 16, 2, n_feat / 16, groups};
    const uint64_t row = K * sizeof(__nv_bfloat16), str[4] = {row, n_feat * row, 16 * row, 2 * n_feat * row};
    const uint32_t box[5] = {(uint32_t)kBlockK, 16u, 2u, (uint32_t)kGatedFeat / 16u, 1u};
    return encode_map(m, w, 5, dims, str, box);
  };
  auto down = [&](CUtensorMap* m, const void* w, uint64_t K, uint64_t n_feat, uint64_t groups) {
    ++plan.encoded;
    const uint64_t dims[3] = {K, n_feat, groups};
    const uint64_t str[2] = {K * sizeof(__nv_bfloat16), n_feat * K * sizeof(__nv_bfloat16)};
    const uint32_t box[3] = {(uint32_t)kBlockK, (uint32_t)kDownFeat, 1u};
    return encode_map(m, w, 3, dims, str, box);
  };
  auto rows = [&](CUtensorMap* m, const void* a, uint64_t K, uint64_t n_rows, int box_rows) {
    ++plan.encoded;
    const uint64_t dims[2] = {K, n_rows};
    const uint64_t str[1] = {K * sizeof(__nv_bfloat16)};
    const uint32_t box[2] = {(uint32_t)kBlockK, (uint32_t)box_rows};
    return encode_map(m, a, 2, dims, str, box);
  };
  // (the layer's sizes and the workspace are a context's own and never change)
  if (!kept || had.w1 != f.w1) if (!gated(&plan.maps.w1, f.w1, f.H, f.I, f.E)) return false;
  if (!kept || had.w2 != f.w2) if (!down(&plan.maps.w2, f.w2, f.I, f.H, f.E)) return false;
  if (!kept)
    for (int i = 0; i < kRowMaps; ++i)
      if (!rows(&plan.maps.x[i], f.x, f.H, (uint64_t)f.rows_cap, 16 * (i + 1)) ||
          !rows(&plan.maps.a[i], f.act, f.I, (uint64_t)f.rows_cap, 16 * (i + 1))) return false;
  if (shared) {
    if (!kept || had.w1_sh != f.w1_sh) if (!gated(&plan.maps.w1_sh, f.w1_sh, f.H, f.Is, 1)) return false;
    if (!kept || had.w2_sh != f.w2_sh) if (!down(&plan.maps.w2_sh, f.w2_sh, f.Is, f.H, 1)) return false;
    const int box = (f.T + 15) & ~15;
    if (!kept || had.T != f.T || had.x_sh != f.x_sh) {
      if (!rows(&plan.maps.x_sh, f.x_sh, f.H, (uint64_t)f.T, box)) return false;
      if (!rows(&plan.maps.a_sh, f.act_sh, f.Is, (uint64_t)f.T, box)) return false;
    }
  }
  plan.had = f;
  plan.valid = true;
  return true;
}

cudaError_t launch_step_ffn(const StepFfn& f, StepPlan* plan, int max_ctas, cudaStream_t stream, int* n_launches) {
  if (plan == nullptr || f.T < 1 || f.T > kStepMaxTokens || max_ctas < 1) return cudaErrorInvalidValue;
  if (!encode_step_maps(*plan, f)) return cudaErrorInvalidValue;
  StepParams prm;
  memset(&prm, 0, sizeof prm);
  prm.offsets = f.offsets;
  prm.E = f.E;
  prm.T = f.T;
  prm.k = f.k;
  prm.H = f.H;
  prm.I = f.I;
  prm.Is = f.Is;
  prm.act = static_cast<__nv_bfloat16*>(f.act);
  prm.act_sh = static_cast<__nv_bfloat16*>(f.act_sh);
  prm.y = static_cast<__nv_bfloat16*>(f.y);
  prm.y_sh = static_cast<__nv_bfloat16*>(f.y_sh);
  prm.out = static_cast<__nv_bfloat16*>(f.out);
  prm.inv_perm = f.inv_perm;
  prm.topk_w = f.topk_w;
  prm.ctr = f.counters;
  prm.status = f.status;
  prm.wait_limit_ns = f.wait_limit_ns ? f.wait_limit_ns : kWaitLimitNs;
  prm.inject_producer_stall = f.debug_stall ? 1 : 0;
  constexpr size_t smem = 1024 + (size_t)kSlots * kSlotBytes + kEpilogueWarps * kStagingBytes;
  static_assert(smem + 16 * 1024 <= kSmemBudget, "and the kernel's static shared memory");
  const int64_t groups = (int64_t)f.T * f.k < f.E ? (int64_t)f.T * f.k : f.E;
  const int64_t per_group = f.I / kGatedFeat + (f.H + kDownFeat - 1) / kDownFeat;
  const int64_t tiles = groups * per_group + (f.Is > 0 ? f.Is / kGatedFeat + (f.H + kDownFeat - 1) / kDownFeat : 0);
  const int grid = (int)(tiles < max_ctas ? tiles : max_ctas);
  cudaError_t err = ensure_dynamic_smem(step_ffn_kernel, smem);
  if (err != cudaSuccess) return err;
  err = launch_pdl(true, step_ffn_kernel, dim3(grid), dim3(kThreads), smem, stream, plan->maps, prm);
  if (err == cudaSuccess && n_launches) *n_launches += 1;
  return err;
}

}  // namespace moe
