// What the two swap-AB kernels share -- gemm_stream.cu (one CTA per tile) and gemm_pair.cu (two): weight rows fill the MMA M
// dimension, an expert's tokens sit in N.  The tile list and its order, launch parameters, tensor maps and their plan.
#pragma once
#include <cstring>

#include "kernels.h"
#include "tc_common.cuh"

namespace moe {
namespace tc {

constexpr int kSizeClasses = 256;  // classes of expert size the tile list is ordered by
constexpr int kMaxTileRows = 256;  // largest MMA N
constexpr int kXMaps = 16;         // token-row boxes, one for each multiple of 16 rows of a tile
constexpr int kQ = 4;              // entries of a CTA's tile queue

// Waves' worth of tiles, at the list's end, that are handed out dynamically: a fifth of them, between two and six.  Over
// tens of waves the CTAs drift apart by more than two tiles (V3-shaped decode, 28 and 49 waves: 2089 us with six, 2111 with
// two, 64 tokens; FP8 weights, 128 tokens 1313 and 1332; level on a GPU that runs these steps in 2146 and 1355 us); a launch
// of five waves, or one whose tiles share weights through L2 while the CTAs are in step, wants two (8192-token Qwen3-shaped
// prefill 732 us; 742 with all but the first wave dynamic).
constexpr int kMinDynWaves = 2, kMaxDynWaves = 6, kDynWavesOneIn = 5;

struct StreamParams {
  const int32_t* offsets;  // [E+1] (already advanced to the first expert of the launch) or nullptr
  int32_t fixed_rows;
  int32_t E;               // experts covered by this launch
  int32_t e_base;          // index of the launch's first expert in the weight tensor
  int32_t n_feat;          // output features (I for the gated pass, H for the down pass)
  int32_t ft0, n_ft, n_ft2;  // feature tiles of this launch: the first, and how many (n_ft2: of the dense group)
  int32_t K;
  __nv_bfloat16* out;      // [rows, n_feat]
  int32_t ring_slots;
  int* status;
  int32_t inject_producer_stall;  // failure-detection test hook: the TMA producer issues nothing
  unsigned long long wait_limit_ns;
  // optional dense group (shared expert) computed by the same launch; rows2 == 0: none
  int32_t rows2;
  int32_t n_feat2;
  int32_t K2;
  __nv_bfloat16* out2;
  // FP8 variant: the accumulator is scaled by row_scale[row] * w_scale[weight row]
  const float* row_scale;
  const float* row_scale2;
  const float* w_scale;
  const float* w_scale2;
  // The launch's tile counter and the count of CTAs (pairs) that take no more tiles (two words in device memory, zero
  // before the first launch that uses them; the last one puts them back to zero).
  int* tile_ctr;
  int* done_ctr;
  int32_t all_dynamic;  // every tile comes from the counter (a pass that may be launched again to go on)
  // preemption at tile granularity (both null: off)
  const int* yield_req;
  int* stopped;
  // The expert offsets are older than every kernel that may still be running (and the weights always are): the tile list
  // is built and weight boxes are fetched before this kernel waits for the previous one, which only the token rows (and
  // the FP8 row scales) depend on.
  int32_t early_setup;
  int32_t sort_tiles;  // 0: every group has at most one tile of the smallest size, so their order does not matter
  // row gather (the gated pass of bf16 layers, gemm_stream.cu): row r is gather_src[perm[r] / top_k], of the dense group gather_src2[r]
  const __nv_bfloat16* gather_src;
  const __nv_bfloat16* gather_src2;
  const int32_t* perm;
  int32_t top_k;
};

// Token rows in boxes of 16, 32, ..., 256 rows; the dense group's in the two sizes it has, its equal chunks and its last one.
// (With sixteen of those, too, a launch's parameters are 4.6 KB instead of 2.8.)
struct StreamMaps {
  CUtensorMap x[kXMaps], x2[2];
};

// A tile as the producer hands it to the other roles: one entry of the CTA's queue.
struct __align__(16) STile {
  int e;  // expert; kDenseTile: a tile of the dense group; kNoTile: no more tiles
  int row0, rows, ft;
};
constexpr int kDenseTile = -1, kNoTile = -2;

// An expert's (or the dense group's) rows in ceil(cnt / 256) chunks of equal size, rounded up to 16.
__device__ __forceinline__ void chunking(int cnt, int& tiles, int& chunk) {
  tiles = (cnt + kMaxTileRows - 1) / kMaxTileRows;
  chunk = tiles > 0 ? (((cnt + tiles - 1) / tiles) + 15) & ~15 : 0;
}

// Size class of an expert, 0 = largest: exact up to 256 rows in steps of 16, then eight classes per octave.
__device__ __forceinline__ int size_class(int cnt) {
  const unsigned u = (unsigned)(cnt + 15) >> 4;
  if (u < 16u) return kSizeClasses - 1 - (int)u;
  const int msb = 31 - __clz(u);  // 4..27
  return kSizeClasses - 1 - (16 + (msb - 4) * 8 + (int)((u >> (msb - 3)) & 7u));
}

// tile -> (expert, first row, valid rows, feature tile), by a whole warp.  The dense group's tiles come first (chunk major),
// then the experts' in the order `order` (largest first): prefix[i] = chunks of the experts at positions < i.
__device__ __forceinline__ STile decode_tile(int tile, int dense_tiles, const StreamParams& p, const int* prefix,
                                             const int* order, const int* beg, const int* cnts) {
  STile t;
  int tiles, chunk;
  if (tile < dense_tiles) {
    const int rt = tile / p.n_ft2;
    chunking(p.rows2, tiles, chunk);
    t.e = kDenseTile;
    t.ft = p.ft0 + tile - rt * p.n_ft2;
    t.row0 = rt * chunk;
    t.rows = min(chunk, p.rows2 - t.row0);
    return t;
  }
  tile -= dense_tiles;
  const int rt = tile / p.n_ft;
  // largest position in [0,E) with prefix[position] <= rt: 32 places at a time
  int lo = 0;
  for (int span = p.E; span > 1;) {
    const int step = (span + 31) >> 5, at = lo + (int)(threadIdx.x & 31) * step;
    const unsigned below = __ballot_sync(0xffffffffu, at < lo + span && prefix[at] <= rt);
    const int skip = (__popc(below) - 1) * step;
    lo += skip;
    span = min(step, span - skip);
  }
  const int e = order[lo], cnt = cnts[e];
  chunking(cnt, tiles, chunk);
  const int mt = rt - prefix[lo];
  t.e = e;
  t.ft = p.ft0 + tile - rt * p.n_ft;
  t.row0 = beg[e] + mt * chunk;
  t.rows = min(chunk, cnt - mt * chunk);
  return t;
}

// The map of a tile's token rows, n of them with the padding to 16.
__device__ __forceinline__ const CUtensorMap* rows_map(const StreamMaps& maps, const StreamParams& p, const STile& t,
                                                       uint32_t n) {
  return t.e != kDenseTile ? maps.x + ((n >> 4) - 1u) : maps.x2 + (t.row0 + t.rows == p.rows2 ? 1 : 0);
}

// First tiles of a launch that are dealt statically, in waves of `takers` (CTAs, or pairs of them).
__device__ __forceinline__ int static_waves(int total_tiles, int takers) {
  const int waves = total_tiles / takers;
  return max(1, waves - min(kMaxDynWaves, max(kMinDynWaves, waves / kDynWavesOneIn)));
}

// The tile list, built by all THREADS threads of a CTA (ends without a barrier behind its last writes).
template <int THREADS>
__device__ __forceinline__ void build_tile_list(const StreamParams& p, int* prefix, int* order, int* beg, int* cnts,
                                                int* class_pos, int* chunk_sum) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // The tile list: experts by size class, largest first, ascending index within a class.  A stable counting sort --
  // counts per class by shared-memory atomics, a scan over the classes, then one warp places 32 experts at a time and
  // ranks equals by __match_any_sync -- because every CTA of every launch builds the list before its first copy.
  // (24 tokens over 512 experts 384 us a step; 403 when each expert was ranked against all others, a shared-memory read per
  // pair; 37 over 128 184.0 and 186.2, 64 over 256 2152 and 2161.)
  // Where the order does not matter the prefix is taken as the counts come in: one barrier instead of three, none up to 32
  // experts.
  auto fetch = [&](int e, int& b, int& c) {
    b = p.offsets ? p.offsets[e] : 0;
    c = p.offsets ? p.offsets[e + 1] - b : p.fixed_rows;
    if (c < 0) c = 0;
    beg[e] = b;
    cnts[e] = c;
  };
  if (p.sort_tiles) {
    for (int c = threadIdx.x; c < kSizeClasses; c += THREADS) class_pos[c] = 0;
    __syncthreads();
    for (int e = threadIdx.x; e < p.E; e += THREADS) {
      int b, c;
      fetch(e, b, c);
      atomicAdd(&class_pos[size_class(c)], 1);
    }
    __syncthreads();
    if (warp == 0) {
      constexpr int kPer = kSizeClasses / 32;  // consecutive classes per lane
      int v[kPer], sum = 0;
#pragma unroll
      for (int i = 0; i < kPer; ++i) {
        v[i] = sum;
        sum += class_pos[lane * kPer + i];
      }
      int incl = sum;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const int n = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += n;
      }
#pragma unroll
      for (int i = 0; i < kPer; ++i) class_pos[lane * kPer + i] = incl - sum + v[i];
      __syncwarp();
      const unsigned lt_mask = (1u << lane) - 1u;
      for (int b = 0; b < p.E; b += 32) {
        const int e = b + lane;
        const int key = e < p.E ? size_class(cnts[e]) : kSizeClasses;
        const unsigned peers = __match_any_sync(0xffffffffu, key);
        int pos = 0;
        if (e < p.E) pos = class_pos[key] + __popc(peers & lt_mask);
        __syncwarp();
        if (e < p.E) {
          order[pos] = e;
          if ((peers & lt_mask) == 0u) class_pos[key] += __popc(peers);
        }
        __syncwarp();
      }
    }
    __syncthreads();
  }
  // prefix[i]: row chunks of the experts at positions < i; warp w scans the 32-expert groups w, w + warps, ...
  for (int g = warp; 32 * g < p.E; g += THREADS / 32) {
    const int i = 32 * g + lane;
    int begin, cnt = 0;
    if (p.sort_tiles) {
      if (i < p.E) cnt = cnts[order[i]];
    } else if (i < p.E) {
      fetch(i, begin, cnt);
      order[i] = i;
    }
    const int tiles = (cnt + kMaxTileRows - 1) / kMaxTileRows;
    int incl = tiles;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int n = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += n;
    }
    if (i < p.E) prefix[i] = incl - tiles;
    if (lane == 31) (p.E <= 32 ? prefix[p.E] : chunk_sum[g]) = incl;
  }
  if (p.E <= 32) return;
  __syncthreads();
  for (int g = warp; 32 * g < p.E; g += THREADS / 32) {
    int before = lane < g ? chunk_sum[lane] : 0;  // at most 32 groups
    before = __reduce_add_sync(0xffffffffu, before);
    const int i = 32 * g + lane;
    if (i < p.E) prefix[i] += before;
    if (32 * g + 32 >= p.E && lane == 0) prefix[p.E] = before + chunk_sum[g];
  }
}

// ---------------------------------------------------------------------------------------------- host side
// What an operand's tensor maps depend on.
struct OperandKey {
  const void* W = nullptr;
  const void* A = nullptr;
  int64_t rows = 0;
  int32_t groups = 0, n_feat = 0, K = 0;
  bool gated = false, fp8 = false;
  bool same_weights(const OperandKey& o) const {
    return W == o.W && groups == o.groups && n_feat == o.n_feat && K == o.K && gated == o.gated && fp8 == o.fp8;
  }
  bool same_rows(const OperandKey& o) const { return A == o.A && rows == o.rows && K == o.K && fp8 == o.fp8; }
};

}  // namespace tc

// (of one kernel: the boxes of the two-CTA kernel are not those of the other)
struct StreamPlan {
  tc::OperandKey key, key2;  // the routed problem's and the dense group's
  CUtensorMap mw, mw2;
  tc::StreamMaps xm;
  int64_t encoded = 0;  // maps encoded so far
};

namespace tc {

// Whether the kernels take the problem at all.
inline bool swap_ab_supports(const GemmProblem& p, const GemmDenseGroup* dense) {
  if (dense != nullptr && (dense->K % 8 != 0 || dense->n_feat % 8 != 0)) return false;
  if (!encoder_ready()) return false;
  if (p.K % 8 != 0 || p.n_feat % 8 != 0 || p.E < 1 || p.E > 1024) return false;
  if (p.rows_bound > 0x7fffffffLL / 2) return false;
  return !(p.fp8 && (p.row_scale == nullptr || p.w_scale == nullptr || p.K % 16 != 0 || p.n_feat % 64 != 0 ||
                     (dense != nullptr && (dense->row_scale == nullptr || dense->w_scale == nullptr || dense->K % 16 != 0 ||
                                           dense->n_feat % 64 != 0))));
}

// Brings the plan's maps up to date with the launch's operands.  pair: two CTAs share a tile, each with half of its weight
// rows and half of its token rows.
//   weights  one box holds the 256 weight rows of a k-block (pair: 128).  Gated pass: [groups][2][n_feat][K] with a box of
//            128 rows x 2 (gate rows and the matching up rows); pair: 16 gate rows, the 16 matching up rows, and so on, four
//            times, so that a warp's 32 accumulator lanes hold both.  Down pass: [groups][n_feat][K], 256 or 128 rows.
//   rows     the routed rows' maps span the buffer's capacity, not this call's rows, so that a call with another T finds
//            them as they are: a tile's last box may then read rows that an earlier, larger step left there; their columns
//            of the accumulator are never stored.  The dense group has two box sizes at most (its equal chunks and the last
//            one).
inline cudaError_t update_plan(StreamPlan& plan, const GemmProblem& p, const GemmDenseGroup* dense, int groups, bool pair) {
  const bool fp8 = p.fp8;
  const uint64_t esz = fp8 ? 1 : 2;                                // bytes per operand element
  const uint32_t box_k = (uint32_t)(fp8 ? 2 * kBlockK : kBlockK);  // 128 bytes of K per k-block row
  auto encode_w = [&](CUtensorMap* m, const OperandKey& k) {
    ++plan.encoded;
    const uint64_t K = (uint64_t)k.K, n_feat = (uint64_t)k.n_feat, n_groups = (uint64_t)k.groups;
    if (k.gated && pair) {
      const uint64_t dims[5] = {K, 16, 2, n_feat / 16, n_groups};
      const uint64_t str[4] = {K * esz, n_feat * K * esz, 16 * K * esz, 2 * n_feat * K * esz};
      const uint32_t box[5] = {box_k, 16u, 2u, (uint32_t)kWBoxRows / 32u, 1u};
      return encode_map(m, k.W, 5, dims, str, box, fp8);
    }
    if (k.gated) {
      const uint64_t dims[4] = {K, n_feat, 2, n_groups};
      const uint64_t str[3] = {K * esz, n_feat * K * esz, 2 * n_feat * K * esz};
      const uint32_t box[4] = {box_k, (uint32_t)kWBoxRows, 2u, 1u};
      return encode_map(m, k.W, 4, dims, str, box, fp8);
    }
    const uint64_t dims[3] = {K, n_feat, n_groups};
    const uint64_t str[2] = {K * esz, n_feat * K * esz};
    const uint32_t box[3] = {box_k, (pair ? 1u : 2u) * kWBoxRows, 1u};
    return encode_map(m, k.W, 3, dims, str, box, fp8);
  };
  auto encode_x = [&](CUtensorMap* m, const OperandKey& k, int b) {  // the box of a tile of 16 (b + 1) rows
    ++plan.encoded;
    const uint64_t dims[2] = {(uint64_t)k.K, (uint64_t)k.rows};
    const uint64_t str[1] = {(uint64_t)k.K * esz};
    const uint32_t box[2] = {box_k, (pair ? 8u : 16u) * (uint32_t)(b + 1)};
    return encode_map(m, k.A, 2, dims, str, box, fp8);
  };
  {
    const OperandKey k{p.W, p.A, p.rows_cap, groups, p.n_feat, p.K, p.gated, fp8}, had = plan.key;
    plan.key = OperandKey{};  // a failure half way leaves no valid key
    if (!had.same_weights(k) && !encode_w(&plan.mw, k)) return cudaErrorInvalidValue;
    if (!had.same_rows(k))
      for (int b = 0; b < kXMaps; ++b)
        if (!encode_x(&plan.xm.x[b], k, b)) return cudaErrorInvalidValue;
    plan.key = k;
  }
  if (dense != nullptr) {
    const OperandKey k{dense->W, dense->A, dense->rows, 1, dense->n_feat, dense->K, p.gated, fp8}, had = plan.key2;
    plan.key2 = OperandKey{};
    if (!had.same_weights(k) && !encode_w(&plan.mw2, k)) return cudaErrorInvalidValue;
    if (!had.same_rows(k)) {
      const int chunks = (dense->rows + kMaxTileRows - 1) / kMaxTileRows;
      const int chunk = ((dense->rows + chunks - 1) / chunks + 15) & ~15;
      const int last = (dense->rows - (chunks - 1) * chunk + 15) & ~15;
      if (!encode_x(&plan.xm.x2[0], k, chunk / 16 - 1) || !encode_x(&plan.xm.x2[1], k, last / 16 - 1)) return cudaErrorInvalidValue;
    }
    plan.key2 = k;
  }
  return cudaSuccess;
}

// Fills the parameters (without the ring's size) and counts the tiles there can be; false: a bad range.
inline bool fill_params(StreamParams& prm, int64_t& tiles, const GemmProblem& p, const GemmDenseGroup* dense, int e_begin,
                        int e_end, int* status) {
  prm.offsets = p.offsets ? p.offsets + e_begin : nullptr;
  prm.fixed_rows = p.fixed_rows;
  prm.E = e_end - e_begin;
  prm.e_base = e_begin;
  prm.n_feat = p.n_feat;
  prm.K = p.K;
  prm.out = static_cast<__nv_bfloat16*>(p.out);
  prm.status = status;
  prm.inject_producer_stall = p.debug_stall ? 1 : 0;
  prm.wait_limit_ns = p.wait_limit_ns ? p.wait_limit_ns : kWaitLimitNs;
  prm.rows2 = dense ? dense->rows : 0;
  prm.n_feat2 = dense ? dense->n_feat : 8;
  prm.K2 = dense ? dense->K : 8;
  prm.out2 = dense ? static_cast<__nv_bfloat16*>(dense->out) : nullptr;
  prm.row_scale = p.row_scale;
  prm.w_scale = p.w_scale;
  prm.row_scale2 = dense ? dense->row_scale : nullptr;
  prm.w_scale2 = dense ? dense->w_scale : nullptr;
  prm.tile_ctr = p.tile_counters;
  prm.done_ctr = p.tile_counters + 1;
  prm.all_dynamic = p.resumable ? 1 : 0;
  const bool preemptible = p.yield_req != nullptr && p.stopped != nullptr;
  prm.sort_tiles = (p.max_group_rows > 0 && p.max_group_rows <= 16) ? 0 : 1;
  prm.early_setup = (p.offsets_settled && !preemptible) ? 1 : 0;
  prm.yield_req = preemptible ? p.yield_req : nullptr;
  prm.stopped = preemptible ? p.stopped : nullptr;

  const int feat_per_tile = p.gated ? 128 : 256;
  const int f_end = p.f_end < 0 ? p.n_feat : p.f_end;
  const bool part = p.f_begin != 0 || f_end != p.n_feat;
  if (p.f_begin < 0 || p.f_begin % 256 != 0 || f_end > p.n_feat || p.f_begin >= f_end ||
      (f_end % feat_per_tile != 0 && f_end != p.n_feat) || (part && dense != nullptr && dense->n_feat != p.n_feat))
    return false;
  const int64_t n_ft = (f_end + feat_per_tile - 1) / feat_per_tile - p.f_begin / feat_per_tile;
  prm.ft0 = p.f_begin / feat_per_tile;
  prm.n_ft = (int)n_ft;
  prm.n_ft2 = dense == nullptr ? 1 : part ? (int)n_ft : (dense->n_feat + feat_per_tile - 1) / feat_per_tile;
  const int64_t row_tiles = p.rows_bound / kMaxTileRows + (prm.E < p.rows_bound ? prm.E : p.rows_bound);
  tiles = row_tiles * n_ft;
  if (dense != nullptr)
    tiles += (int64_t)((dense->rows + kMaxTileRows - 1) / kMaxTileRows) * prm.n_ft2;
  return true;
}

}  // namespace tc
}  // namespace moe
