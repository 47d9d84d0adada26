// Stages a6-a8, two-CTA variant of the grouped expert GEMM (sm_100a): swap-AB on the 5th-generation tensor cores, a tile
// multiplied by a pair of SMs (tcgen05 cta_group::2).
//
//   tile       (expert, token chunk, feature tile) as in gemm_stream.cu: 256 weight rows fill the MMA M dimension, 128 in
//              each CTA; an expert's rows in equal chunks of at most 256, rounded up to 16, are N.
//   operands   a k-block (64 K-elements = 128-byte rows, 128-byte swizzle) is, in each CTA, one TMA copy of its own 128
//              weight rows (16 KB) and one of HALF of the tile's token rows; the tensor cores of both SMs read the two halves.
//              Gated pass: a warp's 32 accumulator lanes are 16 gate rows and the 16 matching up rows (one 5-D box), so
//              SwiGLU needs no second accumulator.
//   TMEM       two accumulators of N <= 256 columns: the epilogue of a tile always overlaps the next tile's MMAs.
//   epilogue   in each CTA for its own 128 weight rows, by fragments and stmatrix as in gemm_stream.cu.
//   schedule   as in gemm_stream.cu, a pair taking the place of a CTA: the leader's producer takes the tiles and publishes
//              them to both CTAs.
//
// Per k-block and SM that is 32 KB into shared memory and 32 KB of operand reads for 128 x 256 outputs, against 32 and 48 in
// gemm_stream.cu (which can overlap no epilogue of a tile of more than 128 tokens) and 48 and 48 in gemm_tc.cu.
//
// Warp roles (320 threads): warps 0-7 epilogue (two per TMEM lane group), warp 8 TMA producer, warp 9 TMEM owner and, in
// the leader, MMA issuer.
// Every mbarrier wait is bounded: on expiry the kernel records a timeout in the status word, raises the abort flag of both
// CTAs, lets copies in flight land, frees its TMEM and returns.
#include <cuda.h>
#include <cuda_bf16.h>

#include "swap_ab.cuh"

namespace moe {
namespace {

using namespace tc;

constexpr int kEpilogueWarps = 8;
constexpr int kProducerWarp = kEpilogueWarps;
constexpr int kMmaWarp = kEpilogueWarps + 1;
constexpr int kThreads = 32 * (kEpilogueWarps + 2);
constexpr int kWBytes = kWBoxBytes;                       // this CTA's 128 weight rows of a k-block
constexpr int kStageBytes = kWBytes + kMaxTileRows * 64;  // ... and up to 128 token rows
constexpr int kMaxStages = 6;
constexpr uint32_t kAccCols = 256, kTmemCols = 512;
constexpr int kStagingBytes = 1024;  // epilogue, per warp: 16 tokens x 32 features or (gated) 32 tokens x 16 features
// arrivals that free a queue entry: the issuer, the other CTA's producer, the epilogue warps of both
constexpr int kQueueReaders = 2 + 2 * kEpilogueWarps;

// ---------------------------------------------------------------------------------- PTX wrappers (pairs)
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Address of the same place in the shared memory of CTA `rank` of the cluster
__device__ __forceinline__ uint32_t at_rank(uint32_t addr, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(rank));
  return a;
}
// Arrives on a barrier of either CTA.  Releases to this CTA only, which does not wait for the thread's global stores; what it
// hands back (a queue entry read, an accumulator read) is no memory that the other CTA could see half written.
__device__ __forceinline__ void arrive_remote(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void store_remote(uint32_t addr, int v) {
  asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
// ... asynchronously, counted as 16 bytes by the other CTA's barrier (an arrival that releases this thread's stores to it
// instead waits for everything the thread has in flight: 2000 clocks a tile)
__device__ __forceinline__ void store_remote(uint32_t addr, const STile& t, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr),
               "r"(t.e), "r"(t.row0), "r"(t.rows), "r"(t.ft), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
// Tiled loads of a pair: into this CTA's shared memory, completing on a barrier of either CTA
__device__ __forceinline__ void pair_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1)
      : "memory");
}
__device__ __forceinline__ void pair_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}
__device__ __forceinline__ void pair_load_5d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2,
                                             int c3, int c4) {
  asm volatile(
      "cp.async.bulk.tensor.5d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6, %7}], [%2];"
      ::"r"(dst), "l"(map), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4)
      : "memory");
}
template <bool FP8>
__device__ __forceinline__ void pair_mma(uint32_t tmem_d, uint32_t a_lo, uint32_t b_lo, uint32_t desc_hi, uint32_t idesc,
                                         uint32_t accumulate) {
  if (FP8)
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "mov.b64 da, {%1, %3};\n\t"
        "mov.b64 db, {%2, %3};\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], da, db, %4, p;\n\t}"
        ::"r"(tmem_d), "r"(a_lo), "r"(b_lo), "r"(desc_hi), "r"(idesc), "r"(accumulate)
        : "memory");
  else
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "mov.b64 da, {%1, %3};\n\t"
        "mov.b64 db, {%2, %3};\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], da, db, %4, p;\n\t}"
        ::"r"(tmem_d), "r"(a_lo), "r"(b_lo), "r"(desc_hi), "r"(idesc), "r"(accumulate)
        : "memory");
}
// One arrival on the barrier at this offset in both CTAs when every MMA issued so far by this thread has completed
__device__ __forceinline__ void pair_commit(uint32_t bar) {
  const uint16_t both = 3;
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar), "h"(both)
      : "memory");
}
__device__ __forceinline__ void pair_tmem_alloc(uint32_t dst_smem, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(cols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void pair_tmem_dealloc(uint32_t taddr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}

// ------------------------------------------------------------------------------------- the kernel
// grid 2 x pairs: CTAs 2 i and 2 i + 1 are pair i
template <bool GATED, bool FP8>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
grouped_gemm_pair_kernel(const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_w2,
                         const __grid_constant__ StreamMaps xmaps, const __grid_constant__ StreamParams p) {
  constexpr int kbk = FP8 ? 2 * kBlockK : kBlockK;  // K elements per k-block
  extern __shared__ uint8_t smem_raw[];
  // carve (the same in both CTAs: barriers and operands are addressed across the pair by their offset):
  //   stages: weight rows | token rows | epilogue staging | full[S] empty[S] tfull[2] tempty[2] tqfull[kQ] tqempty[kQ] | tq[kQ]
  //   | tmem slot | abort | prefix[E+1] | order[E] | beg[E] | cnts[E] | classes | chunk sums
  const uint32_t raw_addr = smem_u32(smem_raw);
  const uint32_t base_addr = (raw_addr + 1023u) & ~1023u;
  uint8_t* base = smem_raw + (base_addr - raw_addr);
  const uint32_t n_stages = (uint32_t)p.ring_slots;
  uint8_t* const staging = base + (size_t)n_stages * kStageBytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(staging + kEpilogueWarps * kStagingBytes);
  const uint32_t bar_full = smem_u32(bars);
  const uint32_t bar_empty = bar_full + 8u * kMaxStages;
  const uint32_t bar_tfull = bar_empty + 8u * kMaxStages;
  const uint32_t bar_tempty = bar_tfull + 16u;
  const uint32_t bar_tqfull = bar_tempty + 16u;
  const uint32_t bar_tqempty = bar_tqfull + 8u * kQ;
  static_assert((2 * kMaxStages + 4 + 2 * kQ) % 2 == 0, "the queue's entries are 16-byte aligned");
  STile* tq = reinterpret_cast<STile*>(bars + 2 * kMaxStages + 4 + 2 * kQ);  // tile queue
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tq + kQ);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int* prefix = reinterpret_cast<int*>(tmem_slot + 2);
  int* order = prefix + (p.E + 1);
  int* beg = order + p.E;
  int* cnts = beg + p.E;
  int* class_pos = cnts + p.E;
  int* chunk_sum = class_pos + kSizeClasses;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const bool leader = rank == 0;
  constexpr int kFeatPerTile = GATED ? 128 : 256;  // of the pair; half of them in each CTA
  const int num_kb1 = (p.K + kbk - 1) / kbk, num_kb2 = (p.K2 + kbk - 1) / kbk;
  const int dense_tiles = p.rows2 > 0 ? ((p.rows2 + kMaxTileRows - 1) / kMaxTileRows) * p.n_ft2 : 0;
  const unsigned long long limit = p.wait_limit_ns;

  // ---- set-up: barriers and TMEM, then the tile list
  if (threadIdx.x == 32 * kProducerWarp) {
    for (int s = 0; s < kMaxStages; ++s) {
      mbar_init(bar_full + 8u * s, 1);   // leader: its producer's announcement (and both CTAs' bytes)
      mbar_init(bar_empty + 8u * s, 1);  // the issuer's commit
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(bar_tfull + 8u * a, 1);
      mbar_init(bar_tempty + 8u * a, 2 * kEpilogueWarps);  // leader
    }
    for (int q = 0; q < kQ; ++q) {
      mbar_init(bar_tqfull + 8u * q, 1);               // leader: its producer; the other CTA: its own, for the 16 bytes to come
      mbar_init(bar_tqempty + 8u * q, kQueueReaders);  // leader
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == kMmaWarp) pair_tmem_alloc(smem_u32(tmem_slot), kTmemCols);
  pdl_wait();
  pdl_launch_dependents();
  if (leader) build_tile_list<kThreads>(p, prefix, order, beg, cnts, class_pos, chunk_sum);  // it hands the tiles to both
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // both CTAs' barriers exist
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const int total_tiles = leader ? dense_tiles + prefix[p.E] * p.n_ft : 0;
  auto give_up = [&]() {
    *abort_flag = 1;
    store_remote(at_rank(smem_u32(const_cast<int*>(abort_flag)), rank ^ 1u), 1);
    atomicCAS(p.status, kStOk, kStTimeout);
  };

  if (warp == kProducerWarp) {
    // ================================================================= TMA producer (one in each CTA)
    if (!p.inject_producer_stall) {
      RingCursor ring;
      uint32_t tcount = 0;
      bool ok = true;
      const uint32_t full_at_leader = at_rank(bar_full, 0);
      const uint32_t tq_at_peer = at_rank(smem_u32(tq), 1), tqfull_at_peer = at_rank(bar_tqfull, 1);
      const uint32_t tqempty_at_leader = at_rank(bar_tqempty, 0);
      const int pairs = (int)gridDim.x / 2, pair = (int)blockIdx.x / 2;
      const int w_static = static_waves(total_tiles, pairs);
      int sw = 0;
      auto next_tile = [&]() -> int {  // leader; lane 0's counts
        if (sw < w_static) {
          const int w = sw++;
          return w * pairs + ((w & 1) ? pairs - 1 - pair : pair);
        }
        return lane == 0 ? w_static * pairs + atomicAdd(p.tile_ctr, 1) : 0;
      };
      // Leader: finds the tile's place and hands it to both CTAs' roles.
      auto publish = [&](int tile, STile& t) -> bool {
        const uint32_t q = tcount % kQ, par = ((tcount / kQ) & 1u) ^ 1u;
        ++tcount;
        if (tile < total_tiles) t = decode_tile(tile, dense_tiles, p, prefix, order, beg, cnts);
        else t.e = kNoTile;
        if (!mbar_wait_warp(bar_tqempty + 8u * q, par, abort_flag, limit)) return false;
        if (elect_one()) {
          tq[q] = t;
          mbar_arrive(bar_tqfull + 8u * q);
          store_remote(tq_at_peer + (uint32_t)sizeof(STile) * q, t, tqfull_at_peer + 8u * q);
        }
        return true;
      };
      STile next{kNoTile, 0, 0, 0};
      if (leader) ok = publish(__shfl_sync(0xffffffffu, next_tile(), 0), next);
      else if (elect_one())
        for (int q = 0; q < kQ; ++q) mbar_expect_tx(bar_tqfull + 8u * q, (uint32_t)sizeof(STile));
      bool ready = false;  // the stage to fill next was seen to be free
      while (ok) {
        STile t = next;
        if (!leader) {
          const uint32_t q = tcount % kQ;
          if (!mbar_wait_warp(bar_tqfull + 8u * q, (tcount / kQ) & 1u, abort_flag, limit)) { ok = false; break; }
          ++tcount;
          t = tq[q];
          __syncwarp();
          if (elect_one()) {
            mbar_expect_tx(bar_tqfull + 8u * q, (uint32_t)sizeof(STile));  // the entry's next use
            arrive_remote(tqempty_at_leader + 8u * q);
          }
        }
        if (t.e == kNoTile) break;
        const bool dense = t.e == kDenseTile;
        const uint32_t n = (uint32_t)((t.rows + 15) & ~15);
        const CUtensorMap* mw = dense ? &map_w2 : &map_w;
        const CUtensorMap* mx = rows_map(xmaps, p, t, n);  // the box of n / 2 rows
        const int w_e = dense ? 0 : p.e_base + t.e;
        const int w_row0 = t.ft * kFeatPerTile + (int)rank * (kFeatPerTile / 2);
        const int x_row0 = t.row0 + (int)(rank * (n >> 1));
        const int num_kb = dense ? num_kb2 : num_kb1;
        const int fetch_kb = num_kb > 4 ? num_kb - 4 : 0;
        int taken = 0;
        for (int kb = 0, k0 = 0; kb < num_kb; ++kb, k0 += kbk) {
          // The counter is read a few k-blocks before the tile's last copy, so that its round trip hides behind those, and the
          // next tile is published before the last: the other CTA's producer has it when it gets there.
          if (leader && kb == fetch_kb) taken = next_tile();
          if (leader && kb == num_kb - 1 && !publish(__shfl_sync(0xffffffffu, taken, 0), next)) { ok = false; break; }
          if (!ready && !mbar_wait_warp(bar_empty + 8u * ring.stage, ring.phase ^ 1u, abort_flag, limit)) { ok = false; break; }
          const uint32_t full = full_at_leader + 8u * ring.stage, full_here = bar_full + 8u * ring.stage;
          const uint32_t st = base_addr + ring.stage * (uint32_t)kStageBytes;
          ring.advance(n_stages);
          const bool seen = mbar_test(bar_empty + 8u * ring.stage, ring.phase ^ 1u);
          if (elect_one()) {
            if (leader) mbar_expect_tx(full_here, 2u * kWBytes + n * 128u);  // both CTAs' bytes
            if (GATED) pair_load_5d(st, mw, full, k0, 0, 0, w_row0 >> 4, w_e);
            else pair_load_3d(st, mw, full, k0, w_row0, w_e);
            pair_load_2d(st + kWBytes, mx, full, k0, x_row0);
          }
          ready = __all_sync(0xffffffffu, seen);
        }
      }
      // the last stages are free again: no commit of the issuer's is on its way to this CTA's barriers when it leaves
      for (uint32_t i = 0; i < n_stages && ok; ++i) {
        if (!mbar_wait_warp(bar_empty + 8u * ring.stage, ring.phase ^ 1u, abort_flag, limit)) ok = false;
        ring.advance(n_stages);
      }
      if (!ok && lane == 0) give_up();
    }
    if (lane == 0 && leader) {
      // this pair takes no more tiles; the last one that says so puts the counters back for the next launch that uses them
      __threadfence();
      if (atomicAdd(p.done_ctr, 1) == (int)gridDim.x / 2 - 1) {
        *p.done_ctr = 0;
        *p.tile_ctr = 0;
      }
    }
  } else if (warp == kMmaWarp) {
    // ================================================================= MMA issuer (leader)
    if (leader) {
      RingCursor ring;
      uint32_t tcount = 0, acc = 0, acc_phase = 0;
      bool ok = true, ready = false;  // ready: the stage to multiply next was seen to be full
      const uint32_t desc_hi = (uint32_t)(umma_smem_desc(0) >> 32);
      const uint32_t lo_base = (uint32_t)umma_smem_desc(base_addr);
      constexpr uint32_t lo_stage = (uint32_t)kStageBytes >> 4, lo_x = (uint32_t)kWBytes >> 4;
      for (;;) {
        const uint32_t q = tcount % kQ;
        if (!mbar_wait_warp(bar_tqfull + 8u * q, (tcount / kQ) & 1u, abort_flag, limit)) { ok = false; break; }
        const STile t = tq[q];
        __syncwarp();
        if (elect_one()) mbar_arrive(bar_tqempty + 8u * q);
        ++tcount;
        if (t.e == kNoTile) break;
        const uint32_t n = (uint32_t)((t.rows + 15) & ~15);
        if (!mbar_wait_warp(bar_tempty + 8u * acc, acc_phase ^ 1u, abort_flag, limit)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d = tmem_base + acc * kAccCols;
        const uint32_t idesc = FP8 ? umma_idesc_e4m3(256, n) : umma_idesc(256, n);
        const int num_kb = t.e == kDenseTile ? num_kb2 : num_kb1;
        for (int kb = 0; kb < num_kb; ++kb) {
          if (!ready && !mbar_wait_warp(bar_full + 8u * ring.stage, ring.phase, abort_flag, limit)) { ok = false; break; }
          tc_fence_after();
          const uint32_t lo_w = lo_base + ring.stage * lo_stage, empty = bar_empty + 8u * ring.stage;
          ring.advance(n_stages);
          const bool seen = mbar_test(bar_full + 8u * ring.stage, ring.phase);
          if (elect_one()) {
#pragma unroll
            for (int kk = 0; kk < kBlockK / kUmmaK; ++kk) {
              const uint32_t adv = (uint32_t)((kk * kUmmaK * 2) >> 4);  // +32 bytes per MMA, in 16-byte units
              pair_mma<FP8>(d, lo_w + adv, lo_w + lo_x + adv, desc_hi, idesc, (kb | kk) != 0 ? 1u : 0u);
            }
            pair_commit(empty);  // the stage is free in both CTAs once these MMAs have read it
          }
          ready = __all_sync(0xffffffffu, seen);
        }
        if (!ok) break;
        if (elect_one()) pair_commit(bar_tfull + 8u * acc);
        acc ^= 1u;
        if (acc == 0) acc_phase ^= 1u;
      }
      if (!ok && lane == 0) give_up();
    }
  } else {
    // ================================================================= epilogue (warps 0-7)
    // Fragments and stmatrix as in gemm_stream.cu; warps w and w + 4 share a lane group and take alternate chunks of 32
    // tokens.  Down pass: 32 features x 2 x 16 tokens; gated: 16 features (lanes 0-15 gate, 16-31 up) x 32 tokens.
    uint32_t tcount = 0, acc = 0, acc_phase = 0;
    bool ok = true;
    const int lg = warp & 3;
    const int c_first = 32 * (warp >> 2), c_step = 64;
    const uint32_t tqempty_at_leader = at_rank(bar_tqempty, 0), tempty_at_leader = at_rank(bar_tempty, 0);
    const int f_in_tile = (int)rank * (kFeatPerTile / 2) + lg * (GATED ? 16 : 32);  // this warp's first feature
    // staging, 16-byte pieces XOR-swizzled: tokens of 64 bytes (by pairs of tokens) or, gated, of 32 (by fours)
    uint8_t* const stg = staging + warp * kStagingBytes;
    auto piece = [](int tok, int i) {
      return GATED ? tok * 32 + ((i ^ ((tok >> 2) & 1)) << 4) : tok * 64 + ((i ^ ((tok >> 1) & 3)) << 4);
    };
    const int st_tok = (lane & 7) + 8 * (lane >> 4), st_piece = (lane >> 3) & 1;  // stmatrix: this lane's row of 8 features
    const uint32_t st0 = smem_u32(stg) + (uint32_t)piece(st_tok, st_piece);
    const uint32_t st1 = smem_u32(stg) + (uint32_t)(GATED ? piece(st_tok + 16, st_piece) : piece(st_tok, st_piece + 2));
    const int ld_tok = GATED ? lane >> 1 : lane >> 2, ld_piece = GATED ? lane & 1 : lane & 3;  // what this lane stores
    const int fr_row = lane >> 2, fr_col = 2 * (lane & 3);                                     // its feature and token
    for (;;) {
      const uint32_t q = tcount % kQ;
      if (!mbar_wait_warp(bar_tqfull + 8u * q, (tcount / kQ) & 1u, abort_flag, limit)) { ok = false; break; }
      const STile t = tq[q];
      __syncwarp();
      if (lane == 0) arrive_remote(tqempty_at_leader + 8u * q);
      ++tcount;
      if (t.e == kNoTile) break;
      const bool dense = t.e == kDenseTile;
      __nv_bfloat16* const out = dense ? p.out2 : p.out;
      const int n_feat = dense ? p.n_feat2 : p.n_feat;
      const int f0 = t.ft * kFeatPerTile + f_in_tile;
      // FP8: the scales of this thread's four weight rows, and of its tokens in the next chunk
      float ws[4], rs[8];
      const float* rsp = nullptr;
      auto fetch_scales = [&](int c) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int tok = c + fr_col + (i & 1) + 8 * (i >> 1);
          rs[i] = tok < t.rows ? __ldg(rsp + tok) : 0.f;
        }
      };
      if (FP8) {
        rsp = (dense ? p.row_scale2 : p.row_scale) + t.row0;
        const float* const wsp = dense ? p.w_scale2 : p.w_scale + (size_t)(p.e_base + t.e) * (GATED ? 2 : 1) * n_feat;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int f = f0 + fr_row + 8 * (GATED ? i & 1 : i);
          ws[i] = f < n_feat ? __ldg(wsp + (GATED && i >= 2 ? n_feat + f : f)) : 0.f;
        }
        fetch_scales(c_first);
      }
      if (!mbar_wait_warp(bar_tfull + 8u * acc, acc_phase, abort_flag, limit)) { ok = false; break; }
      tc_fence_after();
      const uint32_t d = tmem_base + acc * kAccCols + ((uint32_t)(lg * 32) << 16);
      auto release_acc = [&]() {  // hand the accumulator back to the MMA issuer
        tc_fence_before();
        __syncwarp();
        if (lane == 0) arrive_remote(tempty_at_leader + 8u * acc);
      };
      // stages 16 tokens x 32 features (gated: 32 x 16) and stores them
      auto put = [&](const uint32_t (&q0)[4], const uint32_t (&q1)[4], int c) {
        stmatrix_trans(st0, q0);
        stmatrix_trans(st1, q1);
        __syncwarp();
        constexpr int kTokStep = GATED ? 16 : 8;
        uint4 v[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) v[i] = *reinterpret_cast<const uint4*>(stg + piece(ld_tok + kTokStep * i, ld_piece));
        __syncwarp();  // read: the staging may be written again
        const int f = f0 + 8 * ld_piece;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int tok = c + ld_tok + kTokStep * i;
          if (tok < t.rows && f < n_feat) *reinterpret_cast<uint4*>(out + (size_t)(t.row0 + tok) * n_feat + f) = v[i];
        }
      };
      // the loads of the next chunk are in flight while this one is converted and stored
      uint32_t next[2][2][8];  // [16 tokens][lanes 0-15, 16-31][fragments]
      auto load = [&](int c) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int k = 0; k < 2; ++k) tmem_ld_frag(d + ((uint32_t)(16 * k) << 16) + (uint32_t)(c + 16 * h), next[h][k]);
      };
      if (c_first < t.rows) load(c_first);
      else release_acc();
      for (int c = c_first; c < t.rows; c += c_step) {
        uint64_t v[2][2][4];  // pairs of neighbouring tokens
        tmem_ld_wait();
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int k = 0; k < 2; ++k)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              v[h][k][i] = f32x2(__uint_as_float(next[h][k][2 * i]), __uint_as_float(next[h][k][2 * i + 1]));
              if (FP8) {
                const float w = ws[2 * k + (i & 1)];
                v[h][k][i] = mul2(v[h][k][i], mul2(f32x2(rs[4 * h + 2 * (i >> 1)], rs[4 * h + 2 * (i >> 1) + 1]), f32x2(w, w)));
              }
            }
        if (c + c_step < t.rows) {
          load(c + c_step);
          if (FP8) fetch_scales(c + c_step);
        } else {
          release_acc();  // read completely
        }
        uint32_t o[2][4];
        if (GATED) {
#pragma unroll
          for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int i = 0; i < 4; ++i) o[h][i] = pack_bf16(silu_mul2(v[h][0][i], v[h][1][i]));
          put(o[0], o[1], c);
        } else {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
              for (int i = 0; i < 4; ++i) o[k][i] = pack_bf16(v[h][k][i]);
            put(o[0], o[1], c + 16 * h);
          }
        }
      }
      acc ^= 1u;
      if (acc == 0) acc_phase ^= 1u;
    }
    if (!ok && lane == 0) give_up();
  }

  // ---- teardown
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    // give copies still in flight time to land in the CTAs' shared memory before it is released
    for (int i = 0; i < 64; ++i) __nanosleep(1000);
  }
  cluster_sync();  // nothing of the other CTA's is on its way to this one's barriers
  if (warp == kMmaWarp) {
    __syncwarp();
    tc_fence_after();
    pair_tmem_dealloc(tmem_base, kTmemCols);
  }
}

}  // namespace

cudaError_t launch_gemm_pair(const GemmProblem& p, const GemmDenseGroup* dense, int max_ctas, int* status,
                             cudaStream_t stream, int* n_launches) {
  if (dense != nullptr && dense->rows <= 0) dense = nullptr;
  if (p.rows_bound <= 0 && dense == nullptr) return cudaSuccess;
  if (p.rows_bound <= 0) return cudaErrorInvalidValue;  // a dense group never comes without its routed pass
  if (!swap_ab_supports(p, dense) || max_ctas < 2 || p.resumable || p.gather_src != nullptr || p.n_feat % 16 != 0 ||
      (dense != nullptr && dense->n_feat % 16 != 0))
    return cudaErrorNotSupported;
  const int groups = p.offsets ? p.E : 1;
  const int e_begin = p.offsets ? p.e_begin : 0;
  const int e_end = (p.offsets && p.e_end >= 0) ? p.e_end : groups;
  if (e_begin < 0 || e_end > groups || e_begin >= e_end) return cudaErrorInvalidValue;
  if (p.plan == nullptr || p.tile_counters == nullptr) return cudaErrorInvalidValue;
  StreamPlan& plan = *p.plan;
  cudaError_t err = update_plan(plan, p, dense, groups, true);
  if (err != cudaSuccess) return err;
  StreamParams prm;
  int64_t tiles;
  if (!fill_params(prm, tiles, p, dense, e_begin, e_end, status)) return cudaErrorInvalidValue;

  const size_t tail = kEpilogueWarps * kStagingBytes + (2 * kMaxStages + 4 + 2 * kQ) * sizeof(uint64_t) + kQ * sizeof(STile) +
                      2 * sizeof(uint32_t) + (4 * (size_t)(prm.E + 1) + kSizeClasses + 32) * sizeof(int);
  int stages = (kSmemBudget - 1024 - (int)tail) / kStageBytes;
  if (stages > kMaxStages) stages = kMaxStages;
  if (stages < 2) return cudaErrorNotSupported;
  prm.ring_slots = stages;
  const size_t smem = 1024 + (size_t)stages * kStageBytes + tail;
  const int64_t most = max_ctas / 2;
  const int pairs = (int)(tiles < most ? (tiles < 1 ? 1 : tiles) : most);
  auto launch = [&](auto kern) -> cudaError_t {
    cudaError_t e = ensure_dynamic_smem(kern, smem);
    if (e != cudaSuccess) return e;
    return launch_pdl(false, kern, dim3(2 * pairs), dim3(kThreads), smem, stream, plan.mw, plan.mw2,
                      plan.xm, prm);
  };
  if (p.fp8) err = p.gated ? launch(grouped_gemm_pair_kernel<true, true>) : launch(grouped_gemm_pair_kernel<false, true>);
  else err = p.gated ? launch(grouped_gemm_pair_kernel<true, false>) : launch(grouped_gemm_pair_kernel<false, false>);
  if (err == cudaSuccess && n_launches) *n_launches += 1;
  return err;
}

}  // namespace moe
