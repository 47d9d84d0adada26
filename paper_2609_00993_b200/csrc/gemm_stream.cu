// Stages a6-a8, weight-streaming variant of the grouped expert GEMM (sm_100a): swap-AB on the 5th-generation
// tensor cores.  128 weight rows fill the MMA M dimension, the expert's tokens sit in N, and N follows the expert:
//
//   tile       (expert, token chunk, feature tile).  An expert's rows are cut into ceil(rows / 256) equal chunks
//              (rounded up to 16), so an expert of up to 256 rows is ONE tile per feature tile and its weights
//              enter an SM once; the MMA N is the chunk's row count rounded up to 16 (16..256).
//   operands   a k-block (64 K-elements = 128-byte rows, 128-byte swizzle) is two 128-row weight boxes (32 KB,
//              gated: gate rows + the matching up rows; one TMA copy through a 4-D map) and exactly N token rows
//              (one TMA copy through the map whose box has N rows: 16 maps, one per multiple of 16).  What bounds
//              this regime is the bytes an SM ingests, so nothing is fetched that is not multiplied.
//   ring       k-blocks live in a byte ring of 2 KB slots with FIFO allocation (a k-block takes 16 slots for its
//              weights and N/16 for its token rows, two pieces that need not be adjacent), so a tile of few
//              tokens keeps more k-blocks in flight than a tile of many; up to 8 k-blocks in flight, each with
//              a full/empty mbarrier pair.  Producer and MMA issuer derive the same slot positions from the
//              same tile sequence.
//   TMEM       512 columns = two halves.  A tile of N <= 128 takes one half (its two accumulators side by side)
//              and alternates halves, so its epilogue overlaps the next tile's MMAs; a tile of N > 128 takes both.
//   epilogue   tcgen05.ld of 8 x 8 fragments -> (scale) -> SwiGLU -> bf16 -> stmatrix, which transposes (TMEM lanes are
//              features, columns tokens), into a per-warp staging tile -> 16-byte stores.
//   schedule   the tile list is ordered by expert size, largest first.  Its first waves are dealt statically (CTAs
//              in step share weights and rows through L2), the last waves' worth of tiles -- the smallest -- are
//              handed out by an atomic counter to whichever CTA is free; the producer publishes the tiles it takes
//              in a four-entry queue that the MMA issuer and the epilogue warps follow.
//   set-up     with the launch overlap, the tile list is built and weight boxes are requested before the kernel
//              waits for the previous kernel of the stream; only the token rows and the stores wait for it.
//
// Warp roles (320 threads): warps 0-7 epilogue (two per TMEM lane group), warp 8 TMA producer, warp 9 MMA issuer
// and TMEM owner.
// The row-gather instantiation (gated pass, bf16; rules.h says when) adds warps 10 and 11, which fetch the token rows of a k-block out
// of the unpermuted x by 16-byte cp.async copies, in TMA's swizzled layout, once the producer has made room for them; TMA then carries the
// weights only.  (TMA's own gather takes 58 clocks for four rows of 128 bytes, three times what the k-block's MMAs take; two warps,
// because with 14 in the CTA the epilogue's registers no longer fit.)
// Every mbarrier wait is bounded: on expiry the kernel records a timeout in the status word, raises a CTA-wide
// abort flag, lets copies in flight land, frees its TMEM and returns.
// The same kernel serves E4M3 operands (kind::f8f6f4, 128 K-elements per k-block, accumulator scaled by the
// row's and the weight row's scale in the epilogue).
#include <cuda.h>
#include <cuda_bf16.h>

#include <cstdlib>
#include <new>

#include "swap_ab.cuh"

namespace moe {
namespace {

using namespace tc;

constexpr int kEpilogueWarps = 8;  // two per TMEM lane group, taking alternate 16-token chunks
constexpr int kProducerWarp = kEpilogueWarps;
constexpr int kMmaWarp = kEpilogueWarps + 1;
constexpr int kThreads = 32 * (kEpilogueWarps + 2);
constexpr int kGatherWarp0 = kEpilogueWarps + 2, kGatherWarps = 2;
constexpr int kThreadsGather = 32 * (kGatherWarp0 + kGatherWarps);
constexpr int kSlotBytes = 2048;                        // ring granularity: 16 token rows of one k-block
constexpr int kWSlots = 2 * kWBoxBytes / kSlotBytes;    // 16 slots: the two weight boxes
constexpr int kNB = 8;                                  // k-blocks in flight at most (barrier pairs)
constexpr uint32_t kTmemCols = 512;
constexpr int kStagingBytes = 16 * 64;  // epilogue, per warp: 16 tokens x 32 features
#ifdef MOE_STREAM_PROF
// Debug build only: per-CTA role timings of the last launches (8 words per CTA, accumulated).
__device__ unsigned long long g_stream_prof[8 * 256];
__device__ unsigned long long g_stream_ts[8 * 256];  // global-timer stamps of the last launch, 8 per CTA
#define PROF_T0() const long long prof_t0 = clock64()
#define PROF_ADD(var) var += clock64() - prof_t0
#define PROF_STAMP(slot) g_stream_ts[8 * blockIdx.x + (slot)] = global_ns()
#else
#define PROF_T0()
#define PROF_ADD(var)
#define PROF_STAMP(slot)
#endif

template <bool GATED, bool FP8, bool GATHER>
__global__ void __launch_bounds__(GATHER ? kThreadsGather : kThreads, 1)
grouped_gemm_stream_kernel(const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_w2,
                           const __grid_constant__ StreamMaps xmaps, const __grid_constant__ StreamParams p) {
  static_assert(!GATHER || (GATED && !FP8), "rows are gathered for the gated pass of bf16 layers only");
  constexpr int kbk = FP8 ? 2 * kBlockK : kBlockK;  // K elements per k-block
  constexpr int kCtaThreads = GATHER ? kThreadsGather : kThreads;
  extern __shared__ uint8_t smem_raw[];
  // carve: ring (ring_slots x 2 KB) | epilogue staging | full[kNB] empty[kNB] tfull[2] tempty[2] tqfull[kQ] tqempty[kQ] (go[kNB])
  //        | tq[kQ] | tmem slot | abort | stopped | sizes[kNB] | prefix[E+1] | order[E] | beg[E] | cnts[E] | classes | chunk sums
  const uint32_t raw_addr = smem_u32(smem_raw);
  const uint32_t base_addr = (raw_addr + 1023u) & ~1023u;
  uint8_t* base = smem_raw + (base_addr - raw_addr);
  uint8_t* const staging = base + (size_t)p.ring_slots * kSlotBytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(staging + kEpilogueWarps * kStagingBytes);
  const uint32_t bar_full = smem_u32(bars);
  const uint32_t bar_empty = bar_full + 8u * kNB;
  const uint32_t bar_tfull = bar_empty + 8u * kNB;
  const uint32_t bar_tempty = bar_tfull + 16u;
  const uint32_t bar_tqfull = bar_tempty + 16u;         // the tile queue: an entry has been published
  const uint32_t bar_tqempty = bar_tqfull + 8u * kQ;    // ... and read by the issuer and every epilogue warp
  const uint32_t bar_go = bar_tqempty + 8u * kQ;        // row gather: there is room for the k-block's rows
  constexpr int kBars = 2 * kNB + 4 + 2 * kQ + (GATHER ? kNB : 0);
  static_assert(kBars % 2 == 0, "the queue's entries are 16-byte aligned");
  STile* tq = reinterpret_cast<STile*>(bars + kBars);  // tile queue
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tq + kQ);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* stopped_here = reinterpret_cast<volatile int*>(tmem_slot + 2);  // the producer stopped on request
  int* sizes = reinterpret_cast<int*>(tmem_slot + 3);  // slots held by the k-blocks in flight (producer only)
  int* prefix = sizes + kNB;
  int* order = prefix + (p.E + 1);
  int* beg = order + p.E;
  int* cnts = beg + p.E;
  int* class_pos = cnts + p.E;               // [kSizeClasses]
  int* chunk_sum = class_pos + kSizeClasses;  // [32]

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  [[maybe_unused]] const int unit = (int)blockIdx.x;
  if (threadIdx.x == 0) PROF_STAMP(0);
  constexpr int kFeatPerTile = GATED ? 128 : 256;
  const int num_kb1 = (p.K + kbk - 1) / kbk, num_kb2 = (p.K2 + kbk - 1) / kbk;
  const int dense_tiles = p.rows2 > 0 ? ((p.rows2 + kMaxTileRows - 1) / kMaxTileRows) * p.n_ft2 : 0;
  const unsigned long long limit = p.wait_limit_ns;

  // ---- set-up: barriers and TMEM (before the previous kernel of the stream is known to be complete), then the
  // tile list (experts ordered by size, largest first)
  if (threadIdx.x == 32 * kProducerWarp) {
    for (int s = 0; s < kNB; ++s) {
      mbar_init(bar_full + 8u * s, GATHER ? 1 + 32 * kGatherWarps : 1);  // (a gathering thread's copies are an arrival of it)
      mbar_init(bar_empty + 8u * s, 1);
      if (GATHER) mbar_init(bar_go + 8u * s, 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(bar_tfull + 8u * a, 1);
      mbar_init(bar_tempty + 8u * a, kEpilogueWarps);
    }
    for (int q = 0; q < kQ; ++q) {
      mbar_init(bar_tqfull + 8u * q, 1);
      mbar_init(bar_tqempty + 8u * q, 1 + kEpilogueWarps + (GATHER ? kGatherWarps : 0));
    }
    *abort_flag = 0;
    *stopped_here = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == kMmaWarp) tmem_alloc(smem_u32(tmem_slot), kTmemCols);
  // With early set-up only the threads that touch what the previous kernel wrote wait for it: the producer before
  // its first token-row copy, the epilogue warps before their first store.  Dependents are released only by
  // threads that have waited, so a later kernel never starts before the kernel two places back has completed.
  if (!p.early_setup) {
    pdl_wait();
    pdl_launch_dependents();
  }
  if (threadIdx.x == 0) PROF_STAMP(1);
  build_tile_list<kCtaThreads>(p, prefix, order, beg, cnts, class_pos, chunk_sum);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  if (threadIdx.x == 0) PROF_STAMP(2);
  const int total_tiles = dense_tiles + prefix[p.E] * p.n_ft;
  const uint32_t R = (uint32_t)p.ring_slots;

  // Row gather (warps 10 and 11).  Row r of a tile is x[perm[row0 + r] / top_k]; the dense group's rows are their own.  Warp g takes
  // rows 8 i + 4 g .. + 3 of a k-block, a lane 16 bytes of one of them, and puts them where TMA's 128-byte swizzle would.  A row past
  // the tile's end is the tile's last one again.
  [[maybe_unused]] auto gather_rows = [&]() -> bool {
    uint32_t head = 0, kb_idx = 0, tcount = 0;
    bool ok = true;
    const int r0 = 4 * (warp - kGatherWarp0) + (lane >> 3), piece = lane & 7;
    const uint32_t dst0 = base_addr + (uint32_t)(r0 * 128 + ((piece ^ r0) << 4));
    for (;;) {
      const uint32_t q = tcount % kQ;
      if (!mbar_wait_warp(bar_tqfull + 8u * q, (tcount / kQ) & 1u, abort_flag, limit)) { ok = false; break; }
      const STile t = tq[q];
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_tqempty + 8u * q);
      ++tcount;
      if (t.e == kNoTile) break;
      const bool dense = t.e == kDenseTile;
      const uint32_t n = (uint32_t)((t.rows + 15) & ~15), nx = n >> 4;
      const uint32_t row_bytes = (uint32_t)(dense ? p.K2 : p.K) * 2u;
      const char* src = reinterpret_cast<const char*>(dense ? p.gather_src2 : p.gather_src);
      uint32_t off[kMaxTileRows / 8];  // of this lane's piece in its rows
#pragma unroll
      for (int i = 0; i < kMaxTileRows / 8; ++i) {
        if (8u * i >= n) break;
        const int row = t.row0 + min(8 * i + r0, t.rows - 1);
        off[i] = (uint32_t)(dense ? row : __ldg(p.perm + row) / p.top_k) * row_bytes + 16u * (uint32_t)piece;
      }
      const int num_kb = dense ? num_kb2 : num_kb1;
      for (int kb = 0; kb < num_kb; ++kb, src += 2 * kBlockK) {
        if (head + (uint32_t)kWSlots > R) head = 0;  // the producer's allocation, step for step
        head += (uint32_t)kWSlots;
        if (head + nx > R) head = 0;
        const uint32_t dst = dst0 + head * (uint32_t)kSlotBytes;
        head += nx;
        if (!mbar_wait_warp(bar_go + 8u * (kb_idx % kNB), (kb_idx / kNB) & 1u, abort_flag, limit)) { ok = false; break; }
#pragma unroll
        for (int i = 0; i < kMaxTileRows / 8; ++i) {
          if (8u * i >= n) break;
          cp_async_16(dst + (uint32_t)(i * 1024), src + off[i]);
        }
        cp_async_arrive_on(bar_full + 8u * (kb_idx % kNB));
        ++kb_idx;
      }
      if (!ok) break;
    }
    return ok;
  };

  if (warp == kProducerWarp) {
    // ================================================================= TMA producer
    if (!p.inject_producer_stall) {
      uint32_t head = 0, free_slots = R, kb_idx = 0, oldest = 0;
      bool ok = true;
      // Early set-up: until this thread has waited for the previous kernel, token-row copies are put off (their
      // ring space is allocated and their bytes announced) while the weight boxes of up to kNB k-blocks of the first
      // tile go out.  The copies put off are the ring's first allocations, so they are found again by walking it from
      // its start (a list of them would live in local memory, which is cold here).
      bool dep_waited = !p.early_setup;
      uint32_t n_def = 0, def_nx = 0;
      int def_row0 = 0;
      const CUtensorMap* def_map = nullptr;
      auto dep_wait_and_flush = [&]() {
        pdl_wait();
        pdl_launch_dependents();
        dep_waited = true;
        uint32_t h = 0;
        for (uint32_t i = 0; i < n_def; ++i) {
          if (h + (uint32_t)kWSlots > R) h = 0;
          h += (uint32_t)kWSlots;
          if (h + def_nx > R) h = 0;
          if (elect_one())
            tma_load_2d(base_addr + h * (uint32_t)kSlotBytes, def_map, bar_full + 8u * i, (int)i * kbk, def_row0);
          h += def_nx;
        }
      };
      [[maybe_unused]] long long prof_wait_empty = 0, prof_tiles = 0;
      [[maybe_unused]] const long long prof_start = clock64();
      int yield_seen = 0;
      if (p.yield_req != nullptr)
        asm volatile("ld.volatile.global.s32 %0, [%1];" : "=r"(yield_seen) : "l"(p.yield_req) : "memory");
      // Tiles are handed out by a counter in device memory, in the list's order (largest experts first): a CTA
      // that finishes early takes the next tile, whichever CTA would have had it.  The producer publishes every tile
      // it takes -- and finally that there are no more -- in a small queue that the issuer and the epilogue warps follow.
      uint32_t tcount = 0;
      auto publish = [&](const STile& t) -> bool {
        const uint32_t q = tcount % kQ, par = ((tcount / kQ) & 1u) ^ 1u;
        // the epilogue warps free an entry only after the tile before it, which needs its token rows: the copies
        // put off by the early set-up go out before this warp blocks
        if (!dep_waited && !__all_sync(0xffffffffu, mbar_try_wait(bar_tqempty + 8u * q, par))) dep_wait_and_flush();
        if (!mbar_wait_warp(bar_tqempty + 8u * q, par, abort_flag, limit)) return false;
        if (elect_one()) {
          tq[q] = t;
          mbar_arrive(bar_tqfull + 8u * q);
        }
        ++tcount;
        return true;
      };
      const STile no_more{kNoTile, 0, 0, 0};
      // The counter is read a few k-blocks before the current tile's last copy, so that the atomic's round trip hides
      // behind those copies -- and no earlier, so that a CTA does not hold a second tile while another CTA has none.
      // A stop on request therefore takes effect after the tile that had already been taken.
      // The first waves are dealt statically (wave w: tile w * grid + the CTA's index, alternately forwards and
      // backwards): CTAs that run in step start the tiles that share an expert's weights or rows together, and the
      // second reader finds them in L2.  The last few waves' worth of tiles -- the smallest ones, the list being
      // ordered by size -- go to whichever CTA is free, which evens out what the static part left uneven.  A pass that
      // can be stopped on request is dynamic throughout: its next launch only needs the counter to go on.
      const int grid = (int)gridDim.x;
      // (At least the first wave is static, which also spares every CTA a contended atomic at the start.)
      const int w_static = p.all_dynamic ? 0 : static_waves(total_tiles, grid);
      int sw = 0;
      auto next_tile = [&]() -> int {
        if (sw < w_static) {
          const int w = sw++;
          return w * grid + ((w & 1) ? grid - 1 - (int)blockIdx.x : (int)blockIdx.x);
        }
        return lane == 0 ? w_static * grid + atomicAdd(p.tile_ctr, 1) : 0;
      };
      int taken = next_tile();  // lane 0's counts
      for (;;) {
        const int tile = __shfl_sync(0xffffffffu, taken, 0);
        const STile t = tile < total_tiles ? decode_tile(tile, dense_tiles, p, prefix, order, beg, cnts) : no_more;
        if (!publish(t)) {
          ok = false;
          break;
        }
        if (t.e == kNoTile) break;
        const bool dense = t.e == kDenseTile;
        bool stop_after = false;
        const uint32_t n = (uint32_t)((t.rows + 15) & ~15);
        const int w_row0 = t.ft * kFeatPerTile;
        const CUtensorMap* mw = dense ? &map_w2 : &map_w;
        const CUtensorMap* mx = rows_map(xmaps, p, t, n);  // the box of exactly n rows
        const int w_e = dense ? 0 : p.e_base + t.e;
        const int num_kb = dense ? num_kb2 : num_kb1;
        const int fetch_kb = num_kb > 4 ? num_kb - 4 : 0;
        if (!dep_waited) {
          def_nx = n >> 4;
          def_map = mx;
          def_row0 = t.row0;
        }
        for (int kb = 0, k0 = 0; kb < num_kb && ok; ++kb, k0 += kbk) {
          if (kb == fetch_kb) {
            if (p.yield_req != nullptr) {
              // the request word was read a tile ago, so looking at it here does not stall the pipeline; the read for
              // the next tile goes out now
              stop_after = __shfl_sync(0xffffffffu, yield_seen, 0) != 0;
              asm volatile("ld.volatile.global.s32 %0, [%1];" : "=r"(yield_seen) : "l"(p.yield_req) : "memory");
            }
            if (!stop_after) taken = next_tile();
          }
          // The ring is allocated per operand: the weight boxes and the token rows of a k-block are two contiguous
          // pieces that need not be adjacent, so the weights of the next k-block go out as soon as 16 slots are
          // free.  A piece never wraps: it skips what is left at the ring's end.
          const uint32_t nx = n >> 4;
          const bool wrap_w = head + (uint32_t)kWSlots > R;
          const uint32_t pad_w = wrap_w ? R - head : 0u;
          const uint32_t head_w = wrap_w ? 0u : head;
          const bool wrap_x = head_w + (uint32_t)kWSlots + nx > R;
          const uint32_t pad_x = wrap_x ? R - (head_w + (uint32_t)kWSlots) : 0u;
          const uint32_t head_x = wrap_x ? 0u : head_w + (uint32_t)kWSlots;
          auto reclaim = [&](uint32_t need, bool count_limit) {
            // nothing is consumed before the token rows are in: wait for the previous kernel before blocking
            if (!dep_waited && (free_slots < need || (count_limit && kb_idx - oldest >= (uint32_t)kNB)))
              dep_wait_and_flush();
            while (free_slots < need || (count_limit && kb_idx - oldest >= (uint32_t)kNB)) {
              PROF_T0();
              const bool got = mbar_wait_warp(bar_empty + 8u * (oldest % kNB), (oldest / kNB) & 1u, abort_flag, limit);
              PROF_ADD(prof_wait_empty);
              if (!got) return false;
              free_slots += (uint32_t)sizes[oldest % kNB];
              ++oldest;
            }
            return true;
          };
          if (!reclaim((uint32_t)kWSlots + pad_w, true)) { ok = false; break; }
          free_slots -= (uint32_t)kWSlots + pad_w;
          const uint32_t full = bar_full + 8u * (kb_idx % kNB);
          // one copy per operand: both weight boxes (gated: the map's third dimension steps from the gate rows
          // to the up rows; down pass: 256 consecutive rows), then the n token rows
          const uint32_t st_w = base_addr + head_w * (uint32_t)kSlotBytes;
          if (elect_one()) {
            mbar_expect_tx(full, 2u * kWBoxBytes + (GATHER ? 0u : n * 128u));
            if (GATED) tma_load_4d(st_w, mw, full, k0, w_row0, 0, w_e);
            else tma_load_3d(st_w, mw, full, k0, w_row0, w_e);
          }
          if (!reclaim(nx + pad_x, false)) { ok = false; break; }
          free_slots -= nx + pad_x;
          sizes[kb_idx % kNB] = (int)((uint32_t)kWSlots + pad_w + nx + pad_x);
          if (GATHER) {
            if (elect_one()) mbar_arrive(bar_go + 8u * (kb_idx % kNB));
          } else if (dep_waited) {
            if (elect_one()) tma_load_2d(base_addr + head_x * (uint32_t)kSlotBytes, mx, full, k0, t.row0);
          } else {
            ++n_def;
          }
          head = head_x + nx;
          ++kb_idx;
        }
        // (before the next tile's number is looked at: its atomic is still on its way)
        if (!dep_waited) dep_wait_and_flush();
        if (stop_after && ok) {
          *stopped_here = 1;  // no further tile is taken: the other roles finish the published ones and leave
          if (!publish(no_more)) ok = false;
          break;
        }
      }
      if (!dep_waited) dep_wait_and_flush();
      if (!ok && lane == 0) {
        *abort_flag = 1;
        atomicCAS(p.status, kStOk, kStTimeout);
      }
#ifdef MOE_STREAM_PROF
      if (lane == 0) {
        atomicAdd(&g_stream_prof[8 * unit + 0], (unsigned long long)(clock64() - prof_start));
        atomicAdd(&g_stream_prof[8 * unit + 1], (unsigned long long)prof_wait_empty);
      }
#endif
    }
    if (lane == 0) {
      // This CTA takes no more tiles.  The last one that says so puts the counters back for the next launch that uses them
      // -- here, beside the last tile's MMAs and epilogue, because at the CTA's end the next kernel waits for it (0.7 us).
      // After a stop on request the tile counter stays: the next launch of the pass goes on where this one stopped.
      if (*stopped_here) atomicAdd(p.stopped, 1);
      __threadfence();
      if (atomicAdd(p.done_ctr, 1) == (int)gridDim.x - 1) {
        const bool any_stopped = p.stopped != nullptr && *reinterpret_cast<volatile int*>(p.stopped) != 0;
        *p.done_ctr = 0;
        if (!any_stopped) *p.tile_ctr = 0;
      }
    }
  } else if (warp >= kMmaWarp) {
    // ================================================================= MMA issuer (row gather: and warps 10 and 11)
    uint32_t head = 0, kb_idx = 0, use0 = 0, use1 = 0, next_half = 0;
    bool ok = true;
    [[maybe_unused]] long long prof_wait_full = 0, prof_wait_acc = 0, prof_tiles = 0;
    [[maybe_unused]] const long long prof_start = clock64();
    const uint32_t desc_hi = (uint32_t)(umma_smem_desc(0) >> 32);
    const uint32_t lo_base = (uint32_t)umma_smem_desc(base_addr);  // slot 0
    constexpr uint32_t lo_slot = (uint32_t)kSlotBytes >> 4, lo_box = (uint32_t)kWBoxBytes >> 4;
    uint32_t tcount = 0;
    const bool gathers = GATHER && warp >= kGatherWarp0;
    if (gathers) ok = gather_rows();
    while (!gathers) {
      const uint32_t q = tcount % kQ;
      if (!mbar_wait_warp(bar_tqfull + 8u * q, (tcount / kQ) & 1u, abort_flag, limit)) {
        ok = false;
        break;
      }
      const STile t = tq[q];
      __syncwarp();
      if (elect_one()) mbar_arrive(bar_tqempty + 8u * q);
      ++tcount;
      if (t.e == kNoTile) break;
      const uint32_t n = (uint32_t)((t.rows + 15) & ~15);
      const bool big = n > 128u;
      uint32_t d_a, d_b;
      PROF_T0();
      if (big) {
        if (!mbar_wait_warp(bar_tempty, (use0 & 1u) ^ 1u, abort_flag, limit) ||
            !mbar_wait_warp(bar_tempty + 8u, (use1 & 1u) ^ 1u, abort_flag, limit)) { ok = false; break; }
        d_a = tmem_base;
        d_b = tmem_base + 256u;
      } else {
        const uint32_t h = next_half;
        next_half ^= 1u;
        if (!mbar_wait_warp(bar_tempty + 8u * h, ((h ? use1 : use0) & 1u) ^ 1u, abort_flag, limit)) { ok = false; break; }
        d_a = tmem_base + 256u * h;
        d_b = d_a + 128u;
        if (h) ++use1; else ++use0;
      }
      PROF_ADD(prof_wait_acc);
#ifdef MOE_STREAM_PROF
      ++prof_tiles;
#endif
      tc_fence_after();
      const uint32_t idesc = FP8 ? umma_idesc_e4m3(128, n) : umma_idesc(128, n);
      const int num_kb = t.e == kDenseTile ? num_kb2 : num_kb1;
      for (int kb = 0; kb < num_kb; ++kb) {
        if (head + (uint32_t)kWSlots > R) head = 0;  // the producer's allocation, step for step
        const uint32_t pos_w = head;
        head += (uint32_t)kWSlots;
        if (head + (n >> 4) > R) head = 0;
        const uint32_t pos_x = head;
        head += n >> 4;
        {
          PROF_T0();
          const bool got = mbar_wait_warp(bar_full + 8u * (kb_idx % kNB), (kb_idx / kNB) & 1u, abort_flag, limit);
          PROF_ADD(prof_wait_full);
          if (!got) { ok = false; break; }
        }
        if (kb_idx == 0) PROF_STAMP(3);
        if (GATHER) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the rows came by cp.async
        tc_fence_after();
        const uint32_t lo_w0 = lo_base + pos_w * lo_slot, lo_w1 = lo_w0 + lo_box, lo_x = lo_base + pos_x * lo_slot;
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < kBlockK / kUmmaK; ++kk) {
            const uint32_t adv = (uint32_t)((kk * kUmmaK * 2) >> 4);  // +32 bytes per MMA, in 16-byte units
            const uint32_t acc = (kb | kk) != 0 ? 1u : 0u;
            if (FP8) {
              umma_e4m3_lo(d_a, lo_w0 + adv, lo_x + adv, desc_hi, idesc, acc);
              umma_e4m3_lo(d_b, lo_w1 + adv, lo_x + adv, desc_hi, idesc, acc);
            } else {
              umma_bf16_lo(d_a, lo_w0 + adv, lo_x + adv, desc_hi, idesc, acc);
              umma_bf16_lo(d_b, lo_w1 + adv, lo_x + adv, desc_hi, idesc, acc);
            }
          }
          umma_commit(bar_empty + 8u * (kb_idx % kNB));  // the k-block's slots are free once these MMAs have read them
        }
        ++kb_idx;
      }
      if (!ok) break;
      if (elect_one()) {
        umma_commit(bar_tfull + (big ? 0u : 8u * (next_half ^ 1u)));
        if (big) umma_commit(bar_tfull + 8u);
      }
      if (big) {
        ++use0;
        ++use1;
      }
    }
    if (!ok && lane == 0) {
      *abort_flag = 1;
      atomicCAS(p.status, kStOk, kStTimeout);
    }
    PROF_STAMP(4);
#ifdef MOE_STREAM_PROF
    if (lane == 0) {
      atomicAdd(&g_stream_prof[8 * unit + 2], (unsigned long long)(clock64() - prof_start));
      atomicAdd(&g_stream_prof[8 * unit + 3], (unsigned long long)prof_wait_full);
      atomicAdd(&g_stream_prof[8 * unit + 4], (unsigned long long)prof_wait_acc);
      atomicAdd(&g_stream_prof[8 * unit + 5], (unsigned long long)prof_tiles);
      atomicAdd(&g_stream_prof[8 * unit + 6], (unsigned long long)kb_idx);
    }
#endif
  } else {
    // ================================================================= epilogue (warps 0-7)
    // TMEM lane = weight row (output feature) of each box, column = token.  A warp takes 32 features x 16 tokens at a time, in
    // the fragments of 8 x 8 matrices: a thread then has gate and up of the same elements and neighbouring tokens side by
    // side, stmatrix transposes the bf16 results into the warp's staging, and they leave as 16 bytes of a row.  (With lanes
    // as features and neighbouring lanes exchanging values for 4-byte stores 256 columns of 128 lanes took 5700 clocks, gated
    // 8200; this 3100 and 3400.)
    if (p.early_setup) {
      pdl_wait();
      pdl_launch_dependents();
    }
    uint32_t use0 = 0, use1 = 0, next_half = 0;
    bool ok = true;
    const int lg = warp & 3;                         // TMEM lane group of this warp: lanes 32 lg .. 32 lg + 31
    const int c_first = 16 * (warp >> 2), c_step = 32;
    const uint32_t lane_base = ((uint32_t)(lg * 32)) << 16;
    // staging: 16 tokens of 64 bytes, the 16-byte pieces XOR-swizzled by pairs of tokens (no bank conflicts either way)
    uint8_t* const stg = staging + warp * kStagingBytes;
    auto piece = [](int tok, int i) { return tok * 64 + ((i ^ ((tok >> 1) & 3)) << 4); };
    const int st_tok = (lane & 7) + 8 * (lane >> 4), st_piece = (lane >> 3) & 1;  // stmatrix: this lane's row of 8 features
    const uint32_t st0 = smem_u32(stg) + (uint32_t)piece(st_tok, st_piece), st1 = smem_u32(stg) + (uint32_t)piece(st_tok, st_piece + 2);
    const int ld_tok = lane >> 2, ld_piece = lane & 3;                            // and the token and features it stores
    const int fr_row = lane >> 2, fr_col = 2 * (lane & 3);                        // fragments: its feature and token
    uint32_t tcount = 0;
    for (;;) {
      const uint32_t q = tcount % kQ;
      if (!mbar_wait_warp(bar_tqfull + 8u * q, (tcount / kQ) & 1u, abort_flag, limit)) {
        ok = false;
        break;
      }
      const STile t = tq[q];
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_tqempty + 8u * q);
      ++tcount;
      if (t.e == kNoTile) break;
      const bool dense = t.e == kDenseTile;
      const uint32_t n = (uint32_t)((t.rows + 15) & ~15);
      const bool big = n > 128u;
      __nv_bfloat16* const out = dense ? p.out2 : p.out;
      const int n_feat = dense ? p.n_feat2 : p.n_feat;
      const int f0 = t.ft * kFeatPerTile + lg * 32;  // this warp's first feature (down pass: of box 0, and + 128 of box 1)
      float ws_a[4], ws_b[4];                        // FP8: scales of this thread's weight rows, 8 apart
      float rs[4];                                   // ... and of its tokens in the next chunk
      const float* rsp = nullptr;
      auto fetch_scales = [&](int c) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int tok = c + fr_col + (i & 1) + 8 * (i >> 1);
          rs[i] = tok < t.rows ? __ldg(rsp + tok) : 0.f;
        }
      };
      if (FP8) {
        rsp = (dense ? p.row_scale2 : p.row_scale) + t.row0;
        const float* const wsp = dense ? p.w_scale2 : p.w_scale + (size_t)(p.e_base + t.e) * (GATED ? 2 : 1) * n_feat;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int f = f0 + fr_row + 8 * i, f2 = GATED ? f : f + kWBoxRows;
          ws_a[i] = f < n_feat ? __ldg(wsp + f) : 0.f;
          ws_b[i] = f2 < n_feat ? __ldg(wsp + (GATED ? n_feat + f : f2)) : 0.f;
        }
        fetch_scales(c_first);
      }
      uint32_t h = 0, d_a, d_b;
      if (big) {
        if (!mbar_wait_warp(bar_tfull, use0 & 1u, abort_flag, limit) ||
            !mbar_wait_warp(bar_tfull + 8u, use1 & 1u, abort_flag, limit)) { ok = false; break; }
        ++use0;
        ++use1;
        d_a = tmem_base;
        d_b = tmem_base + 256u;
      } else {
        h = next_half;
        next_half ^= 1u;
        if (!mbar_wait_warp(bar_tfull + 8u * h, (h ? use1 : use0) & 1u, abort_flag, limit)) { ok = false; break; }
        if (h) ++use1; else ++use0;
        d_a = tmem_base + 256u * h;
        d_b = d_a + 128u;
      }
      tc_fence_after();
      d_a += lane_base;
      d_b += lane_base;
      auto release_acc = [&]() {  // hand the accumulator half (or both) back to the MMA issuer
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if (big) {
            mbar_arrive(bar_tempty);
            mbar_arrive(bar_tempty + 8u);
          } else {
            mbar_arrive(bar_tempty + 8u * h);
          }
        }
      };
      // stages 32 features x 16 tokens and stores them: features f.. of tokens c..
      auto put = [&](const uint32_t (&lo)[4], const uint32_t (&hi)[4], int f, int c) {
        stmatrix_trans(st0, lo);
        stmatrix_trans(st1, hi);
        __syncwarp();
        uint4 v[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) v[i] = *reinterpret_cast<const uint4*>(stg + piece(ld_tok + 8 * i, ld_piece));
        __syncwarp();  // read: the staging may be written again
        f += 8 * ld_piece;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int tok = c + ld_tok + 8 * i;
          if (tok < t.rows && f < n_feat) *reinterpret_cast<uint4*>(out + (size_t)(t.row0 + tok) * n_feat + f) = v[i];
        }
      };
      // the loads of the next 16-token chunk are in flight while this one is converted and stored
      uint32_t na[2][8], nb[2][8];  // [features 0-15 or 16-31][fragments]
      auto load = [&](int c) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          tmem_ld_frag(d_a + ((uint32_t)(16 * k) << 16) + (uint32_t)c, na[k]);
          tmem_ld_frag(d_b + ((uint32_t)(16 * k) << 16) + (uint32_t)c, nb[k]);
        }
      };
      if (c_first < t.rows) load(c_first);
      else release_acc();
      for (int c = c_first; c < t.rows; c += c_step) {
        uint64_t va[2][4], vb[2][4];  // pairs of neighbouring tokens
        tmem_ld_wait();
#pragma unroll
        for (int k = 0; k < 2; ++k)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            va[k][i] = f32x2(__uint_as_float(na[k][2 * i]), __uint_as_float(na[k][2 * i + 1]));
            vb[k][i] = f32x2(__uint_as_float(nb[k][2 * i]), __uint_as_float(nb[k][2 * i + 1]));
            if (FP8) {
              const uint64_t r = f32x2(rs[2 * (i >> 1)], rs[2 * (i >> 1) + 1]);
              const float wa = ws_a[2 * k + (i & 1)], wb = ws_b[2 * k + (i & 1)];
              va[k][i] = mul2(va[k][i], mul2(r, f32x2(wa, wa)));
              vb[k][i] = mul2(vb[k][i], mul2(r, f32x2(wb, wb)));
            }
          }
        if (c + c_step < t.rows) {
          load(c + c_step);
          if (FP8) fetch_scales(c + c_step);
        } else {
          release_acc();  // read completely
        }
        uint32_t q[2][4];
#pragma unroll
        for (int k = 0; k < 2; ++k)
#pragma unroll
          for (int i = 0; i < 4; ++i) q[k][i] = pack_bf16(GATED ? silu_mul2(va[k][i], vb[k][i]) : va[k][i]);
        put(q[0], q[1], f0, c);
        if (!GATED) {
#pragma unroll
          for (int k = 0; k < 2; ++k)
#pragma unroll
            for (int i = 0; i < 4; ++i) q[k][i] = pack_bf16(vb[k][i]);
          put(q[0], q[1], f0 + kWBoxRows, c);
        }
      }
    }
    if (!ok && lane == 0) {
      *abort_flag = 1;
      atomicCAS(p.status, kStOk, kStTimeout);
    }
  }

  // ---- teardown
  if (threadIdx.x == 0) PROF_STAMP(5);
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0) PROF_STAMP(6);
  if (*abort_flag) {
    // give copies still in flight time to land in this CTA's shared memory before it is released
    for (int i = 0; i < 64; ++i) __nanosleep(1000);
    __syncthreads();
  }
  if (warp == kMmaWarp) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kTmemCols);
  }
}

template <typename Kernel>
cudaError_t launch_variant(Kernel kern, const CUtensorMap& mw, const CUtensorMap& mw2, const StreamMaps& xm,
                           const StreamParams& prm, int grid, int threads, size_t smem, cudaStream_t stream, bool overlap) {
  cudaError_t err = ensure_dynamic_smem(kern, smem);
  if (err != cudaSuccess) return err;
  return launch_pdl(overlap, kern, dim3(grid), dim3(threads), smem, stream, mw, mw2, xm, prm);
}

}  // namespace

StreamPlan* stream_plan_create() {
  StreamPlan* p = new (std::nothrow) StreamPlan();
  if (p != nullptr) {
    memset(&p->mw, 0, sizeof p->mw);
    memset(&p->mw2, 0, sizeof p->mw2);
    memset(&p->xm, 0, sizeof p->xm);
  }
  return p;
}
void stream_plan_destroy(StreamPlan* plan) { delete plan; }
int64_t stream_plan_encoded(const StreamPlan* plan) { return plan->encoded; }

cudaError_t launch_gemm_stream(const GemmProblem& p, const GemmDenseGroup* dense, int max_ctas, int* status,
                               cudaStream_t stream, int* n_launches) {
  if (dense != nullptr && dense->rows <= 0) dense = nullptr;
  if (p.rows_bound <= 0 && dense == nullptr) return cudaSuccess;
  if (p.rows_bound <= 0) return cudaErrorInvalidValue;  // a dense group never comes without its routed pass
  if (!swap_ab_supports(p, dense)) return cudaErrorNotSupported;
  const bool gather = p.gather_src != nullptr;
  // (a row's offset in the source is 32 bits; what it reads comes from the kernel in front of it, so it does without the overlap)
  if (gather && (!p.gated || p.fp8 || p.perm == nullptr || p.top_k < 1 || p.K % kBlockK != 0 ||
                 (dense != nullptr && (dense->A == nullptr || dense->K % kBlockK != 0 ||
                                       dense->rows * (int64_t)dense->K * 2 > 0xffffffffLL)) ||
                 (p.rows_bound / p.top_k + 1) * (int64_t)p.K * 2 > 0xffffffffLL || p.rows_bound <= kGemmOverlapMaxRows))
    return cudaErrorNotSupported;
  const int groups = p.offsets ? p.E : 1;
  const int e_begin = p.offsets ? p.e_begin : 0;
  const int e_end = (p.offsets && p.e_end >= 0) ? p.e_end : groups;
  if (e_begin < 0 || e_end > groups || e_begin >= e_end) return cudaErrorInvalidValue;

  if (p.plan == nullptr || p.tile_counters == nullptr) return cudaErrorInvalidValue;
  StreamPlan& plan = *p.plan;
  cudaError_t err = update_plan(plan, p, dense, groups, false);
  if (err != cudaSuccess) return err;
  StreamParams prm;
  int64_t tiles;
  if (!fill_params(prm, tiles, p, dense, e_begin, e_end, status)) return cudaErrorInvalidValue;

  const size_t tail = kEpilogueWarps * kStagingBytes + (2 * kNB + 4 + 2 * kQ + (gather ? kNB : 0)) * sizeof(uint64_t) + 3 * sizeof(uint32_t) + kNB * sizeof(int) + kQ * sizeof(STile) +
                      (4 * (size_t)(prm.E + 1) + kSizeClasses + 32) * sizeof(int);
  const int slots = (int)((kSmemBudget - 1024 - (int)tail) / kSlotBytes);
  if (slots < 2 * (kWSlots + kMaxTileRows / 16)) return cudaErrorNotSupported;
  prm.ring_slots = slots;
#ifdef MOE_STREAM_PROF
  if (const char* rs = getenv("MOE_STREAM_RING_SLOTS")) {  // debug build only: a smaller ring, to see what in-flight bytes buy
    const int v = atoi(rs);
    if (v >= 2 * (kWSlots + kMaxTileRows / 16) && v < slots) prm.ring_slots = v;
  }
#endif
  const size_t smem = 1024 + (size_t)slots * kSlotBytes + tail;

  int grid = (int)(tiles < (int64_t)max_ctas ? tiles : (int64_t)max_ctas);
  if (grid < 1) grid = 1;
  // one tile per CTA at most: any order will do (1.3 us of the tiny layer's 64-token step)
  if (tiles <= (int64_t)grid) prm.sort_tiles = 0;
  const bool overlap = p.rows_bound <= kGemmOverlapMaxRows;
  if (gather) {
    prm.early_setup = 0;
    prm.gather_src = static_cast<const __nv_bfloat16*>(p.gather_src);
    prm.gather_src2 = dense ? static_cast<const __nv_bfloat16*>(dense->A) : nullptr;
    prm.perm = p.perm;
    prm.top_k = p.top_k;
  }
  auto launch = [&](auto kern, int threads) {
    return launch_variant(kern, plan.mw, plan.mw2, plan.xm, prm, grid, threads, smem, stream, overlap);
  };
  if (p.fp8)
    err = p.gated ? launch(grouped_gemm_stream_kernel<true, true, false>, kThreads) : launch(grouped_gemm_stream_kernel<false, true, false>, kThreads);
  else if (gather)
    err = launch(grouped_gemm_stream_kernel<true, false, true>, kThreadsGather);
  else
    err = p.gated ? launch(grouped_gemm_stream_kernel<true, false, false>, kThreads) : launch(grouped_gemm_stream_kernel<false, false, false>, kThreads);
  if (err == cudaSuccess && n_launches) *n_launches += 1;
  return err;
}

#ifdef MOE_STREAM_PROF
}  // namespace moe
extern "C" int moe_debug_stream_ts(unsigned long long* host) {
  return (int)cudaMemcpyFromSymbol(host, moe::g_stream_ts, sizeof(unsigned long long) * 8 * 256);
}
extern "C" int moe_debug_stream_prof(unsigned long long* host, int clear) {
  cudaError_t e = cudaMemcpyFromSymbol(host, moe::g_stream_prof, sizeof(unsigned long long) * 8 * 256);
  if (e == cudaSuccess && clear) {
    static unsigned long long zeros[8 * 256] = {};
    e = cudaMemcpyToSymbol(moe::g_stream_prof, zeros, sizeof zeros);
  }
  return (int)e;
}
namespace moe {
#endif

}  // namespace moe
