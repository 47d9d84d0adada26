// Rules by which the host cuts launches and picks kernels: plain functions of sizes, without CUDA.
#pragma once
#include <stdint.h>

namespace moe {

// ---- dispatch layout (layout.cu): slots per chunk, that is per CTA; a multiple of kLayoutMinChunk.
// About 64 chunks of 1024 to 4096 slots (half as many for more than 512 experts: every CTA reads all chunks' counts, so
// fewer, larger chunks where there are many).  That reading is chunks x chunks x E words in all, so behind 148 chunks of
// 4096 -- one CTA per SM -- the chunk grows instead of their number.  Back to back, us, 148 chunks | chunks of 4096 slots |
// count -> scan -> place over chunks of 256:
//   2^20 slots: 64 experts 16 | 22 | 37, 256 19 | 27 | 41, 1024 25 | 48 | 53;  2^22: 42 | 84 | 124, 49 | 153 | 135,
//   57 | 414 | 194;  2^24: 220 | - | 487, 228 | - | 638, 238 | - | 1143.  (296 chunks: 2^20 22, 27, 48; 2^24 201, 218, 250.)
constexpr int64_t kLayoutMinChunk = 1024;  // one step of 32 slots per warp
constexpr int64_t kLayoutMidChunk = 4096;
constexpr int kLayoutChunkTarget = 64, kLayoutMaxChunks = 148;

inline int64_t layout_chunk_slots(int64_t n_slots, int E) {
  const auto per_cta = [&](int64_t ctas) {
    return ((n_slots + ctas - 1) / ctas + kLayoutMinChunk - 1) / kLayoutMinChunk * kLayoutMinChunk;
  };
  const int64_t wanted = per_cta(E > 512 ? kLayoutChunkTarget / 2 : kLayoutChunkTarget), least = per_cta(kLayoutMaxChunks);
  if (wanted <= kLayoutMidChunk) return wanted;
  return least > kLayoutMidChunk ? least : kLayoutMidChunk;
}

// ---- which tensor-core kernel takes a pass of a PREFILL context (AUTO), for problems of more than 8192 rows
// From the rows per expert R = rows / experts, the pass's K and output features, and how many CTAs the grid has.  The small-M
// kernel reads an expert's weights once for up to 256 rows, multiplies exactly the rows there are and moves fewer bytes per
// flop; the large-M kernel multiplies rows in steps of 128, but its tiles are half as large and its epilogue always overlaps
// the next tile, which counts where K is short.  Both draw the GPU's power limit in steps of a millisecond and more.
// Measured with an epilogue of the small-M kernel that took twice as long as today's.  A context that has all SMs asks
// pair_is_faster, below, first; one with an SM budget goes by these lines alone.  Measured again with budgets of 48, 74 and 100
// SMs, 96 layers and sizes, today's kernels: the choice is within 1.5 % of the best of the four combinations in 77 of them.  It is
// behind with FP8 where the large-M kernel multiplies much padding (2048 / 768 x 128, 162 rows per expert, that is 256: ll
// against ss 1.14 with every budget, 281 rows 1.03; 2560 / 1024 x 512, 187 rows sl 1.06 with 100 SMs), and with 48 SMs where experts
// have half a large-M tile of rows (64: ss 1.08, with FP8 1.15; 72: sl 1.05).
// Whole steps in the sustained state, us, gated pass / down pass on s = small-M, l = large-M; "K / K' x E" is a layer of
// hidden K, inter K' and E experts (the gated pass has K and K' features, the down pass K' and K).
//   bf16, gated pass (sl : ll)
//     512 / 2048 x 8    R = 1100 100 : 84, 8000 508 : 472;  768 / 512 x 128  100 102 : 99, 160 130 : 131, 300 182 : 181
//     1024 / 512 x 64   192 (256 tiles of 256 rows) 101 : 96, 400 (512) 157 : 153, 700 (768) 231 : 233;  x 512  24 313 : 338, 160
//                       (2048) 528 : 589;  1024 / 256 x 256  40 116 : 121, 200 (512) 212 : 208, 300 (1024) 277 : 284
//     1280 / 768 x 128  72 181 : 182, 96 195 : 193, 160 250 : 271, 600 594 : 604;  1536 / 512 x 128  72 156 : 158, 96 169 : 168,
//                       160 216 : 229, 300 319 : 331
//     2048 / 768 x 128  72 261 : 268, 96 281 : 282, 108 291 : 289, 120 308 : 309, 144 348 : 392, 220 415 : 436;
//                x 512  24 809 : 922, 48 890 : 963, 96 1024 : 1051, 160 1363 : 1679
//     few tiles: 2048 / 768 x 4  2100 (216 tiles of 256 rows on 148 CTAs) 131 : 120, 4000 (384) 221 : 216, 8000 411 : 409;
//                7168 / 512 x 8  1100 (160) 297 : 278, 2000 (256) 467 : 493
//   bf16, down pass (ss : sl)
//     2048 / 256 x 128  160 182 : 178, 400 352 : 330;  1536 / 512 x 128  160 218 : 216, 200 251 : 239, 600 553 : 521
//     2048 / 768 x 128  72 263 : 261, 120 308 : 308, 144 339 : 348, 180 378 : 381, 200 403 : 395;  x 512  24 794 : 809, 48 869 :
//                890, 96 1041 : 1024, 144 1236 : 1317, 200 1479 : 1457
//     1792 / 1024 x 128  72 293 : 296, 112 331 : 329, 160 387 : 402, 300 603 : 610, 600 1019 : 996
//     7168 / 2048 x 256 + shared  256 8222 : 8616, 500 14097 : 14535, 750 20305 : 20791, 1024 26879 : 26662
//   FP8, gated pass (sl : ll)
//     1024 / 256 x 256  40 95 : 94, 64 107 : 102;  1536 / 512 x 128  72 112 : 105, 160 166 : 160;  1792 / 1024 x 128  72 182 : 181,
//                       160 273 : 288, 300 416 : 413
//     2048 / 768 x 128  72 168 : 169, 96 182 : 179, 120 209 : 197, 160 250 : 254, 220 292 : 279;  x 512  24 464 : 514, 48 519 :
//                560, 72 573 : 596, 96 628 : 632, 300 1417 : 1437;  2048 / 256 x 128  80 106 : 99, 160 154 : 143
//     2560 / 1024 x 256  96 481 : 480, 128 569 : 607, 180 714 : 770;  2560 / 1536 x 128  250 634 : 659, 350 842 : 793
//     4096 / 1536 x 128  320 1101 : 1179, 1000 2821 : 2926;  7168 / 2048 x 256 + shared  256 4681 : 5073, 1024 14100 : 14878;
//     few features: 2560 / 768 x 64  140 157 : 157, 250 209 : 199;  3072 / 768 x 128  160 343 : 368, 250 438 : 436, 400 634 : 665;
//                       4096 / 512 x 128  160 339 : 357, 200 378 : 375;  x 32  260 144 : 140, 800 331 : 316
//   FP8, down pass (ss : sl)
//     2560 / 1024 x 512  64 860 : 871, 96 972 : 960, 140 1208 : 1261, 180 1414 : 1429, 220 1678 : 1558;  x 128  96 261 : 256, 160
//                360 : 352;  2560 / 1536 x 128  72 327 : 330, 112 383 : 378, 160 481 : 490, 200 558 : 538
//     7168 / 2048 x 256 + shared  256 4603 : 4681, 384 6227 : 6163, 750 11352 : 10958
constexpr int kMinGatedK = 640, kShortGatedK = 1152;               // bf16 gated pass
constexpr int kMinDownK = 640, kMidDownK = 960, kLongDownK = 2048;  // down pass
constexpr int kFp8ShortGatedK = 1792, kFp8MidGatedK = 2432, kFp8LongGatedK = 3584, kFp8FewFeatures = 1024;

inline bool small_m_is_faster(bool fp8, bool gated, int K, int n_feat, int64_t rows, int64_t E, int ctas) {
  const auto up_to = [&](int64_t r) { return rows <= r * E; };
  // the small-M kernel's tiles, in half waves of the grid; of fewer than one and a half waves half the second is idle, which
  // 128-row tiles fill
  const int64_t chunks = (rows + 255) / 256 > E ? (rows + 255) / 256 : E, feat_per_tile = gated ? 128 : 256;
  const int64_t half_waves = 2 * chunks * ((n_feat + feat_per_tile - 1) / feat_per_tile) / ctas;
  if (half_waves < 3) return false;
  if (gated && !fp8) return K >= kShortGatedK || (K >= kMinGatedK && (up_to(64) || half_waves >= 8));
  if (gated) {
    if (K < kFp8MidGatedK) return K >= kFp8ShortGatedK && up_to(64);
    return n_feat < kFp8FewFeatures ? up_to(200) : K >= kFp8LongGatedK || up_to(300);
  }
  if (fp8) return K >= kLongDownK ? up_to(400) : K >= kMidDownK && up_to(180);
  if (K >= kLongDownK) return true;
  if (K >= kMidDownK) return up_to(350);
  return K >= kMinDownK && (up_to(64) || (!up_to(120) && up_to(190)));
}

// ---- ... and whether the two-CTA kernel takes it before either of them, where it may use all SMs (gemm_pair.cu)
// It multiplies exactly the rows there are, like the small-M kernel, and every epilogue overlaps the next tile, like the
// large-M kernel's; but a tile's operands come in the same number of bytes as the small-M kernel's (per flop) through twice as
// many k-blocks, so with long K the small-M kernel stays ahead.  Whole steps in the sustained state, each over the best of the
// nine combinations, gated pass / down pass on s = small-M, l = large-M, p = pairs (ls is never near the best).  Medians of eight
// interleaved blocks of 0.1 s; the medians of the odd and of the even blocks are up to 1.5 % apart in 40 of 53 measurements, up
// to 2.5 % in 47, and 6.5 % at worst (steps of a millisecond and more, where a block may meet another power state).
//                               R     ss    sl    sp    ll    lp    ps    pl    pp
//   bf16  2048 / 768 x 128    162  1.023 1.064 1.013 1.178 1.124 1.015 1.051 1.000
//                             281  1.000 1.017 1.013 1.095 1.084 1.038 1.047 1.046
//                             375  1.019 1.011 1.000 1.050 1.041 1.020 1.017 1.007
//                             512  1.019 1.017 1.000 1.087 1.048 1.019 1.023 1.004
//         4096 / 1536 x 128   300  1.000 1.031 1.000 1.139 1.102 1.032 1.063 1.034
//                             350  1.006 1.003 1.000 1.061 1.059 1.022 1.034 1.022
//                             420  1.017 1.052 1.000 1.185 1.139 1.042 1.084 1.045
//                             480  1.013 1.040 1.000 1.105 1.080 1.047 1.076 1.073
//                             540  1.008 1.028 1.000 1.107 1.079 1.023 1.047 1.015
//         2560 / 1536 x 128   300  1.000 1.036 1.014 1.139 1.147 1.041 1.064 1.049
//                             375  1.003 1.010 1.000 1.078 1.067 1.007 1.028 1.006
//                             450  1.007 1.031 1.000 1.127 1.091 1.014 1.041 1.014
//                             540  1.005 1.026 1.002 1.079 1.058 1.003 1.025 1.000
//         2048 / 1408 x 64    300  1.000 1.032 1.017 1.099 1.085 1.030 1.061 1.046
//                             375  1.003 1.016 1.003 1.037 1.033 1.001 1.015 1.000
//                             450  1.024 1.046 1.018 1.094 1.070 1.015 1.028 1.000
//   FP8   2048 / 768 x 128    128  1.008 1.022 1.008 1.063 1.034 1.000 1.026 1.000
//                             156  1.040 1.076 1.018 1.157 1.097 1.021 1.061 1.000
//                             260  1.019 1.018 1.000 1.040 1.021 1.017 1.018 1.000
//                             300  1.003 1.007 1.000 1.034 1.025 1.017 1.021 1.016
//                             340  1.019 1.004 1.007 1.000 1.004 1.017 1.002 1.006
//                             375  1.033 1.017 1.018 1.030 1.033 1.024 1.009 1.000
//                             420  1.042 1.048 1.010 1.086 1.050 1.022 1.036 1.000
//                             540  1.019 1.009 1.006 1.024 1.015 1.005 1.007 1.000
//         2560 / 1024 x 512   125  1.000 1.030 1.013 1.099 1.075 1.023 1.048 1.030
//                             187  1.018 1.037 1.002 1.147 1.105 1.000 1.040 1.003
//                             312  1.003 1.000 1.000 1.049 1.041 1.008 1.021 1.007
//         2560 / 1024 x 128   187  1.046 1.058 1.023 1.132 1.092 1.024 1.043 1.000
//                             260  1.009 1.012 1.000 1.057 1.047 1.014 1.019 1.007
//                             375  1.029 1.012 1.012 1.024 1.023 1.013 1.006 1.000
//         1280 / 768 x 128    160  1.046 1.077 1.033 1.134 1.088 1.018 1.045 1.000
//                             300  1.011 1.002 1.006 1.000 1.005 1.016 1.006 1.012
//                             512  1.037 1.028 1.015 1.021 1.007 1.022 1.016 1.000
//         1536 / 512 x 128    160  1.048 1.093 1.029 1.125 1.065 1.016 1.063 1.000
//                             300  1.002 1.011 1.000 1.030 1.023 1.015 1.019 1.015
//                             512  1.040 1.034 1.015 1.033 1.015 1.031 1.018 1.000
//         1024 / 512 x 64     156  1.041 1.043 1.030 1.037 1.026 1.018 1.021 1.000
//                             260  1.081 1.047 1.069 1.000 1.022 1.053 1.015 1.033
//                             375  1.077 1.048 1.069 1.000 1.013 1.034 1.013 1.032
//                             512  1.056 1.029 1.040 1.000 1.007 1.026 1.006 1.016
//                             700  1.058 1.035 1.033 1.006 1.001 1.023 1.004 1.000
//                            1250  1.053 1.031 1.032 1.000 1.001 1.017 1.003 1.005
// An earlier sweep, the layers and sizes it has alone, two blocks each (up to 4 % apart):
//   bf16  2048 / 768 x 128    R = 69 ss 1.007 sl 1.000 sp 1.006 pp 1.009; 96 ss 1.011 sl 1.000 sp 1.015 pp 1.013; 1000 ss 1.040 sl 1.035
//                             sp 1.012 pp 1.000; 1875 ss 1.062 sl 1.035 sp 1.014 pp 1.000
//         4096 / 1536 x 128   125 ss 1.000 sl 1.026 sp 1.010 pp 1.029; 1000 ss 1.014 sl 1.029 sp 1.000 pp 1.038
//         2560 / 1024 x 512   64 ss 1.004 sl 1.019 sp 1.014 pp 1.040; 187 ss 1.000 sl 1.053 sp 1.004 pp 1.016; 312 ss 1.001 sl 1.030
//                             sp 1.018 pp 1.016; 469 ss 1.000 sl 1.021 sp 1.002 pp 1.035
//         7168 / 2048 x 256   64 ss 1.015 sl 1.058 sp 1.019 pp 1.045; 128 ss 1.008 sl 1.048 sp 1.000 pp 1.031; 250 ss 1.010 sl 1.050
//          + shared           sp 1.000 pp 1.042; 500 ss 1.024 sl 1.017 sp 1.000 pp 1.097; 937 ss 1.037 sl 1.009 sp 1.000 pp 1.111
//         1024 / 512 x 64     156 ss 1.051 sl 1.022 ll 1.060 pl 1.000 pp 1.003; 375 ss 1.067 sl 1.031 ll 1.022 pl 1.000 pp 1.021; 1250
//                             ss 1.059 sl 1.029 ll 1.035 pl 1.000 pp 1.007
//         1536 / 512 x 128    156 ss 1.030 sl 1.030 ll 1.117 pl 1.018 pp 1.000; 625 ss 1.048 sl 1.009 ll 1.048 pl 1.000 pp 1.010
//         few tiles: 512 / 2048 x 8  R = 1125 ll 1.005 pl 1.038; 7500 ll 1.018 pl 1.015;  7168 / 512 x 8  1125 ll 1.000 pl 1.022; 2000
//                             ll 1.062 pl 1.007
//   FP8   2048 / 768 x 128    69 sl 1.005 ll 1.019 pl 1.003 pp 1.007; 96 sl 1.006 ll 1.001 pl 1.000 pp 1.008; 1000 sl 1.045 ll 1.048 pl
//                             1.026 pp 1.000; 1875 sl 1.056 ll 1.041 pl 1.045 pp 1.000
//         2560 / 1024 x 512   64 ss 1.017 sl 1.009 ps 1.010 pp 1.027; 469 ss 1.026 sl 1.025 ps 1.000 pp 1.001
//         4096 / 1536 x 128   125 ss 1.000 sp 1.002 ps 1.010 pp 1.015; 375 ss 1.028 sp 1.000 ps 1.003 pp 1.003; 1000 ss 1.035 sp 1.005
//                             ps 1.009 pp 1.000
//         7168 / 2048 x 256   128 ss 1.000 sp 1.002 pp 1.021; 250 ss 1.005 sp 1.000 pp 1.015; 500 ss 1.000 sp 1.002 pp 1.030; 937
//          + shared           ss 1.027 sp 1.000 pp 1.050; skewed experts, 500 ss 1.025 sp 1.000 pp 1.031
//         2048 / 256 x 128    156 ps 1.000 pl 1.094 pp 1.000; 625 ps 1.013 pl 1.014 pp 1.000
// FP8 down passes with the shortest K and few tiles (1024 / 512 x 64): pairs while an expert is one chunk (156 rows 70.1 us, large-M
// 71.6), not with two (260 rows 88.2 and 86.4, 375 102.8 and 102.4, 512 129.3 and 128.3), level with three (700 165.2).
inline bool pair_is_faster(bool fp8, bool gated, int K, int n_feat, int64_t rows, int64_t E, int ctas) {
  const auto over = [&](int64_t r) { return rows > r * E; };
  const int64_t chunks = (rows + 255) / 256 > E ? (rows + 255) / 256 : E, feat_per_tile = gated ? 128 : 256;
  const int64_t half_waves = 2 * chunks * ((n_feat + feat_per_tile - 1) / feat_per_tile) / ctas;
  if (half_waves < 3) return false;
  if (gated && !fp8) {
    if (K < 640) return half_waves >= 16;
    return K < 1792 ? over(96) : K < 2304 && over(768);
  }
  if (gated) return K < 1280 ? false : K < 2304 ? over(64) : K < 3072 ? over(160) : K < 5632 && over(256);
  if (fp8) return K < 640 ? over(128) && (!over(208) || half_waves >= 8) : K < 896 ? over(128) : K < 1280 ? over(180) : over(256);
  if (K < 896) return K >= 640 && over(128);
  return K < 1792 ? over(350) : over(96);
}

// ---- whether the gated pass of a whole bf16 step gathers its rows itself, where the small-M kernel takes it (gemm_stream.cu)
// It saves the launch that moves the rows, and its write and re-read of them; it costs the two gathering warps' loads once for every 128
// features.  Up to 8192 rows that launch is hidden behind the set-up of the gated pass, which would have to wait for the layout
// instead; with whole tiles of 256 rows the threads that gather cost what they save.  Between the two, time with moved rows over time with
// gathered ones, whole steps of 511 layers and sizes at random (hidden 512 to 7168, inter 128 to 2048, 33 to 512 experts, three in ten skewed),
// geometric mean and worst:
//   inter up to 512                                  1.10, 0.97
//   hidden from 4 inter on                           1.04, 0.97
//   hidden from 2 inter on, up to 144 rows an expert 1.02, 0.98
//   what is left                                     0.98, 0.87:  hidden from 2 inter on, more rows 0.99, 0.94;  hidden below 2 inter 0.97, 0.87
// us, rows moved | gathered (rows per expert):  2048 / 768 x 128  69 255 | 247, 125 299 | 293, 144 317 | 308, 162 333 | 335, 206 370 | 376;  from
//   host buffers 96 490 | 474;  2560 / 1024 x 512  17 1234 | 1210, 64 1425 | 1404, 128 1753 | 1734, 172 1991 | 2050, 250 2626 | 2689;  4096 / 1536 x
//   128  69 852 | 834, 125 987 | 982, 206 1209 | 1275;  2048 / 1408 x 64 + shared  141 288 | 292, 244 390 | 411;  7168 / 2048 x 256 + shared  34 3484 |
//   3457, 128 5185 | 5160, 188 6419 | 6463;  skewed 128 4156 | 4188, 253 6867 | 6955
// A context on part of the SMs moves its rows: V3-shaped, 1500 tokens on 48 SMs beside decode steps 13029 | 13224, skewed 2500 6129 | 6201.
inline bool gather_is_faster(int64_t rows, int64_t E, int H, int I) {
  return rows > 8192 && rows < 256 * E && (I <= 512 || H >= 4 * I || (H >= 2 * I && rows <= 144 * E));
}

// ---- whether a bf16 step of up to 64 tokens makes its passes and its combine in one launch (step_ffn.cu)
// It gains a chain of launches, and tiles half as large where the 256-row tiles of a pass are fewer than the CTAs or fill half of a
// second wave; it loses 1.2 to 1.5 us of an SM for each tile, which shows where a tile's k-blocks are few, and seams between the tiles of a
// CTA.  So few slots (T * k) gain at nearly any shape, many only where each CTA has about one tile, or where the weights take so long that
// the stream over the seam between the passes counts.  The lines were drawn through 3600 layers and sizes at random (hidden and
// inter 64 to 7168, 4 to 512 experts, top-1 to top-32, with and without a shared expert): steps called one by one, and steps replayed from a
// graph over layers with weights of their own (in brackets), where a launch costs less.  Time with three launches over time with one,
// geometric mean and worst:
//   both passes' tiles on 7/8 of the CTAs, top-16 at most     1.14, 0.91 (1.12, 0.98);  with 132 to 148 tiles 1.07, 0.72 (0.97, 0.77)
//   up to 12 slots                                            1.25, 1.02 (1.17, 0.97)
//   hidden or inter from 1024 on, up to 28 slots              1.18, 1.01 (1.13, 0.95);  29 to 40 slots 1.11, 0.96 (1.03, 0.88);  where the
//     256-row tiles of a pass fit the CTAs and its 128-row tiles do not: few tiles 1.12, 0.98 (1.06, 0.96), more 1.03, 0.96 (1.00, 0.94)
//   both shorter, up to 16 slots and 4 tiles a CTA            1.12, 1.08 (0.99, 0.94);  17 to 28 slots 1.07, 0.93 (0.99, 0.90)
//   4 tiles a CTA, up to 128 slots, top-8 at most             1.15, 0.97 (1.15, 1.04) with hidden or inter from 2048 on; 1.09, 0.94 (1.01, 0.93)
//     where the 256-row tiles of a pass end within half a second wave
//   what is left                                              1.01, 0.56 (0.96, 0.70):  256 / 256 x 32, top-16, 64 tokens 21.8 us | 29.9,
//     960 / 640 x 16, 8, 31 tokens 24.6 | 30.5, 1024 / 512 x 16, 8, 64 25.0 | 28.4, 512 / 1472 x 8, 8, 61 28.4 | 32.5
// A longer down pass, us from a graph, slots over experts in brackets: 7168 / 2048 x 256 + shared, 8  4 tokens 415 | 389, 32 (1) 1544 | 1515, 64
//   (2) 2078 | 2048, skewed 64 617 | 625;  2560 / 1024 x 512, 8  8 160 | 153, 64 (1) 749 | 735;  4096 / 1536 x 128, 8  48 (3) 682 | 673;
//   4096 / 2048 x 32, 4  24 (3) 246 | 237;  2048 / 768 x 128, 8  4 (0.25) 60.3 | 57.1, 5 66.6 | 65.4, 6 (0.38) 73.3 | 74.9;  7168 / 1024 x 64 +
//   shared, 16  12 (3) 426 | 415, 64 (16) 463 | 479;  shorter hidden  1024 / 2048 x 64, 8  16 (2) 117 | 121.5;  1536 / 1536 x 64, 8  8 (1) 99.6 |
//   101.8
// A context on part of the SMs takes it for few tiles only: its decode steps run beside a prefill batch on the others, from which a steadier
// stream takes HBM that those SMs cannot make up for later (V3-shaped, skewed: 64 tokens beside 900, 4540 | 4642 for both).
inline bool step_at_once_is_faster(int64_t T, int k, int E, int H, int I, int Is, int ctas, bool all_sms) {
  const int64_t slots = T * k, groups = slots < E ? slots : E, dense = Is > 0 ? 1 : 0;
  const auto over = [](int64_t n, int64_t d) { return (n + d - 1) / d; };
  const int64_t gated = groups * (I / 64) + Is / 64, down = (groups + dense) * over(H, 128), tiles = gated + down;   // this kernel's
  const int64_t gated256 = groups * over(I, 128) + over(Is, 128), down256 = (groups + dense) * over(H, 256);          // the small-M kernel's
  const bool few = tiles <= 4 * (int64_t)ctas, is_long = H >= 1024 || I >= 1024;
  if (!all_sms && !few) return false;
  if (8 * tiles <= 7 * (int64_t)ctas) return k <= 16;
  if (slots <= 12) return true;
  // a wave of 256-row tiles against two of half as many rows
  const bool level = (gated > ctas && gated256 <= ctas) || (down > ctas && down256 <= ctas);
  if (level && few) return is_long && slots <= 28;
  if (all_sms && H >= 2048 && (I >= 1024 ? slots <= 3 * (int64_t)E : I >= 640 && 3 * slots <= (int64_t)E)) return true;
  if (level) return false;
  if (is_long ? slots <= 28 : few && slots <= 16) return true;
  const auto part = [&](int64_t t) { return t > ctas && 2 * t <= 3 * (int64_t)ctas; };
  return few && k <= 8 && slots <= 128 && (H >= 2048 || I >= 2048 || part(gated256) || part(down256));
}

}  // namespace moe
