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
// (Measured with an epilogue of the small-M kernel that took twice as long as today's, before pair_is_faster, below, was asked
// first: the sizes at which the small-M kernel lost by its epilogue are now mostly the pair kernel's.)
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
// nine combinations, gated pass / down pass on s = small-M, l = large-M, p = pairs (two runs of one differ by up to 1.5 %):
//   bf16  2048 / 768 x 128    R = 69 ss 1.007 sl 1.000 sp 1.006 pp 1.009; 96 1.011 1.000 1.015 1.013; 162 1.021 1.065 1.009 1.000;
//                             281 1.000 1.021 1.007 1.051; 512 1.030 1.021 1.000 1.022; 1000 1.040 1.035 1.012 1.000; 1875 1.062
//                             1.035 1.014 1.000
//         2560 / 1024 x 512   64 1.004 1.019 1.014 1.040; 187 1.000 1.053 1.004 1.016; 312 1.001 1.030 1.018 1.016; 469 1.000 1.021
//                             1.002 1.035
//         4096 / 1536 x 128   125 1.000 1.026 1.010 1.029; 375 1.000 1.033 1.012 1.033; 1000 1.014 1.029 1.000 1.038
//         7168 / 2048 x 256   64 1.015 1.058 1.019 1.045; 128 1.008 1.048 1.000 1.031; 250 1.010 1.050 1.000 1.042; 500 1.024 1.017
//          + shared           1.000 1.097; 937 1.037 1.009 1.000 1.111
//         1024 / 512 x 64     156 ss 1.051 sl 1.022 ll 1.060 pl 1.000 pp 1.003; 375 1.067 1.031 1.022 1.000 1.021; 1250 1.059 1.029
//                             1.035 1.000 1.007;  1536 / 512 x 128  156 1.030 1.030 1.117 1.018 1.000; 625 1.048 1.009 1.048 1.000 1.010
//         few tiles: 512 / 2048 x 8  R = 1125 ll 1.005 pl 1.038; 7500 1.018 1.015;  7168 / 512 x 8  1125 1.000 1.022; 2000 1.062 1.007
//   FP8   2048 / 768 x 128    69 sl 1.005 ll 1.019 pl 1.003 pp 1.007; 96 1.006 1.001 1.000 1.008; 156 1.082 1.156 1.062 1.000; 250 1.023
//                             1.043 1.017 1.000; 375 1.022 1.005 1.000 1.030; 1000 1.045 1.048 1.026 1.000; 1875 1.056 1.041 1.045 1.000
//         2560 / 1024 x 512   64 ss 1.017 sl 1.009 ps 1.010 pp 1.027; 125 1.004 1.030 1.015 1.023; 187 1.028 1.044 1.002 1.000; 312 1.008
//                             1.005 1.000 1.003; 469 1.026 1.025 1.000 1.001
//         4096 / 1536 x 128   125 ss 1.000 sp 1.002 ps 1.010 pp 1.015; 375 1.028 1.000 1.003 1.003; 1000 1.035 1.005 1.009 1.000
//         7168 / 2048 x 256   128 ss 1.000 sp 1.002 pp 1.021; 250 1.005 1.000 1.015; 500 1.000 1.002 1.030; 937 1.027 1.000 1.050; skewed
//          + shared           experts, 500 1.025 1.000 1.031
//         1024 / 512 x 64     156 ll 1.028 pl 1.010 pp 1.000; 375 1.000 1.014 1.028; 1250 1.012 1.012 1.012
//         2048 / 256 x 128    156 ps 1.000 pl 1.094 pp 1.000; 625 1.013 1.014 1.000
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
  if (fp8) return K < 896 ? over(128) : K < 1280 ? over(180) : over(256);
  if (K < 896) return K >= 640 && over(128);
  return K < 1280 ? over(350) : K < 1792 ? over(512) : over(96);
}

}  // namespace moe
