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

}  // namespace moe
