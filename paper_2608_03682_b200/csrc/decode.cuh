// Weight codes -> the bf16 operand image of the tensor core, in shared memory (the per-channel scale stays in the epilogue).
#pragma once

#include "common.cuh"

namespace phyai {

// Four e4m3 codes (one 32-bit word) -> two bf16 pairs, exactly, without the (slow-rate) conversion instructions.
// A code is S EEEE MMM (bias 7).  Its byte goes to the high byte of a 16-bit half (byte permute): the sign is then
// in place; the magnitude, moved down by four bits, puts EEEE into the low bits of bf16's exponent field and MMM
// at the top of its mantissa, i.e. the bf16 number 2^(E - 127) (1 + M/8) -- for E = 0 the bf16 subnormal
// 2^-126 (M/8).  One exact bf16x2 multiplication by 2^120 restores the bias: 2^(E - 7)(1 + M/8), and for E = 0
// 2^-6 (M/8), which is the value of e4m3's subnormals; zero stays zero.  (bf16 multiplication has no flush-to-zero
// mode: subnormal inputs are honoured.)  Five full-rate instructions per pair.
__device__ __forceinline__ void e4m3x4_to_bf16x4(uint32_t w, uint32_t& lo, uint32_t& hi) {
  uint32_t x0, x1;
  asm("prmt.b32 %0, %1, 0, 0x1404;" : "=r"(x0) : "r"(w));   // [b1 0 b0 0]
  asm("prmt.b32 %0, %1, 0, 0x3424;" : "=r"(x1) : "r"(w));   // [b3 0 b2 0]
  const uint32_t t0 = (x0 & 0x80008000u) | ((x0 >> 4) & 0x07F007F0u);
  const uint32_t t1 = (x1 & 0x80008000u) | ((x1 >> 4) & 0x07F007F0u);
  const uint32_t c = 0x7B807B80u;   // (2^120, 2^120)
  asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(lo) : "r"(t0), "r"(c));
  asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(hi) : "r"(t1), "r"(c));
}

// One warp: rows row0 .. row0 + 63 of a block of codes (64 per row: WB = 8, e4m3, 64 bytes; WB = 4, int4, 32 bytes: byte j =
// codes 2 j (low nibble) and 2 j + 1) at `codes` -> rows of 128 bytes of the swizzled K-major image at `image`.  A lane takes
// 16 codes of every eighth row and writes them as 32 bytes.  The codes may sit at the end of the image they expand into:
// they are read into registers first, then `sync` (every warp that decodes the block), then written.
template <int WB, class Sync>
__device__ __forceinline__ void decode_rows64(uint32_t codes, uint32_t image, int row0, int lane, Sync sync) {
  const int r0 = row0 + (lane >> 2), cq = lane & 3;
  if constexpr (WB == 8) {
    uint4 raw[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint32_t src = codes + (uint32_t)(r0 + 8 * j) * 64 + (uint32_t)cq * 16;
      asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(raw[j].x), "=r"(raw[j].y), "=r"(raw[j].z), "=r"(raw[j].w) : "r"(src) : "memory");
    }
    sync();
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int r = r0 + 8 * j;
      const uint32_t words[4] = {raw[j].x, raw[j].y, raw[j].z, raw[j].w};
#pragma unroll
      for (int c = 0; c < 2; ++c) {       // 16-byte chunk 2 cq + c of the row: 8 codes = words[2c], words[2c + 1]
        uint32_t o0, o1, o2, o3;
        e4m3x4_to_bf16x4(words[2 * c], o0, o1);
        e4m3x4_to_bf16x4(words[2 * c + 1], o2, o3);
        const uint32_t dst = image + (uint32_t)r * 128 + (uint32_t)((((2 * cq + c) ^ (r & 7))) << 4);
        asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(dst), "r"(o0), "r"(o1), "r"(o2), "r"(o3) : "memory");
      }
    }
  } else {
    // A nibble c becomes the bf16 number 128 + c by bit insertion (0x4300 | c: the unit of the mantissa at 128 is 1), and
    // one exact bf16x2 subtraction of 136 makes it c - 8.
    uint2 raw[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint32_t src = codes + (uint32_t)(r0 + 8 * j) * 32 + (uint32_t)cq * 8;
      asm volatile("ld.shared.v2.b32 {%0,%1}, [%2];" : "=r"(raw[j].x), "=r"(raw[j].y) : "r"(src) : "memory");
    }
    sync();
    auto pair = [](uint32_t byte) -> uint32_t {       // one byte -> (bf16(lo - 8), bf16(hi - 8))
      uint32_t w = 0x43004300u | (byte & 15u) | ((byte & 0xF0u) << 12), o;
      asm("sub.rn.bf16x2 %0, %1, %2;" : "=r"(o) : "r"(w), "r"(0x43084308u));
      return o;
    };
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int r = r0 + 8 * j;
      const uint32_t words[2] = {raw[j].x, raw[j].y};
#pragma unroll
      for (int c = 0; c < 2; ++c) {       // 16-byte chunk 2 cq + c: codes of bytes 4c .. 4c + 3 of my 8
        const uint32_t w4 = words[c];
        const uint32_t dst = image + (uint32_t)r * 128 + (uint32_t)((((2 * cq + c) ^ (r & 7))) << 4);
        asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(dst), "r"(pair(w4 & 0xFFu)), "r"(pair((w4 >> 8) & 0xFFu)),
                     "r"(pair((w4 >> 16) & 0xFFu)), "r"(pair(w4 >> 24))
                     : "memory");
      }
    }
  }
}

}  // namespace phyai
