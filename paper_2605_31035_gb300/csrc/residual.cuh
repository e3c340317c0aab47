// The residual E2M1 codes of E1M2 nibbles, shared by the few-row kernels.
#pragma once
#include <cstdint>

#include "ptx.cuh"

// One three-input logic instruction (truth-table byte from a = 0xF0, b = 0xCC,
// c = 0xAA).
#define MIXFP4_LOP3(d, a, b, c, LUT) asm("lop3.b32 %0, %1, %2, %3, " #LUT ";" : "=r"(d) : "r"(a), "r"(b), "r"(c))

namespace mixfp4 {

// Residual E2M1 codes of eight nibbles (sign in bit 3, payload p in bits
// 0-2): payload {0,1,2,3,4,4,4,2}[p] = p & F with F's bit 0 = ~p2, bit 1 =
// ~p2 | p0, bit 2 = ~(p1 & p0), and the sign kept.  Checked exhaustively on
// the host against the table.
__device__ __forceinline__ uint32_t residual_word(uint32_t w) {
  const uint32_t r1 = w >> 1, r2 = w >> 2, l1 = w << 1, l2 = w << 2;
  uint32_t a, b, c, d;
  MIXFP4_LOP3(a, 0x22222222u, r1, l1, 0xBF);        // ~K | ~r1 | l1
  MIXFP4_LOP3(b, 0x44444444u, l1, l2, 0x7F);        // ~K | ~(l1 & l2)
  MIXFP4_LOP3(c, w, a, b, 0x80);                    // w & a & b
  MIXFP4_LOP3(d, c, r2, 0x11111111u, 0x70);         // c & (~r2 | ~K)
  return d;
}

// Byte offset of row r's four ue4m3 scales of a K step in the tensor core's tiled
// layout of 128 rows.
__device__ __forceinline__ uint32_t tiled_scale_row(int r) { return (uint32_t)((r & 31) * 16 + (r >> 5) * 4); }

// All ones where block b (0..3) of the four scale bytes s4 is E1M2, else 0
// (prmt with the sign-replicate selectors).
__device__ __forceinline__ uint32_t type_mask(uint32_t s4, int b) {
  return prmt(s4, 0u, 0x8888u + 0x1111u * (uint32_t)b);
}

}  // namespace mixfp4
