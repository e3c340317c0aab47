// Decode of MixFP4 codes to f16 (Sec. 3.3, App. B.5): the value u * s8 with
// u = 2v has at most 7 significant bits and lies in [2^-9, 14 * 448], so it
// is exact in f16.  Shared by the GEMM kernels, the operand decode pass and
// the quantizer that writes the decoded operand directly.
#pragma once
#include <cstdint>

#include "ptx.cuh"

namespace mixfp4 {

__device__ __forceinline__ uint32_t hmul2(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("mul.rn.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}

// f16 high bytes of u = 2v by payload (the low byte of every such f16 is 0):
//   E2M1 u = {0,1,2,3,4,6,8,12} -> 00 3C 40 42 | 44 46 48 4A
//   E1M2 u = {0,2,4,...,14}     -> 00 40 44 46 | 48 49 4A 4B
constexpr uint32_t kLutE2M1Lo = 0x42403C00u, kLutE2M1Hi = 0x4A484644u;
constexpr uint32_t kLutE1M2Lo = 0x46444000u, kLutE1M2Hi = 0x4B4A4948u;

// Decode one 32-bit code word (8 elements, element 2j in the low nibble of
// byte j) of a block with f16x2 scale s2 into four f16x2 words, in the order
// (e0,e1) (e2,e3) (e4,e5) (e6,e7): byte LUT of the payloads (prmt), the
// nibble sign moved into bit 7 of each byte (prmt + lop3), bytes placed as f16
// high bytes (prmt), times s8 (exact).
__device__ __forceinline__ void decode8(uint32_t w, uint32_t lut_lo, uint32_t lut_hi, uint32_t s2,
                                        uint32_t* out) {
  const uint32_t wp = w & 0x77777777u;
  const uint32_t ws = w * 16u;
  const uint32_t u0 = prmt(lut_lo, lut_hi, wp);
  const uint32_t u1 = prmt(lut_lo, lut_hi, __umulhi(wp, 0x10000u));
  const uint32_t g0 = prmt(w, ws, 0x1504u);  // byte i bit 7 = sign of element i   (i = 0..3)
  const uint32_t g1 = prmt(w, ws, 0x3726u);  // byte i bit 7 = sign of element 4+i
  const uint32_t v0 = u0 | (g0 & 0x80808080u);
  const uint32_t v1 = u1 | (g1 & 0x80808080u);
  out[0] = hmul2(prmt(v0, 0u, 0x1404u), s2);
  out[1] = hmul2(prmt(v0, 0u, 0x3424u), s2);
  out[2] = hmul2(prmt(v1, 0u, 0x1404u), s2);
  out[3] = hmul2(prmt(v1, 0u, 0x3424u), s2);
}

// Decode 32 codes (one 16-byte chunk = two 16-element blocks) with their two
// scale bytes s2b into 16 f16x2 words in K order.
__device__ __forceinline__ void decode_chunk(const uint4& c, uint32_t s2b, uint32_t* out) {
  const uint32_t h01 = cvt_f16x2_from_e4m3x2((uint16_t)(s2b & 0x7F7Fu));
  const uint32_t sv[2] = {prmt(h01, 0u, 0x1010u), prmt(h01, 0u, 0x3232u)};
  const uint32_t w[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    const bool e1m2 = (s2b >> (8 * b + 7)) & 1u;
    const uint32_t lut_lo = e1m2 ? kLutE1M2Lo : kLutE2M1Lo;
    const uint32_t lut_hi = e1m2 ? kLutE1M2Hi : kLutE2M1Hi;
    decode8(w[2 * b], lut_lo, lut_hi, sv[b], out + 8 * b);
    decode8(w[2 * b + 1], lut_lo, lut_hi, sv[b], out + 8 * b + 4);
  }
}

}  // namespace mixfp4
