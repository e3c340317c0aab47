// Candidate-set and block-size quantize-dequantize (reading R14): Algorithm 1
// with the per-block MSE choice taken over any subset of four FP4 candidates
// -- E2M1 with largest value 6 (Algorithm 1's E2M1), E1M2 in x2 units, E2M1
// with the block max mapped to 4, and E3M0 (Eq. 1-2 with W_E = 3, W_M = 0:
// {0, 1/4, ..., 16}) -- and blocks of g = 8, 16, 32 or 64 elements.  These are
// the paper's ablations (Sec. 2.4 candidate sets, Sec. 4.3 Table 5 block
// sizes).  The stored MixFP4 format holds one type bit, so the kernel returns
// what the ablations measure: the dequantized tensor (fp32 or bf16) and each
// block's chosen candidate.
//
// One thread holds 16 consecutive elements of a row (one 32-byte load).  A
// g = 8 thread carries two blocks; a g = 32 / 64 block spans 2 / 4 adjacent
// lanes, which combine the block max and each candidate's error sum with xor
// shuffles (lane i with i ^ 1, then i ^ 2: the pairwise tree of the 16-element
// sums, the same on every lane because fp32 addition is commutative).  The
// divisions are the quantizer's (quant_core.cuh): x / s32, B / 6, B / 7 and
// |a| / s8 in the checked two-instruction form on packed pairs (x / s32 with
// Markstein's correction where the run-time check asks for it); B / 4 and
// B / 16 are exact scalings.  The E4M3 scale and the E2M1 codes come from the
// hardware conversions (round to nearest even, saturating), E1M2 from the
// 1.5 2^23 addition, E3M0 from the exponent and mantissa bits.  Bound by
// instruction issue, so candidates are compared and selected as packed payload
// words and only the chosen one is turned back into values (f16 by table, as in
// the GEMMs' decode), and dense tensors need no division to find a block.
// 8192 x 8192, bf16 out, scale given: {E2M1(6), E1M2} 90 -> 67 us, with E3M0
// 120 -> 102, all four 133 -> 113 (values kept in registers and a 64-bit
// division per block before).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cstdint>

#include "decode.cuh"
#include "host_util.cuh"
#include "kernels.cuh"
#include "ptx.cuh"
#include "quant_core.cuh"

namespace mixfp4 {
namespace {

constexpr int kFqThreads = 256;

// The candidates of a block part held by one thread (kPairs element pairs of
// |X_FP8|, t = {s8, 1/s8 as (zh, zl)}): the 3-bit payloads packed into words of
// eight (element i of a word at bits 4 i, the stored order) and the error sum.
// Payloads, not values, are kept per candidate: two words instead of sixteen
// registers to compare and select.  Each chain of errors runs over the even
// (odd) elements, as R5.
template <int kPairs>
__device__ __forceinline__ void cand_e2m1(const u64* a, const float4 t, uint32_t* pw, float& S) {
  const u64 zh8 = pack2(t.y, t.y), zl8 = pack2(t.z, t.z);
  const uint16_t ns8h = __half_as_ushort(__float2half_rn(-t.x));  // exact: E4M3 values are f16 values
  u64 acc = 0;
#pragma unroll
  for (int g = 0; g < kPairs / 4; ++g) {
    float ylo[4], yhi[4];
    uint32_t hq[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) unpack2(div_kd2(a[4 * g + i], zh8, zl8), ylo[i], yhi[i]);  // fl32(|a| / s8)
    pw[g] = e2m1_quad(ylo, yhi, hq);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float alo, ahi, dlo, dhi;
      unpack2(a[4 * g + i], alo, ahi);
      asm("{ .reg .f16 ql, qh; mov.b32 {ql, qh}, %2;\n"
          " fma.rn.f32.f16 %0, ql, %3, %4;\n fma.rn.f32.f16 %1, qh, %3, %5; }"
          : "=f"(dlo), "=f"(dhi) : "r"(hq[i]), "h"(ns8h), "f"(alo), "f"(ahi));
      const u64 d = pack2(dlo, dhi);
      acc = fma2(d, d, acc);
    }
  }
  float se, so;
  unpack2(acc, se, so);
  S = __fadd_rn(se, so);
}

template <int kPairs>
__device__ __forceinline__ void cand_e1m2(const u64* a, const float4 t, uint32_t* pw, float& S) {
  const u64 ns8 = pack2(-t.x, -t.x), zh8 = pack2(t.y, t.y), zl8 = pack2(t.z, t.z);
  const u64 magic = pack2(12582912.0f, 12582912.0f), nmagic = pack2(-12582912.0f, -12582912.0f);  // 1.5 * 2^23
  u64 acc = 0;
#pragma unroll
  for (int g = 0; g < kPairs / 4; ++g) {
    uint32_t pb[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const u64 tq = add2(div_kd2(a[4 * g + i], zh8, zl8), magic);  // RNE to an integer, saturated at 7
      const uint32_t tlo = min(lo32(tq), 0x4B400007u), thi = min(hi32(tq), 0x4B400007u);
      pb[i] = tlo + (thi << 4);
      const u64 d = fma2(add2(bits2(tlo, thi), nmagic), ns8, a[4 * g + i]);
      acc = fma2(d, d, acc);
    }
    pw[g] = pack_low_bytes(pb[0], pb[1], pb[2], pb[3]);
  }
  float se, so;
  unpack2(acc, se, so);
  S = __fadd_rn(se, so);
}

// E3M0 magnitude nearest to y >= 0: 0 or 2^e, e = -2..4, ties to the even
// payload.  The payload of 2^e is e + 3, so between 2^e and 2^(e+1) a tie
// (mantissa exactly 1.5) goes up iff the biased fp32 exponent of 2^e is odd:
// round up iff mantissa + (exponent bit 0) > 2^22, i.e. iff adding 2^22 - 1 and
// that bit carries into the exponent.  Then 16 caps the top; below 1/4 the
// neighbours are 0 and 1/4, with the tie 1/8 going to 0.
__device__ __forceinline__ uint32_t e3m0_bits(float y) {
  const uint32_t u = __float_as_uint(y);
  const uint32_t r = (u + 0x003FFFFFu + ((u >> 23) & 1u)) & 0x7F800000u;
  return y > 0.125f ? max(min(r, 0x41800000u), 0x3E800000u) : 0u;
}

template <int kPairs>
__device__ __forceinline__ void cand_e3m0(const u64* a, const float4 t, uint32_t* pw, float& S) {
  const u64 ns8 = pack2(-t.x, -t.x), zh8 = pack2(t.y, t.y), zl8 = pack2(t.z, t.z);
  u64 acc = 0;
#pragma unroll
  for (int g = 0; g < kPairs / 4; ++g) {
    uint32_t word = 0u;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float ylo, yhi;
      unpack2(div_kd2(a[4 * g + i], zh8, zl8), ylo, yhi);
      const uint32_t qlo = e3m0_bits(ylo), qhi = e3m0_bits(yhi);
      // Payload: biased exponent - 124 (1/4 -> 1, ..., 16 -> 7), 0 for zero.
      word += (uint32_t)max((int)(qlo >> 23) - 124, 0) << (8 * i);
      word += (uint32_t)max((int)(qhi >> 23) - 124, 0) << (8 * i + 4);
      const u64 d = fma2(bits2(qlo, qhi), ns8, a[4 * g + i]);  // |a| - q s8, the product exact
      acc = fma2(d, d, acc);
    }
    pw[g] = word;
  }
  float se, so;
  unpack2(acc, se, so);
  S = __fadd_rn(se, so);
}

// f16 high bytes of the values v by payload (the low bytes are 0), candidates
// E2M1, E1M2 and E3M0.
constexpr uint32_t kValE2M1Lo = 0x3E3C3800u, kValE2M1Hi = 0x46444240u;
constexpr uint32_t kValE1M2Lo = 0x42403C00u, kValE1M2Hi = 0x47464544u;
constexpr uint32_t kValE3M0Lo = 0x3C383400u, kValE3M0Hi = 0x4C484440u;

// pw: the chosen payloads of the thread's 16 elements; code: the scale code of
// each block (part) it holds.
template <int kG>
__device__ __forceinline__ void fake_quantize_unit(const u64 a[8], const TensorConsts& tc,
                                                   const float4* __restrict__ tab, int mask, uint32_t pw[2],
                                                   uint32_t code[2], int best_c[2]) {
  constexpr int kParts = kG == 8 ? 2 : 1;  // blocks per thread
  constexpr int kPairs = 8 / kParts;      // element pairs of a block held by one thread
  constexpr int kWords = kPairs / 4;
#pragma unroll
  for (int p = 0; p < kParts; ++p) {
    const u64* ap = a + p * kPairs;
    float B = 0.0f;
#pragma unroll
    for (int j = 0; j < kPairs; ++j) {
      float lo, hi;
      unpack2(ap[j], lo, hi);
      B = max3f(B, lo, hi);
    }
    if (kG >= 32) B = fmaxf(B, __shfl_xor_sync(0xffffffffu, B, 1));
    if (kG == 64) B = fmaxf(B, __shfl_xor_sync(0xffffffffu, B, 2));
    float best_S = 0.0f;
    best_c[p] = -1;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      if (!((mask >> c) & 1)) continue;  // uniform over the launch
      float bd;  // fl32(B / divisor): 6 and 7 by the checked two-instruction form, 4 and 16 exactly
      if (c == 0) bd = __fmaf_rn(B, tc.kd6.x, __fmul_rn(B, tc.kd6.y));
      else if (c == 1) bd = __fmaf_rn(B, tc.kd7.x, __fmul_rn(B, tc.kd7.y));
      else if (c == 2) bd = __fmul_rn(B, 0.25f);
      else bd = __fmul_rn(B, 0.0625f);
      const uint32_t sc = cvt_e4m3x2(0.0f, bd) & 0x7Fu;  // R2: E4M3 RNE, saturating
      const float4 t = tab[sc];
      uint32_t w[kWords];
      float S;
      if (c == 1) cand_e1m2<kPairs>(ap, t, w, S);
      else if (c == 3) cand_e3m0<kPairs>(ap, t, w, S);
      else cand_e2m1<kPairs>(ap, t, w, S);
      if (kG >= 32) S = __fadd_rn(S, __shfl_xor_sync(0xffffffffu, S, 1));
      if (kG == 64) S = __fadd_rn(S, __shfl_xor_sync(0xffffffffu, S, 2));
      if (best_c[p] < 0 || S <= best_S) {  // a later candidate wins a tie
        best_c[p] = c;
        best_S = S;
        code[p] = sc;
#pragma unroll
        for (int k = 0; k < kWords; ++k) pw[p * kWords + k] = w[k];
      }
    }
  }
  if (kParts == 1) {
    code[1] = code[0];
    best_c[1] = best_c[0];
  }
}

// kDense: rows of x and out follow one another without gaps.
template <int kG, bool kDense>
__global__ void __launch_bounds__(kFqThreads, 4)
fake_quantize_kernel(const uint16_t* x, int64_t rows, int64_t K, int64_t ldx, int mask,
                     float* tensor_scale, const uint32_t* amax_word, int scale_given, void* __restrict__ out,
                     int out_bf16, int64_t ldo, uint8_t* __restrict__ choice) {
  __shared__ float4 tab[128];  // E4M3 code -> {s8, zh, zl, 0}
  fill_scale_table(tab);
  griddep_wait();
  griddep_launch_dependents();
  const TensorConsts tc = tensor_consts(tensor_scale, amax_word, scale_given);
  const bool markstein = markstein_needed(tc);  // ends with a CTA barrier (tab is ready)
  const float s32 = tc.scaled ? scalbnf(tc.s32, -tc.k) : tc.s32;  // the tensor's own s32 (exact)
  const int lane = threadIdx.x & 31;
  const int64_t kb = K / 16, nsub = rows * kb;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  // Warp-uniform loop: the lanes of a g > 16 block shuffle together.
  for (int64_t base = warp * 32; base < nsub; base += nwarps * 32) {
    const int64_t b = base + lane;
    const bool live = b < nsub;
    const int64_t r = kDense || !live ? 0 : b / kb, j = kDense ? b : (live ? b - r * kb : 0);  // dense: one long row
    uint32_t w[8];
    if (live) {
      ldg256_stream(x + r * ldx + j * 16, w);
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) w[i] = 0u;
    }
    int best_c[2] = {0, 0};
    uint32_t pw[2] = {0u, 0u}, code[2] = {0u, 0u};
    u64 a[8];  // |X_FP8| pairs (R1, R7)
    if (tc.scaled) x_fp8_magnitudes<true, true>(w, tc, a);
    else if (markstein) x_fp8_magnitudes<false, true>(w, tc, a);
    else x_fp8_magnitudes<false, false>(w, tc, a);
    const uint32_t sg[2] = {sign_bits(w[0], w[1], w[2], w[3]), sign_bits(w[4], w[5], w[6], w[7])};
    fake_quantize_unit<kG>(a, tc, tab, mask, pw, code, best_c);
    if (live) {
      // sign(x) fl32(v s8 s32): v s8 is exact in f16, one rounding in fp32.
      const u64 s32s = pack2(s32, s32);
      uint32_t ow[16];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c = best_c[h];
        const uint32_t lut_lo = c == 1 ? kValE1M2Lo : (c == 3 ? kValE3M0Lo : kValE2M1Lo);
        const uint32_t lut_hi = c == 1 ? kValE1M2Hi : (c == 3 ? kValE3M0Hi : kValE2M1Hi);
        const uint32_t s2 = prmt(cvt_f16x2_from_e4m3x2((uint16_t)code[h]), 0u, 0x1010u);
        uint32_t f[4];
        decode8(pw[h] | sg[h], lut_lo, lut_hi, s2, f);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          float lo, hi;
          f16x2_to_f32(f[i], lo, hi);
          const u64 v = mul2(pack2(lo, hi), s32s);
          ow[8 * h + 2 * i] = lo32(v);
          ow[8 * h + 2 * i + 1] = hi32(v);
        }
      }
      if (out_bf16) {
        uint32_t hw[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(ow[2 * i]), __uint_as_float(ow[2 * i + 1]));
          hw[i] = *reinterpret_cast<const uint32_t*>(&h);  // low half: element 2i
        }
        stg256(static_cast<uint16_t*>(out) + r * ldo + j * 16, hw);
      } else {
        float* dst = static_cast<float*>(out) + r * ldo + j * 16;
        stg256(dst, ow);
        stg256(dst + 8, ow + 8);
      }
      if (choice) {
        constexpr int kLanes = kG >= 16 ? kG / 16 : 1;  // lanes sharing one block
        if constexpr (kG == 8) {
          *reinterpret_cast<uint16_t*>(choice + 2 * b) = (uint16_t)(best_c[0] | (best_c[1] << 8));
        } else if ((lane & (kLanes - 1)) == 0) {
          choice[b / kLanes] = (uint8_t)best_c[0];
        }
      }
    }
  }
}

}  // namespace

int launch_fake_quantize(const uint16_t* x, int64_t rows, int64_t K, int64_t ldx, int candidates, int block,
                         float* tensor_scale, const uint32_t* amax_word, int scale_given, void* out, int out_bf16,
                         int64_t ldo, uint8_t* choice, cudaStream_t stream) {
  const int64_t nsub = rows * (K / 16);
  if (nsub == 0) return 0;
  int64_t grid = (nsub + kFqThreads - 1) / kFqThreads;
  if (grid > num_sms() * 8) grid = num_sms() * 8;
  cudaError_t e;
#define MIXFP4_LAUNCH_FQ(G)                                                                                  \
  e = ldx == K && ldo == K                                                                                    \
          ? launch_pdl(fake_quantize_kernel<G, true>, (unsigned)grid, kFqThreads, 0, stream, x, rows, K, ldx,   \
                       candidates, tensor_scale, amax_word, scale_given, out, out_bf16, ldo, choice)            \
          : launch_pdl(fake_quantize_kernel<G, false>, (unsigned)grid, kFqThreads, 0, stream, x, rows, K, ldx,  \
                       candidates, tensor_scale, amax_word, scale_given, out, out_bf16, ldo, choice)
  switch (block) {
    case 8: MIXFP4_LAUNCH_FQ(8); break;
    case 16: MIXFP4_LAUNCH_FQ(16); break;
    case 32: MIXFP4_LAUNCH_FQ(32); break;
    default: MIXFP4_LAUNCH_FQ(64); break;
  }
#undef MIXFP4_LAUNCH_FQ
  return e == cudaSuccess ? 0 : -1;
}

}  // namespace mixfp4
