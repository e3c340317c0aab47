// MixFP4 online quantizer (Algorithm 1, Sec. 3.2), tensor amax, and decoder
// (App. B.2/B.3) for sm_103a.
//
// Design (HBM-bound, 2.5625 algorithmic bytes per element):
//   * one thread owns one 16-element block at a time: a single 256-bit
//     coalesced load (a warp reads 1 KiB of contiguous bf16), one 64-bit code
//     store and one scale-byte store (a warp writes 256 B and 32 B
//     contiguous); each thread quantizes two such blocks side by side;
//   * all per-element fp32 work runs on packed f32x2 instructions;
//   * every division of Algorithm 1 (x/s32, B/6, B/7, |a|/s8) is evaluated as
//     IEEE round-to-nearest with a divisor known in advance, in two packed
//     instructions (N. Brisebarre, J.-M. Muller, S. K. Raina, "Accelerating
//     correctly rounded floating-point division when the divisor is known in
//     advance", IEEE Trans. Computers 53(8), 2004):
//         q = RN(a*zh + RN(a*zl)),  zh = RN(1/b),  zl = RN(RN(1 - b*zh)/b).
//     This is not correctly rounded for every divisor, so each use is covered
//     by a check: exhaustive on the host for the divisors 6, 7 and every E4M3
//     value (every fp32 significand of a), and, for x/s32, at run time in the
//     kernel over all 128 bf16 significands of x (2 of the 2^23 fp32
//     significands of s32 fail; those tensors use Markstein's correction,
//     P. Markstein 1990; Muller et al., Handbook of Floating-Point Arithmetic,
//     Sec. 4.9:  q0 = RN(a*r), e = RN(a - q0*b) (exact via fma),
//     q = RN(q0 + e*r), r = RN(1/b)).  Both return RN(a/b) whenever a >=
//     2^-102 and the quotient is normal; smaller numerators only occur where
//     their exact value cannot change a code or an error sum (see the
//     tiny-value note in quantize_block), and tensors whose s32 lies outside
//     [2^-20, 2^100] are first rescaled by an exact power of two;
//   * E2M1 rounding uses cvt.rn.satfinite.e2m1x2 (RNE, saturating) and E4M3
//     scale rounding cvt.rn.satfinite.e4m3x2; E1M2 rounding adds 1.5*2^23
//     (RNE to an integer) and clamps the integer to 7.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <cstdint>

#include "decode.cuh"
#include "host_util.cuh"
#include "kernels.cuh"
#include "ptx.cuh"
#include "quant_core.cuh"
#include "residual.cuh"
#include "sm100.cuh"

namespace mixfp4 {

namespace {

// Where a quantized block goes: its 8 code bytes and scale byte, or (kF16) the
// 16 decoded f16 values u * s8 of the GEMM that takes a decoded operand.
template <bool kF16>
__device__ __forceinline__ void store_block(uint8_t* __restrict__ codes, uint8_t* __restrict__ scales, int64_t b,
                                            uint32_t lo, uint32_t hi, uint32_t sb) {
  if (kF16) {
    const uint32_t h = cvt_f16x2_from_e4m3x2((uint16_t)(sb & 0x7Fu));
    const uint32_t s2 = prmt(h, 0u, 0x1010u);
    const bool e1m2 = (sb & 0x80u) != 0;
    const uint32_t lut_lo = e1m2 ? kLutE1M2Lo : kLutE2M1Lo, lut_hi = e1m2 ? kLutE1M2Hi : kLutE2M1Hi;
    uint32_t o[8];
    decode8(lo, lut_lo, lut_hi, s2, o);
    decode8(hi, lut_lo, lut_hi, s2, o + 4);
    stg256(codes + b * 32, o);
  } else {
    stg64(codes + b * 8, lo, hi);
    scales[b] = (uint8_t)sb;
  }
}

// Persistent grid: each thread walks blocks b, b + nthr, b + 2 nthr, ... two
// at a time (a, b): both blocks of a pair are quantized before either is
// stored, so their independent dependency chains interleave, and the loads of
// the next pair are in flight meanwhile.  The division method is fixed per
// launch, so each method gets its own copy of the loop; the usual one runs on
// 32-bit block indices where they suffice (2^28 elements 177 -> 170 us: the
// kernel is bound by instruction issue, and 64-bit index arithmetic was one
// instruction in thirty).
template <int kMode, bool kContig, bool kF16, bool kScaled, bool kMarkstein, typename Index>
__device__ __forceinline__ void quantize_pairs(const uint16_t* x, Index b, Index nthr,
                                               Index nblocks, int64_t kblocks, int64_t ldx,
                                               uint8_t* __restrict__ codes, uint8_t* __restrict__ scales,
                                               const TensorConsts& tc, const float4* __restrict__ tab,
                                               uint32_t (&wa)[8], uint32_t (&wb)[8]) {
  for (; b < nblocks; b += 2 * nthr) {
    const Index b1 = b + nthr;
    uint32_t lo0, hi0, sb0, lo1, hi1, sb1;
    quantize_block<kMode, kScaled, kMarkstein>(wa, tc, tab, lo0, hi0, sb0);
    quantize_block<kMode, kScaled, kMarkstein>(wb, tc, tab, lo1, hi1, sb1);  // wb past the end: unused
    store_block<kF16>(codes, scales, b, lo0, hi0, sb0);
    if (b + 2 * nthr < nblocks) ldg256_stream(block_src<kContig>(x, b + 2 * nthr, kblocks, ldx), wa);
    if (b1 < nblocks) {
      store_block<kF16>(codes, scales, b1, lo1, hi1, sb1);
      if (b1 + 2 * nthr < nblocks) ldg256_stream(block_src<kContig>(x, b1 + 2 * nthr, kblocks, ldx), wb);
    }
  }
}

// The first loads are issued before any set-up work.
template <int kMode, bool kContig, bool kF16>
__global__ void __launch_bounds__(kQuantThreads, 4)
quantize_kernel(const uint16_t* x, int64_t nblocks, int64_t kblocks, int64_t ldx,
                uint8_t* __restrict__ codes, uint8_t* __restrict__ scales, float* tensor_scale,
                const uint32_t* amax_word, int amax_parts, int scale_given, int after_amax) {
  __shared__ float4 tab[128];  // E4M3 code -> {s8, zh, zl, 0} (zh, zl: see div_kd2)
  // Launched as a programmatic dependent of the amax kernel (after_amax), x
  // is already complete and may be read before that kernel finishes; only
  // the amax word must wait.  Otherwise wait before touching any input.
  if (!after_amax) griddep_wait();
  griddep_launch_dependents();
  const int64_t nthr = (int64_t)gridDim.x * kQuantThreads;
  const int64_t b = (int64_t)blockIdx.x * kQuantThreads + threadIdx.x;
  uint32_t wa[8], wb[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) wb[j] = 0u;  // defined values for a missing second block
  if (b < nblocks) ldg256_stream(block_src<kContig>(x, b, kblocks, ldx), wa);
  if (b + nthr < nblocks) ldg256_stream(block_src<kContig>(x, b + nthr, kblocks, ldx), wb);
  fill_scale_table(tab);
  if (after_amax) griddep_wait();
  if (kF16) {
    // The amax pass's maxima, one per CTA of it.
    __shared__ uint32_t red[kQuantThreads / 32];
    uint32_t m = 0u;
    for (int i = threadIdx.x; i < amax_parts; i += kQuantThreads) m = max(m, amax_word[i]);
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kQuantThreads / 32; ++i) m = max(m, red[i]);
    __syncthreads();
    if (threadIdx.x == 0) red[0] = m;
    __syncthreads();
    amax_word = red;
  }
  const TensorConsts tc = tensor_consts(tensor_scale, amax_word, scale_given);
  const bool markstein = markstein_needed(tc);
  if (tc.scaled)
    quantize_pairs<kMode, kContig, kF16, true, true, int64_t>(x, b, nthr, nblocks, kblocks, ldx, codes, scales, tc, tab, wa, wb);
  else if (markstein)
    quantize_pairs<kMode, kContig, kF16, false, true, int64_t>(x, b, nthr, nblocks, kblocks, ldx, codes, scales, tc, tab, wa, wb);
  else if (nblocks < (1ll << 30))
    quantize_pairs<kMode, kContig, kF16, false, false, uint32_t>(x, (uint32_t)b, (uint32_t)nthr, (uint32_t)nblocks, kblocks, ldx, codes, scales, tc, tab, wa, wb);
  else
    quantize_pairs<kMode, kContig, kF16, false, false, int64_t>(x, b, nthr, nblocks, kblocks, ldx, codes, scales, tc, tab, wa, wb);
}

// Small tensors in one launch: a cluster of eight CTAs holds the whole tensor in
// registers (up to kSmallPer blocks per thread), the CTAs exchange their maxima
// through distributed shared memory, and every thread quantizes the blocks it
// holds.  Such a call is launches and latency, not work: memset, amax_kernel and
// quantize_kernel took 9 us of GPU time and three launches on 16 x 8192.
//   kOut 0: codes and block scales; 1: the activation operand of the few-row
//   GEMM (xr main rows, xr residual rows, scales in the tiled layout), rows from
//   `rows` to xr as zeros.
constexpr int kSmallCtas = 8, kSmallThreads = 512, kSmallPer = 4;

template <int kMode, bool kContig, int kOut>
__global__ void __cluster_dims__(kSmallCtas, 1, 1) __launch_bounds__(kSmallThreads, 1)
quantize_small_kernel(const uint16_t* x, int64_t nblocks, int64_t kblocks, int64_t ldx,
                      uint8_t* __restrict__ codes, uint8_t* __restrict__ scales, float* tensor_scale, int xr) {
  __shared__ float4 tab[128];
  __shared__ uint32_t red[kSmallThreads / 32], maxes[kSmallCtas], amax;
  sm100::cluster_arrive();  // awaited before the first store into another CTA
  griddep_wait();
  griddep_launch_dependents();
  const int64_t b0 = (int64_t)blockIdx.x * kSmallThreads + threadIdx.x;
  constexpr int64_t kStride = (int64_t)kSmallCtas * kSmallThreads;
  const int64_t ntotal = kOut == 1 ? xr * kblocks : nblocks;
  uint32_t w[kSmallPer][8], m = 0u;
#pragma unroll
  for (int i = 0; i < kSmallPer; ++i) {
    const int64_t b = b0 + i * kStride;
#pragma unroll
    for (int j = 0; j < 8; ++j) w[i][j] = 0u;
    if (b < nblocks) ldg256_stream(block_src<kContig>(x, b, kblocks, ldx), w[i]);
  }
  fill_scale_table(tab);
#pragma unroll
  for (int i = 0; i < kSmallPer; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) m = __vmaxu2(m, w[i][j] & 0x7FFF7FFFu);
  m = max(m & 0xFFFFu, m >> 16);
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  // The CTAs of a cluster are scheduled together, but only a cluster barrier says
  // that the others have started; a store into one that has not is undefined.
  sm100::cluster_wait();
  if (threadIdx.x < 32) {
    m = __reduce_max_sync(0xffffffffu, threadIdx.x < kSmallThreads / 32 ? red[threadIdx.x] : 0u);
    if (threadIdx.x < kSmallCtas)
      sm100::st_cluster_u32(sm100::mapa_shared(sm100::smem_u32(&maxes[blockIdx.x % kSmallCtas]), threadIdx.x), m);
  }
  sm100::cluster_sync();
  if (threadIdx.x == 0) {
    for (int i = 0; i < kSmallCtas; ++i) m = max(m, maxes[i]);
    amax = m << 16;
  }
  __syncthreads();
  const TensorConsts tc = tensor_consts(tensor_scale, &amax, 0);
  const bool markstein = markstein_needed(tc);
#pragma unroll
  for (int i = 0; i < kSmallPer; ++i) {
    const int64_t b = b0 + i * kStride;
    if (b >= ntotal) break;
    uint32_t lo, hi, sb;
    if (tc.scaled) quantize_block<kMode, true, true>(w[i], tc, tab, lo, hi, sb);
    else if (markstein) quantize_block<kMode, false, true>(w[i], tc, tab, lo, hi, sb);
    else quantize_block<kMode, false, false>(w[i], tc, tab, lo, hi, sb);
    if (kOut == 0) {
      stg64(codes + b * 8, lo, hi);
      scales[b] = (uint8_t)sb;
    } else {
      const int r = (int)(b / kblocks), c = (int)(b - (int64_t)r * kblocks);
      if (b >= nblocks) lo = hi = sb = 0u;
      const uint32_t e1m2 = (sb & 0x80u) ? 0xFFFFFFFFu : 0u;
      stg64(codes + b * 8, lo, hi);
      stg64(codes + (xr * kblocks + b) * 8, residual_word(lo) & e1m2, residual_word(hi) & e1m2);
      uint8_t* t = scales + (int64_t)(c / 4) * 512 + (c & 3);
      t[tiled_scale_row(r)] = (uint8_t)(sb & 0x7Fu);
      t[tiled_scale_row(xr + r)] = (uint8_t)(sb & 0x7Fu);
    }
  }
}

template <int kMode, bool kContig, typename Index>
__device__ __forceinline__ void rht_pairs(const uint16_t* x, Index b, Index nthr, Index nblocks,
                                          int64_t kblocks, int64_t ldx, uint8_t* __restrict__ codes,
                                          uint8_t* __restrict__ scales, const TensorConsts& tc,
                                          const float4* __restrict__ tab, const uint32_t (&sw)[8], int lane,
                                          uint32_t (&w)[8], uint32_t (&w2)[8]) {
  for (; b < nblocks; b += 2 * nthr) {
    const Index b1 = b + nthr;
    u64 y[8], y2[8];
    rht_rotate(w, sw, lane, y);
    rht_rotate(w2, sw, lane, y2);  // the 8 lanes of a chunk agree on b1 < nblocks
    if (b + 2 * nthr < nblocks) ldg256_stream(block_src<kContig>(x, b + 2 * nthr, kblocks, ldx), w);
    if (b1 + 2 * nthr < nblocks) ldg256_stream(block_src<kContig>(x, b1 + 2 * nthr, kblocks, ldx), w2);
    uint32_t lo, hi, sb, lo2, hi2, sb2;
    if (tc.scaled) {
      rht_block<kMode, true>(y, tc, tab, lo, hi, sb);
      rht_block<kMode, true>(y2, tc, tab, lo2, hi2, sb2);
    } else {
      rht_block<kMode, false>(y, tc, tab, lo, hi, sb);
      rht_block<kMode, false>(y2, tc, tab, lo2, hi2, sb2);
    }
    stg64(codes + (int64_t)b * 8, lo, hi);
    scales[b] = (uint8_t)sb;
    if (b1 < nblocks) {
      stg64(codes + (int64_t)b1 * 8, lo2, hi2);
      scales[b1] = (uint8_t)sb2;
    }
  }
}

// Rotation + Algorithm 1, two blocks per thread side by side (as in
// quantize_kernel); the rotated pairs take 2 CTAs per SM of registers.
template <int kMode, bool kContig>
__global__ void __launch_bounds__(kQuantThreads, 2)
rht_quantize_kernel(const uint16_t* x, int64_t nblocks, int64_t kblocks, int64_t ldx,
                    const uint8_t* signs, uint8_t* __restrict__ codes, uint8_t* __restrict__ scales,
                    float* tensor_scale, const uint32_t* amax_word, int scale_given, int after_amax) {
  __shared__ float4 tab[128];
  if (!after_amax) griddep_wait();
  griddep_launch_dependents();
  const int lane = threadIdx.x & 31;
  const int64_t nthr = (int64_t)gridDim.x * kQuantThreads;
  int64_t b = (int64_t)blockIdx.x * kQuantThreads + threadIdx.x;
  uint32_t w[8], w2[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) w2[j] = 0u;
  if (b < nblocks) ldg256_stream(block_src<kContig>(x, b, kblocks, ldx), w);
  if (b + nthr < nblocks) ldg256_stream(block_src<kContig>(x, b + nthr, kblocks, ldx), w2);
  if (threadIdx.x < 128) {
    float s8 = 0.0f, unused;
    if (threadIdx.x < 0x7F) f16x2_to_f32(cvt_f16x2_from_e4m3x2((uint16_t)threadIdx.x), s8, unused);
    const float2 kd = kd_consts(s8);
    tab[threadIdx.x] = make_float4(s8, kd.x, kd.y, 0.0f);
  }
  uint32_t sw[8];
  rht_sign_words(signs, lane, sw);
  if (after_amax) griddep_wait();
  const TensorConsts tc = tensor_consts(tensor_scale, amax_word, scale_given);
  __syncthreads();
  if (nblocks < (1ll << 30))
    rht_pairs<kMode, kContig, uint32_t>(x, (uint32_t)b, (uint32_t)nthr, (uint32_t)nblocks, kblocks, ldx, codes, scales, tc,
                                        tab, sw, lane, w, w2);
  else
    rht_pairs<kMode, kContig, int64_t>(x, b, nthr, nblocks, kblocks, ldx, codes, scales, tc, tab, sw, lane, w, w2);
}

// max |y| of the rotated tensor as the bit pattern of a non-negative fp32.
template <bool kContig>
__global__ void __launch_bounds__(256)
rht_amax_kernel(const uint16_t* x, int64_t nblocks, int64_t kblocks, int64_t ldx,
                const uint8_t* signs, uint32_t* amax_word) {
  griddep_launch_dependents();
  const int lane = threadIdx.x & 31;
  uint32_t sw[8];
  rht_sign_words(signs, lane, sw);
  uint32_t m = 0;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  uint32_t w[8];
  if (b < nblocks) ldg256_stream(block_src<kContig>(x, b, kblocks, ldx), w);
  for (; b < nblocks; b += stride) {
    uint32_t wn[8];  // the next block's load is in flight during this block's rotation
    if (b + stride < nblocks) ldg256_stream(block_src<kContig>(x, b + stride, kblocks, ldx), wn);
    u64 y[8];
    rht_rotate(w, sw, lane, y);
#pragma unroll
    for (int j = 0; j < 8; ++j) m = max(m, max(lo32(y[j]) & 0x7FFFFFFFu, hi32(y[j]) & 0x7FFFFFFFu));
#pragma unroll
    for (int j = 0; j < 8; ++j) w[j] = wn[j];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  __shared__ uint32_t red[8];
  if (lane == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < (int)(blockDim.x >> 5); ++i) m = max(m, red[i]);
    griddep_wait();  // the word is zeroed by then
    if (m) atomicMax(amax_word, m);
  }
}

__global__ void __launch_bounds__(256)
zero_rows_kernel(float* __restrict__ C, int64_t n, int64_t per_row, int64_t cols, int64_t ldc, int vec) {
  griddep_wait();
  griddep_launch_dependents();
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = i / per_row, c = (i - r * per_row) * (vec ? 4 : 1);
    float* dst = C + r * ldc + c;
    if (vec && c + 4 <= cols) {
      *reinterpret_cast<float4*>(dst) = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    } else {
      for (int64_t k = 0; k < (vec ? cols - c : 1); ++k) dst[k] = 0.0f;
    }
  }
}

// max |x| over the tensor as the bit pattern of a non-negative fp32 (bf16
// magnitudes order like unsigned 16-bit integers).  Each thread keeps four
// 32-byte loads in flight: a register set is loaded again as soon as it has been
// looked at (a set past the end keeps its old values, which change no maximum).
// The tensor is read from its end: the pass that follows starts at the front and
// finds what was read last in L2 (both passes of 8192 x 8192: 69.6 us forward,
// 63.3; 65536 x 4096: 254, 245; no gain for the rotated passes, which arithmetic
// bounds).  Three CTAs per SM of this loop against eight of batches of four
// loads, with the kernel below in place of the memset: 4096 x 4096 21.1 -> 17.6,
// 1024 x 4096 10.4 -> 7.4.  Four CTAs per SM: 18.4 (spills); two: 17.5 and 64.4.
constexpr int kAmaxUnroll = 4, kAmaxCtas = 3;

// The word is zeroed once everything before is complete; the dependents (the
// maximum passes) therefore read their tensor without waiting, and wait only
// before they touch the word.  As a memset it and its gaps cost 3.3 us a call.
__global__ void zero_word_kernel(uint32_t* word) {
  griddep_wait();
  griddep_launch_dependents();
  if (threadIdx.x == 0) *word = 0u;
}

template <bool kContig>
__device__ __forceinline__ const uint16_t* amax_src(const uint16_t* x, int64_t b, int64_t kblocks, int64_t ldx) {
  if (kContig) return x + b * 16;
  const int64_t row = b / kblocks;
  return x + row * ldx + (b - row * kblocks) * 16;
}

// kParts: each CTA leaves its maximum in amax_word[blockIdx.x] for the quantize
// kernel to reduce, so nothing has to be zeroed first (a memset and its gaps
// are about 2.5 us of a call).
template <bool kContig, bool kParts>
__global__ void __launch_bounds__(256, kAmaxCtas)
amax_kernel(const uint16_t* x, int64_t nblocks, int64_t kblocks, int64_t ldx,
            uint32_t* amax_word) {
  if (kParts) griddep_wait();
  uint32_t m = 0;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  uint32_t w[kAmaxUnroll][8];
#pragma unroll
  for (int u = 0; u < kAmaxUnroll; ++u) {
#pragma unroll
    for (int j = 0; j < 8; ++j) w[u][j] = 0u;
    if (b + u * stride < nblocks) ldg256_stream(amax_src<kContig>(x, nblocks - 1 - b - u * stride, kblocks, ldx), w[u]);
  }
  for (; b < nblocks; b += kAmaxUnroll * stride)
#pragma unroll
    for (int u = 0; u < kAmaxUnroll; ++u) {
#pragma unroll
      for (int j = 0; j < 8; ++j) m = __vmaxu2(m, w[u][j] & 0x7FFF7FFFu);
      const int64_t next = b + (kAmaxUnroll + u) * stride;
      if (next < nblocks) ldg256_stream(amax_src<kContig>(x, nblocks - 1 - next, kblocks, ldx), w[u]);
    }
  m = max(m & 0xFFFFu, m >> 16);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  __shared__ uint32_t red[8];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < (int)(blockDim.x >> 5); ++i) m = max(m, red[i]);
    if (kParts) {
      amax_word[blockIdx.x] = m << 16;
    } else {
      griddep_wait();  // the word is zeroed by then
      if (m) atomicMax(amax_word, m << 16);
    }
  }
  // The second pass may start once every CTA got here.  (From the start its CTAs
  // took the SMs this pass left free and spread badly: stochastic rounding of
  // 1024 x 4096 13.9 -> 16.0 us.)
  griddep_launch_dependents();
}

// out = fl32(sign * v * s8 * s32): v * s8 is exact in fp32, one rounding.
__global__ void __launch_bounds__(256)
dequantize_kernel(const uint8_t* __restrict__ codes, const uint8_t* __restrict__ scales,
                  const float* tensor_scale, int64_t nblocks, float* __restrict__ out) {
  const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= nblocks) return;
  const float s32 = *tensor_scale;
  const uint2 c = *reinterpret_cast<const uint2*>(codes + b * 8);
  const uint32_t s = scales[b];
  float s8, unused;
  f16x2_to_f32(cvt_f16x2_from_e4m3x2((uint16_t)(s & 0x7Fu)), s8, unused);
  const bool e1m2 = (s >> 7) != 0;
  uint32_t o[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const uint32_t word = i < 8 ? c.x : c.y;
    const uint32_t nib = (word >> (4 * (i & 7))) & 0xFu;
    const uint32_t p = nib & 7u;
    float vv;
    if (e1m2) {
      vv = (float)p;  // x2 remapped E1M2: the payload as an integer
    } else {
      // E2M1 {0, .5, 1, 1.5, 2, 3, 4, 6}: (1 + m/2) * 2^(e-1), subnormal m/2.
      const uint32_t e = p >> 1, m = p & 1u;
      vv = e ? ldexpf(1.0f + 0.5f * (float)m, (int)e - 1) : 0.5f * (float)m;
    }
    float val = __fmul_rn(__fmul_rn(vv, s8), s32);
    o[i] = __float_as_uint(val) ^ ((nib & 8u) << 28);
  }
  stg256(out + b * 16, o);
  stg256(out + b * 16 + 8, o + 8);
}

}  // namespace

// Zero the word a maximum is taken into, by a kernel instead of a memset: the
// pass over the tensor is its programmatic dependent and overlaps it.
int launch_zero_word(uint32_t* word, cudaStream_t stream) {
  return launch_pdl(zero_word_kernel, 1, 32, 0, stream, word) == cudaSuccess ? 0 : -1;
}

// Zero `rows` rows of `cols` floats (row stride ldc), for a GEMM that adds parts
// into them.  Like launch_zero_word it waits for all before, so the GEMM (its
// programmatic dependent) may load its operands meanwhile and waits only before it
// touches C.  Against a memset: native GEMM 1536 x 4096 x 4096 47.2 -> 45.1 us, 4096^3
// 86.2 -> 81.9, GEMM with A decoded beforehand 2560 x 4096 x 4096 59.6 -> 57.4.
int launch_zero_rows(float* C, int64_t rows, int64_t cols, int64_t ldc, cudaStream_t stream) {
  if (ldc == cols) {  // one long row
    cols *= rows;
    rows = 1;
  }
  const bool vec = (reinterpret_cast<uintptr_t>(C) & 15) == 0 && (rows == 1 || (ldc & 3) == 0);
  const int64_t per_row = vec ? (cols + 3) / 4 : cols, n = rows * per_row;
  int64_t grid = (n + 255) / 256;
  if (grid > num_sms() * 4) grid = num_sms() * 4;
  return launch_pdl(zero_rows_kernel, (unsigned)grid, 256, 0, stream, C, n, per_row, cols, ldc, vec ? 1 : 0) == cudaSuccess
             ? 0
             : -1;
}

// The resident CTAs, or, above 2^23 blocks (268 MB), more than fit at once: over
// such a length the CTAs drift apart and the late ones end alone (tensor out of
// L2, both passes: 65536 x 4096 267 us against 263; 32768 x 4096 140 both ways;
// 8192 x 4096 42 against 44).
static int64_t amax_grid(int64_t nblocks) {
  const int64_t grid = (nblocks + 256 * kAmaxUnroll - 1) / (256 * kAmaxUnroll);
  const int64_t cap = num_sms() * (nblocks > (1 << 23) ? 8 : kAmaxCtas);
  return grid < cap ? grid : cap;
}

int launch_amax(const uint16_t* x, int64_t rows, int64_t K, int64_t ldx, uint32_t* amax_word,
                cudaStream_t stream) {
  const int64_t kblocks = K / 16, nblocks = rows * kblocks;
  if (nblocks == 0) return 0;
  launch_zero_word(amax_word, stream);
  const unsigned grid = (unsigned)amax_grid(nblocks);
  if (ldx == K) launch_pdl(amax_kernel<true, false>, grid, 256, 0, stream, x, nblocks, kblocks, ldx, amax_word);
  else launch_pdl(amax_kernel<false, false>, grid, 256, 0, stream, x, nblocks, kblocks, ldx, amax_word);
  return 0;
}

// Maxima of `*n` parts of the tensor into parts[0 .. *n) (*n <= kMaxAmaxParts).
static void launch_amax_parts(const uint16_t* x, int64_t rows, int64_t K, int64_t ldx, uint32_t* parts, int* n,
                              cudaStream_t stream) {
  const int64_t kblocks = K / 16, nblocks = rows * kblocks;
  int64_t grid = amax_grid(nblocks);
  if (grid > kMaxAmaxParts) grid = kMaxAmaxParts;
  *n = (int)grid;
  if (ldx == K) launch_pdl(amax_kernel<true, true>, (unsigned)grid, 256, 0, stream, x, nblocks, kblocks, ldx, parts);
  else launch_pdl(amax_kernel<false, true>, (unsigned)grid, 256, 0, stream, x, nblocks, kblocks, ldx, parts);
}

namespace {

template <bool kF16>
void launch_quantize_to(const uint16_t* x, int64_t rows, int64_t K, int64_t ldx, uint8_t* codes, uint8_t* scales,
                        float* tensor_scale, const uint32_t* amax_word, int amax_parts, int mode, int scale_given,
                        cudaStream_t stream) {
  const int64_t kblocks = K / 16, nblocks = rows * kblocks;
  // Persistent grid: 4 CTAs per SM of the device, fewer for small tensors
  // (each thread takes at least two blocks).
  int64_t grid = (nblocks + 2 * kQuantThreads - 1) / (2 * kQuantThreads);
  if (grid > num_sms() * 4) grid = num_sms() * 4;
  if (grid == 0) return;
  // Launched as a programmatic dependent: it overlaps its launch with the tail
  // of the kernel before it (see the waits at the top of quantize_kernel).
  const int after_amax = !scale_given;
#define MIXFP4_LAUNCH_Q(MODE)                                                                             \
  do {                                                                                                    \
    if (ldx == K)                                                                                         \
      launch_pdl(quantize_kernel<MODE, true, kF16>, (unsigned)grid, kQuantThreads, 0, stream, x, nblocks,  \
                 kblocks, ldx, codes, scales, tensor_scale, amax_word, amax_parts, scale_given, after_amax); \
    else                                                                                                  \
      launch_pdl(quantize_kernel<MODE, false, kF16>, (unsigned)grid, kQuantThreads, 0, stream, x, nblocks, \
                 kblocks, ldx, codes, scales, tensor_scale, amax_word, amax_parts, scale_given, after_amax); \
  } while (0)
  switch (mode) {
    case MIXFP4_MODE_MIX: MIXFP4_LAUNCH_Q(MIXFP4_MODE_MIX); break;
    case MIXFP4_MODE_E2M1_ONLY: MIXFP4_LAUNCH_Q(MIXFP4_MODE_E2M1_ONLY); break;
    case MIXFP4_MODE_FOUR_SIX: MIXFP4_LAUNCH_Q(MIXFP4_MODE_FOUR_SIX); break;
    default: MIXFP4_LAUNCH_Q(MIXFP4_MODE_E1M2_ONLY); break;
  }
#undef MIXFP4_LAUNCH_Q
}

}  // namespace

int launch_quantize(const uint16_t* x, int64_t rows, int64_t K, int64_t ldx, uint8_t* codes,
                    uint8_t* scales, float* tensor_scale, const uint32_t* amax_word, int mode,
                    int scale_given, cudaStream_t stream) {
  launch_quantize_to<false>(x, rows, K, ldx, codes, scales, tensor_scale, amax_word, 0, mode, scale_given, stream);
  return 0;
}

namespace {

template <int kOut>
bool launch_small(const uint16_t* x, int64_t rows, int64_t K, int64_t ldx, uint8_t* codes, uint8_t* scales,
                  float* tensor_scale, int mode, int xr, cudaStream_t stream) {
  const int64_t kblocks = K / 16, nblocks = rows * kblocks;
  if ((kOut == 1 ? xr * kblocks : nblocks) > (int64_t)kSmallCtas * kSmallThreads * kSmallPer) return false;
#define MIXFP4_LAUNCH_SM(MODE)                                                                                  \
  (ldx == K ? launch_pdl(quantize_small_kernel<MODE, true, kOut>, kSmallCtas, kSmallThreads, 0, stream, x, nblocks, \
                         kblocks, ldx, codes, scales, tensor_scale, xr)                                          \
            : launch_pdl(quantize_small_kernel<MODE, false, kOut>, kSmallCtas, kSmallThreads, 0, stream, x, nblocks, \
                         kblocks, ldx, codes, scales, tensor_scale, xr))
  switch (mode) {
    case MIXFP4_MODE_MIX: MIXFP4_LAUNCH_SM(MIXFP4_MODE_MIX); break;
    case MIXFP4_MODE_E2M1_ONLY: MIXFP4_LAUNCH_SM(MIXFP4_MODE_E2M1_ONLY); break;
    case MIXFP4_MODE_FOUR_SIX: MIXFP4_LAUNCH_SM(MIXFP4_MODE_FOUR_SIX); break;
    default: MIXFP4_LAUNCH_SM(MIXFP4_MODE_E1M2_ONLY); break;
  }
#undef MIXFP4_LAUNCH_SM
  return true;  // a launch error is the caller's cudaGetLastError
}

}  // namespace

// Quantize with the scale computed, in one launch; false (nothing enqueued) for
// a tensor too large for it.
bool launch_quantize_small(const uint16_t* x, int64_t rows, int64_t K, int64_t ldx, uint8_t* codes, uint8_t* scales,
                           float* tensor_scale, int mode, cudaStream_t stream) {
  return launch_small<0>(x, rows, K, ldx, codes, scales, tensor_scale, mode, 0, stream);
}

// The same into the few-row GEMM's activation operand.
bool launch_quantize_fewrows(const uint16_t* x, int64_t rows, int64_t K, int64_t ldx, uint8_t* xop, uint8_t* sfa,
                             float* tensor_scale, int mode, int xr, cudaStream_t stream) {
  return launch_small<1>(x, rows, K, ldx, xop, sfa, tensor_scale, mode, xr, stream);
}

// The tensor quantized with its scale computed, as f16 values u * s8, [rows][K]
// (the operand of launch_gemm_f16a).  parts: scratch of kMaxAmaxParts words.
int launch_quantize_f16(const uint16_t* x, int64_t rows, int64_t K, int64_t ldx, void* out, float* tensor_scale,
                        uint32_t* parts, int mode, cudaStream_t stream) {
  int n = 0;
  launch_amax_parts(x, rows, K, ldx, parts, &n, stream);
  launch_quantize_to<true>(x, rows, K, ldx, static_cast<uint8_t*>(out), nullptr, tensor_scale, parts, n, mode, 0,
                           stream);
  return 0;
}

int launch_rht_amax(const uint16_t* x, int64_t rows, int64_t K, int64_t ldx, const uint8_t* signs,
                    uint32_t* amax_word, cudaStream_t stream) {
  const int64_t kblocks = K / 16, nblocks = rows * kblocks;
  if (nblocks == 0) return 0;
  int64_t grid = (nblocks + 255) / 256;
  if (grid > num_sms() * 8) grid = num_sms() * 8;
  launch_zero_word(amax_word, stream);
  if (ldx == K) launch_pdl(rht_amax_kernel<true>, (unsigned)grid, 256, 0, stream, x, nblocks, kblocks, ldx, signs, amax_word);
  else launch_pdl(rht_amax_kernel<false>, (unsigned)grid, 256, 0, stream, x, nblocks, kblocks, ldx, signs, amax_word);
  return 0;
}

int launch_rht_quantize(const uint16_t* x, int64_t rows, int64_t K, int64_t ldx, const uint8_t* signs,
                        uint8_t* codes, uint8_t* scales, float* tensor_scale, const uint32_t* amax_word, int mode,
                        int scale_given, cudaStream_t stream) {
  const int64_t kblocks = K / 16, nblocks = rows * kblocks;
  int64_t grid = (nblocks + kQuantThreads - 1) / kQuantThreads;
  if (grid > num_sms() * 2) grid = num_sms() * 2;
  if (grid == 0) return 0;
  const int after_amax = !scale_given;
#define MIXFP4_LAUNCH_R(MODE)                                                                            \
  do {                                                                                                   \
    if (ldx == K)                                                                                        \
      launch_pdl(rht_quantize_kernel<MODE, true>, (unsigned)grid, kQuantThreads, 0, stream, x, nblocks,   \
                 kblocks, ldx, signs, codes, scales, tensor_scale, amax_word, scale_given, after_amax);  \
    else                                                                                                 \
      launch_pdl(rht_quantize_kernel<MODE, false>, (unsigned)grid, kQuantThreads, 0, stream, x, nblocks,  \
                 kblocks, ldx, signs, codes, scales, tensor_scale, amax_word, scale_given, after_amax);  \
  } while (0)
  switch (mode) {
    case MIXFP4_MODE_MIX: MIXFP4_LAUNCH_R(MIXFP4_MODE_MIX); break;
    case MIXFP4_MODE_E2M1_ONLY: MIXFP4_LAUNCH_R(MIXFP4_MODE_E2M1_ONLY); break;
    default: MIXFP4_LAUNCH_R(MIXFP4_MODE_E1M2_ONLY); break;
  }
#undef MIXFP4_LAUNCH_R
  return 0;
}

int launch_dequantize(const uint8_t* codes, const uint8_t* scales, const float* tensor_scale,
                      int64_t rows, int64_t K, float* out, cudaStream_t stream) {
  const int64_t nblocks = rows * (K / 16);
  const int64_t grid = (nblocks + 255) / 256;
  if (grid == 0) return 0;
  dequantize_kernel<<<(unsigned)grid, 256, 0, stream>>>(codes, scales, tensor_scale, nblocks, out);
  return 0;
}

}  // namespace mixfp4
