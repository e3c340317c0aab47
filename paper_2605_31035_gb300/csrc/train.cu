// Quantizer orientations of the MixFP4 training flow (Sec. 3.2: FPROP, DGRAD
// and WGRAD all run on MixFP4 operands; weights use 2D blocks) for sm_103a.
//
//   quantize_colwise_kernel  Algorithm 1 with each 16-element block running
//       down a column of an [R][C] bf16 tensor: the operand of a GEMM that
//       reduces over R (WGRAD reduces over tokens).  Output as the row-wise
//       quantization of the transpose: codes [C][R/2], scales [C][R/16].
//       A CTA stages a 64-row x 256-column tile in shared memory with
//       coalesced 16-byte loads; thread t then owns column t, reads its four
//       16-row blocks (2-byte shared loads, consecutive threads on consecutive
//       columns, no bank conflicts) and writes 32 contiguous code bytes.
//   quantize_2d_kernel  Algorithm 1 with 16 x 16 blocks (reading R12): a
//       half-warp holds one tile, lane i one 16-element row of it, so the
//       tile max and the tree of the rows' error sums are warp shuffles
//       (block_core<kMode, true>); the two half-warps of a warp take
//       horizontally adjacent tiles (64 contiguous bytes per row).  Output in
//       the row-wise layout, every row of a tile repeating its scale byte, so
//       mixfp4_gemm consumes it unchanged.
//   quantize_sr_kernel  row-wise quantization with stochastic rounding of the
//       chosen format's codes (reading R13, the gradients of the training
//       flow); quantize_colwise_kernel<.., true> the same down the columns.
//   quantize_colwise_rht_kernel  the column-wise quantizer with the 128-point
//       rotation applied along the rows first (the WGRAD inputs).
//   transpose_2d_kernel  codes and tile scales of the transpose of a
//       2D-quantized tensor (the DGRAD operand of the weights): each lane
//       transposes a 16 x 16 nibble tile in registers.
// Every kernel shares quantize.cu's per-block arithmetic (quant_core.cuh), so
// its codes are those of Algorithm 1 on the same values bit for bit.
#include <cuda_runtime.h>
#include <cstdint>

#include "host_util.cuh"
#include "kernels.cuh"
#include "ptx.cuh"
#include "quant_core.cuh"

namespace mixfp4 {
namespace {

constexpr int kColThreads = 256;        // columns per tile
constexpr int kColRows = 64;            // rows per tile (four 16-row blocks)

template <int kMode, bool kSR>
__global__ void __launch_bounds__(kColThreads, kSR ? 3 : 4)
quantize_colwise_kernel(const uint16_t* x, int64_t R, int64_t C, int64_t ldx,
                        uint8_t* __restrict__ codes, uint8_t* __restrict__ scales, float* tensor_scale,
                        const uint32_t* amax_word, int scale_given, uint64_t seed, uint64_t offset) {
  __shared__ float4 tab[128];
  // Row pairs interleaved: pairs[p][c] = x[2p][c] | x[2p + 1][c] << 16, the
  // bf16 pair of column c that quantize_block takes as one word.
  __shared__ __align__(16) uint32_t pairs[kColRows / 2][kColThreads];
  fill_scale_table(tab);  // under the kernel before; with it 1024 x 4096 takes 0.3 to 0.5 us less
  griddep_wait();
  griddep_launch_dependents();
  const TensorConsts tc = tensor_consts(tensor_scale, amax_word, scale_given);
  const bool markstein = markstein_needed(tc);
  const int tid = threadIdx.x;
  const int64_t ct_n = (C + kColThreads - 1) / kColThreads, rt_n = (R + kColRows - 1) / kColRows;
  const int64_t nblk_t = R / 16;  // blocks per output row
  // One 32-byte code store and one 4-byte scale store per full tile column
  // when every output row starts aligned for them (R a multiple of 64).
  const bool vec = (R % kColRows) == 0 && (reinterpret_cast<uintptr_t>(codes) & 31) == 0 &&
                   (reinterpret_cast<uintptr_t>(scales) & 3) == 0;
  for (int64_t t = blockIdx.x; t < ct_n * rt_n; t += gridDim.x) {
    const int64_t r0 = (t / ct_n) * kColRows, c0 = (t % ct_n) * kColThreads;
    // Stage the tile: 32 row pairs x 32 chunks of 8 columns; a thread loads
    // the chunk from both rows of a pair (two 16-byte loads) and stores the
    // eight interleaved words (two 16-byte stores).
#pragma unroll
    for (int k = 0; k < (kColRows / 2) * (kColThreads / 8) / kColThreads; ++k) {
      const int q = tid + k * kColThreads;
      const int pr = q / (kColThreads / 8), ch = q % (kColThreads / 8);
      uint4 a = make_uint4(0u, 0u, 0u, 0u), b = a;
      if (r0 + 2 * pr < R && c0 + ch * 8 < C) {
        a = *reinterpret_cast<const uint4*>(x + (r0 + 2 * pr) * ldx + c0 + ch * 8);
        b = *reinterpret_cast<const uint4*>(x + (r0 + 2 * pr + 1) * ldx + c0 + ch * 8);
      }
      uint4* dst = reinterpret_cast<uint4*>(&pairs[pr][ch * 8]);
      dst[0] = make_uint4(prmt(a.x, b.x, 0x5410u), prmt(a.x, b.x, 0x7632u), prmt(a.y, b.y, 0x5410u),
                          prmt(a.y, b.y, 0x7632u));
      dst[1] = make_uint4(prmt(a.z, b.z, 0x5410u), prmt(a.z, b.z, 0x7632u), prmt(a.w, b.w, 0x5410u),
                          prmt(a.w, b.w, 0x7632u));
    }
    __syncthreads();
    const int64_t c = c0 + tid;
    if (c < C) {
      // The four row blocks of column c are 32 contiguous code bytes (and 4
      // scale bytes) of output row c: gathered here, stored once.
      uint32_t out[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u}, sc4 = 0u;
      const int nrb = (int)((R - r0) / 16 < kColRows / 16 ? (R - r0) / 16 : kColRows / 16);
#pragma unroll
      for (int rb = 0; rb < kColRows / 16; ++rb) {
        if (rb >= nrb) break;
        uint32_t w[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) w[j] = pairs[rb * 8 + j][tid];
        uint32_t lo, hi, sb;
        const int64_t ob = r0 / 16 + rb;  // block index along R
        if (kSR) {
          const uint64_t e0 = (uint64_t)c * (uint64_t)R + (uint64_t)ob * 16;  // element index in X^T
          if (tc.scaled) quantize_block_sr<kMode, true, true>(w, tc, tab, seed, offset, e0, lo, hi, sb);
          else if (markstein) quantize_block_sr<kMode, false, true>(w, tc, tab, seed, offset, e0, lo, hi, sb);
          else quantize_block_sr<kMode, false, false>(w, tc, tab, seed, offset, e0, lo, hi, sb);
        } else {
          if (tc.scaled) quantize_block<kMode, true, true>(w, tc, tab, lo, hi, sb);
          else if (markstein) quantize_block<kMode, false, true>(w, tc, tab, lo, hi, sb);
          else quantize_block<kMode, false, false>(w, tc, tab, lo, hi, sb);
        }
        out[2 * rb] = lo;
        out[2 * rb + 1] = hi;
        sc4 |= sb << (8 * rb);
      }
      uint8_t* cdst = codes + c * (R / 2) + (r0 / 16) * 8;
      uint8_t* sdst = scales + c * nblk_t + r0 / 16;
      if (vec && nrb == kColRows / 16) {
        stg256(cdst, out);
        *reinterpret_cast<uint32_t*>(sdst) = sc4;
      } else {
#pragma unroll
        for (int rb = 0; rb < kColRows / 16; ++rb) {
          if (rb < nrb) {
            stg64(cdst + rb * 8, out[2 * rb], out[2 * rb + 1]);
            sdst[rb] = (uint8_t)(sc4 >> (8 * rb));
          }
        }
      }
    }
    __syncthreads();  // the tile is restaged next
  }
}

// Grid-stride loop of the stochastic-rounding quantizer with the division
// method fixed; the next block's load is in flight while a block is quantized.
template <int kMode, bool kContig, bool kScaled, bool kMarkstein>
__device__ __forceinline__ void sr_loop(const uint16_t* x, int64_t b, int64_t nthr, int64_t nblocks,
                                        int64_t kblocks, int64_t ldx, uint8_t* __restrict__ codes,
                                        uint8_t* __restrict__ scales, const TensorConsts& tc,
                                        const float4* __restrict__ tab, uint64_t seed, uint64_t offset) {
  uint32_t w[8];
  if (b < nblocks) ldg256_stream(block_src<kContig>(x, b, kblocks, ldx), w);
  for (; b < nblocks; b += nthr) {
    uint32_t wn[8];
    if (b + nthr < nblocks) ldg256_stream(block_src<kContig>(x, b + nthr, kblocks, ldx), wn);
    uint32_t lo, hi, sb;
    quantize_block_sr<kMode, kScaled, kMarkstein>(w, tc, tab, seed, offset, (uint64_t)b * 16, lo, hi, sb);
    stg64(codes + b * 8, lo, hi);
    scales[b] = (uint8_t)sb;
#pragma unroll
    for (int j = 0; j < 8; ++j) w[j] = wn[j];
  }
}

// Row-wise quantization with stochastic rounding (R13): one thread per
// 16-element block, grid-stride; the element index of block b's first element
// is 16 b (row-major over [rows][K]).
template <int kMode, bool kContig>
__global__ void __launch_bounds__(256, 3)
quantize_sr_kernel(const uint16_t* x, int64_t nblocks, int64_t kblocks, int64_t ldx,
                   uint8_t* __restrict__ codes, uint8_t* __restrict__ scales, float* tensor_scale,
                   const uint32_t* amax_word, int scale_given, uint64_t seed, uint64_t offset) {
  __shared__ float4 tab[128];
  fill_scale_table(tab);
  griddep_wait();
  griddep_launch_dependents();
  const TensorConsts tc = tensor_consts(tensor_scale, amax_word, scale_given);
  const bool markstein = markstein_needed(tc);
  const int64_t nthr = (int64_t)gridDim.x * blockDim.x;
  const int64_t b0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (tc.scaled) sr_loop<kMode, kContig, true, true>(x, b0, nthr, nblocks, kblocks, ldx, codes, scales, tc, tab, seed, offset);
  else if (markstein) sr_loop<kMode, kContig, false, true>(x, b0, nthr, nblocks, kblocks, ldx, codes, scales, tc, tab, seed, offset);
  else sr_loop<kMode, kContig, false, false>(x, b0, nthr, nblocks, kblocks, ldx, codes, scales, tc, tab, seed, offset);
}

constexpr int k2dThreads = 256;

template <int kMode>
__global__ void __launch_bounds__(k2dThreads, 4)
quantize_2d_kernel(const uint16_t* x, int64_t rows, int64_t K, int64_t ldx,
                   uint8_t* __restrict__ codes, uint8_t* __restrict__ scales, float* tensor_scale,
                   const uint32_t* amax_word, int scale_given) {
  __shared__ float4 tab[128];
  fill_scale_table(tab);
  griddep_wait();
  griddep_launch_dependents();
  const TensorConsts tc = tensor_consts(tensor_scale, amax_word, scale_given);
  const bool markstein = markstein_needed(tc);
  const int lane = threadIdx.x & 31, i = lane & 15, h = lane >> 4;
  const int64_t nb = K / 16, pairs = (nb + 1) / 2, rt_n = (rows + 15) / 16;
  const int64_t units = rt_n * pairs;  // (row tile, pair of block columns), one per warp
  const int64_t warp0 = ((int64_t)blockIdx.x * k2dThreads + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * k2dThreads) >> 5;
  for (int64_t u = warp0; u < units; u += nwarps) {
    const int64_t r = (u / pairs) * 16 + i, b = (u % pairs) * 2 + h;
    const bool live = r < rows && b < nb;
    uint32_t w[8];
    if (live) {
      ldg256_stream(x + r * ldx + b * 16, w);
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j) w[j] = 0u;  // missing rows of a ragged tile count as zeros (R12)
    }
    uint32_t lo, hi, sb;
    if (tc.scaled) quantize_block<kMode, true, true, true>(w, tc, tab, lo, hi, sb);
    else if (markstein) quantize_block<kMode, false, true, true>(w, tc, tab, lo, hi, sb);
    else quantize_block<kMode, false, false, true>(w, tc, tab, lo, hi, sb);
    if (live) {
      stg64(codes + r * (K / 2) + b * 8, lo, hi);
      scales[r * nb + b] = (uint8_t)sb;
    }
  }
}

// Column-wise quantization with the 128-point rotation along the rows (the
// weight-gradient inputs of the training recipe, Sec. 3.2 / Sec. 4.2: the RHT
// is applied to both WGRAD operands, whose reduction runs over tokens): every
// 128-row chunk of each column is rotated (reading R11: the caller's sign
// vector, the same butterfly order) and the rotated column is quantized down
// its rows -- bit for bit mixfp4_quantize_rht of X^T.
//
// A warp takes 128-row x 16-column tiles on its own (no barriers beyond the
// warp's).  The butterfly works on pairs of adjacent columns, which are the
// halves of a loaded word, so the packed fp32 instructions need no shuffles and
// no transposition: a lane loads 16 rows of a column pair and does strides 1 to
// 8 in registers; the values pass through the warp's shared memory (fp32, 8
// bytes a pair); a lane then holds the 8 values 16 rows apart for strides 16 to
// 64.  kAmax stops there with the maximum; otherwise they pass through shared
// memory once more and a lane quantizes the two 16-row blocks of a column pair,
// four lanes side by side on 32 code bytes of a column.  A block of 16 rows
// starts 272 words after the one before, so that none of the three access
// patterns (16 lanes of 8 bytes each) conflicts.
// Against the former form (bf16 tile scattered by 2-byte stores, 48 shuffles a
// block, CTA barriers) on 4096 x 4096: amax pass 21.3 -> 13.0 us, quantize 31.1
// -> 25.0 us, both on 8192 x 8192 193 -> 131 us; CTA-wide 64-column tiles of this
// form: 14.8 and 29.0 us.  Four CTAs per SM: 128 registers, no spills (five or
// six spill: 41 us for both passes against 38).
constexpr int kCrRows = 128, kCrCols = 16, kCrWarps = 4, kCrBlk = 16 * kCrCols + 16, kCrTile = 8 * kCrBlk;
__device__ __forceinline__ int cr_word(int b, int i, int col) { return b * kCrBlk + i * kCrCols + col; }

// One radix-2 stage: strides of h over v[0..n).
template <int n, int h>
__device__ __forceinline__ void butterfly(u64 (&v)[n]) {
#pragma unroll
  for (int i = 0; i < n; ++i)
    if ((i & h) == 0) {
      const u64 a = v[i], b = v[i + h];
      v[i] = add2(a, b);
      v[i + h] = sub2(a, b);
    }
}

template <int kMode, bool kAmax>
__global__ void __launch_bounds__(32 * kCrWarps, 4)
quantize_colwise_rht_kernel(const uint16_t* x, int64_t R, int64_t C, int64_t ldx,
                            const uint8_t* signs, uint8_t* __restrict__ codes,
                            uint8_t* __restrict__ scales, float* tensor_scale, uint32_t* amax_word, int scale_given) {
  __shared__ float4 tab[128];
  __shared__ __align__(16) float tiles_s[kCrWarps][kCrTile];
  if (!kAmax) {  // the maximum pass follows launch_zero_word, which waits for all before
    fill_scale_table(tab);
    griddep_wait();
  }
  griddep_launch_dependents();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int cp = lane & 7, g = lane >> 3;  // column pair, and which of four blocks / residues
  float* tile = tiles_s[warp];
  uint32_t bits[2] = {0u, 0u};  // sign bits of the 16 rows of blocks g and g + 4 of a chunk
  if (signs)
#pragma unroll
    for (int h = 0; h < 2; ++h)
      bits[h] = (uint32_t)signs[2 * (g + 4 * h)] | ((uint32_t)signs[2 * (g + 4 * h) + 1] << 8);
  TensorConsts tc{};
  if (!kAmax) {
    tc = tensor_consts(tensor_scale, amax_word, scale_given);
    __syncthreads();
  }
  const float c128 = __uint_as_float(kRhtScaleBits);
  const u64 cc = pack2(c128, c128);
  uint32_t m = 0;
  const int64_t ct_n = C / kCrCols, tiles = ct_n * (R / kCrRows);
  const int64_t nwarps = (int64_t)gridDim.x * kCrWarps;
  for (int64_t t = (int64_t)blockIdx.x * kCrWarps + warp; t < tiles; t += nwarps) {
    const int64_t rt = t / ct_n, c0 = (t - rt * ct_n) * kCrCols;
    const uint16_t* src = x + rt * kCrRows * ldx + c0 + 2 * cp;
    uint32_t w[2][16];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int i = 0; i < 16; ++i)
        w[h][i] = *reinterpret_cast<const uint32_t*>(src + (16 * (g + 4 * h) + i) * ldx);
#pragma unroll
    for (int h = 0; h < 2; ++h) {  // strides 1 to 8 of blocks g and g + 4
      u64 v[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const uint32_t u = w[h][i] ^ (((bits[h] >> i) & 1u) ? 0x80008000u : 0u);
        v[i] = bits2(u << 16, u & 0xFFFF0000u);
      }
      butterfly<16, 1>(v);
      butterfly<16, 2>(v);
      butterfly<16, 4>(v);
      butterfly<16, 8>(v);
#pragma unroll
      for (int i = 0; i < 16; ++i) *reinterpret_cast<u64*>(&tile[cr_word(g + 4 * h, i, 2 * cp)]) = v[i];
    }
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 4; ++k) {  // strides 16 to 64 of rows i, 16 + i, ..., 112 + i
      const int i = g + 4 * k;
      u64 v[8];
#pragma unroll
      for (int b = 0; b < 8; ++b) v[b] = *reinterpret_cast<const u64*>(&tile[cr_word(b, i, 2 * cp)]);
      butterfly<8, 1>(v);
      butterfly<8, 2>(v);
      butterfly<8, 4>(v);
#pragma unroll
      for (int b = 0; b < 8; ++b) {
        v[b] = mul2(v[b], cc);
        if (kAmax) m = max(m, max(lo32(v[b]) & 0x7FFFFFFFu, hi32(v[b]) & 0x7FFFFFFFu));
        else *reinterpret_cast<u64*>(&tile[cr_word(b, i, 2 * cp)]) = v[b];
      }
    }
    __syncwarp();
    if (!kAmax) {
#pragma unroll 1
      for (int h = 0; h < 2; ++h) {
        const int b = g + 4 * h;
        u64 y0[8], y1[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const float2 p = *reinterpret_cast<const float2*>(&tile[cr_word(b, 2 * j, 2 * cp)]);
          const float2 q = *reinterpret_cast<const float2*>(&tile[cr_word(b, 2 * j + 1, 2 * cp)]);
          y0[j] = pack2(p.x, q.x);
          y1[j] = pack2(p.y, q.y);
        }
        uint32_t lo0, hi0, sb0, lo1, hi1, sb1;
        if (tc.scaled) {
          rht_block<kMode, true>(y0, tc, tab, lo0, hi0, sb0);
          rht_block<kMode, true>(y1, tc, tab, lo1, hi1, sb1);
        } else {
          rht_block<kMode, false>(y0, tc, tab, lo0, hi0, sb0);
          rht_block<kMode, false>(y1, tc, tab, lo1, hi1, sb1);
        }
        const int64_t c = c0 + 2 * cp, ob = rt * (kCrRows / 16) + b;
        stg64(codes + c * (R / 2) + ob * 8, lo0, hi0);
        stg64(codes + (c + 1) * (R / 2) + ob * 8, lo1, hi1);
        scales[c * (R / 16) + ob] = (uint8_t)sb0;
        scales[(c + 1) * (R / 16) + ob] = (uint8_t)sb1;
      }
      __syncwarp();  // the tile is rewritten next
    }
  }
  if (kAmax) {
    m = __reduce_max_sync(0xffffffffu, m);
    __shared__ uint32_t red[kCrWarps];
    if (lane == 0) red[warp] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int i = 1; i < kCrWarps; ++i) m = max(m, red[i]);
      griddep_wait();  // the word is zeroed by then
      if (m) atomicMax(amax_word, m);
    }
  }
}

// Transpose of a 16 x 16 nibble tile held in registers: row i of the tile is
// lo[i] (elements 0..7, element e at bits 4e) and hi[i] (elements 8..15); on
// return lo[c] / hi[c] hold column c (tile rows 0..7 / 8..15), packed the same
// way.  Block-recursive: swap the off-diagonal 8 x 8 blocks (register
// renaming), then within every 8 x 8 block the 4 x 4 blocks (16-bit fields),
// the 2 x 2 blocks (bytes) and the single nibbles.
__device__ __forceinline__ void transpose_nibbles16(uint32_t lo[16], uint32_t hi[16]) {
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const uint32_t t = lo[r + 8];
    lo[r + 8] = hi[r];
    hi[r] = t;
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t* w = h ? hi : lo;
#pragma unroll
    for (int r = 0; r < 16; ++r)
      if ((r & 7) < 4) {
        const uint32_t x = w[r], y = w[r + 4];
        w[r] = prmt(x, y, 0x5410u);
        w[r + 4] = prmt(x, y, 0x7632u);
      }
#pragma unroll
    for (int r = 0; r < 16; ++r)
      if ((r & 3) < 2) {
        const uint32_t x = w[r], y = w[r + 2];
        w[r] = prmt(x, y, 0x6240u);
        w[r + 2] = prmt(x, y, 0x7351u);
      }
#pragma unroll
    for (int r = 0; r < 16; r += 2) {
      const uint32_t x = w[r], y = w[r + 1];
      w[r] = (x & 0x0F0F0F0Fu) | ((y << 4) & 0xF0F0F0F0u);
      w[r + 1] = ((x >> 4) & 0x0F0F0F0Fu) | (y & 0xF0F0F0F0u);
    }
  }
}

// A warp moves 64 rows x 128 elements per unit; lane (rb = lane & 3,
// kc = lane >> 2) owns the 16 x 16 tile at rows 16 rb.., elements 16 kc..:
// sixteen 8-byte loads (8 lanes cover 64 contiguous bytes of a row), the
// register transpose, sixteen 8-byte stores (the 4 lanes of a kc write 32
// contiguous bytes of an output row).  No shared memory, no barriers.
constexpr int kTrUnitRows = 64, kTrUnitCols = 128;

__global__ void __launch_bounds__(256)
transpose_2d_kernel(const uint8_t* __restrict__ codes, const uint8_t* __restrict__ scales, int64_t rows, int64_t K,
                    uint8_t* __restrict__ codes_t, uint8_t* __restrict__ scales_t) {
  const int lane = threadIdx.x & 31, rb = lane & 3, kc = lane >> 2;
  const int64_t kt_n = (K + kTrUnitCols - 1) / kTrUnitCols, rt_n = (rows + kTrUnitRows - 1) / kTrUnitRows;
  const int64_t nbt = rows / 16, nb = K / 16;
  // The four row blocks of a unit write one 4-byte word of each transposed
  // scale row when those words are aligned (rows a multiple of 64).
  const bool vec = (rows % kTrUnitRows) == 0 && (reinterpret_cast<uintptr_t>(scales_t) & 3) == 0;
  const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x / 32);
  for (int64_t u = (int64_t)blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5); u < kt_n * rt_n; u += nwarps) {
    const int64_t r0 = (u / kt_n) * kTrUnitRows + rb * 16, k0 = (u % kt_n) * kTrUnitCols + kc * 16;
    const bool live = r0 < rows && k0 < K;
    uint32_t lo[16], hi[16], s = 0u;
    if (live) {
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const uint2 v = __ldg(reinterpret_cast<const uint2*>(codes + (r0 + i) * (K / 2) + k0 / 2));
        lo[i] = v.x;
        hi[i] = v.y;
      }
      s = scales[r0 * nb + k0 / 16];  // tile (r0 / 16, k0 / 16): the same byte in all its 16 rows
    } else {
#pragma unroll
      for (int i = 0; i < 16; ++i) lo[i] = hi[i] = 0u;
    }
    transpose_nibbles16(lo, hi);
    // Scales of row blocks rb = 0..3 of this kc, byte rb of s4.
    const int base = lane & ~3;
    const uint32_t s4 = __shfl_sync(0xffffffffu, s, base) | (__shfl_sync(0xffffffffu, s, base + 1) << 8) |
                        (__shfl_sync(0xffffffffu, s, base + 2) << 16) | (__shfl_sync(0xffffffffu, s, base + 3) << 24);
    if (live) {
#pragma unroll
      for (int c = 0; c < 16; ++c) stg64(codes_t + (k0 + c) * (rows / 2) + r0 / 2, lo[c], hi[c]);
      if (vec) {
        // Lane rb writes output rows k0 + 4 rb .. k0 + 4 rb + 3, row blocks r0 / 16 - rb .. + 3.
#pragma unroll
        for (int j = 0; j < 4; ++j)
          *reinterpret_cast<uint32_t*>(scales_t + (k0 + 4 * rb + j) * nbt + r0 / 16 - rb) = s4;
      } else {
#pragma unroll
        for (int c = 0; c < 16; ++c) scales_t[(k0 + c) * nbt + r0 / 16] = (uint8_t)s;
      }
    }
  }
}

}  // namespace

int launch_quantize_colwise(const uint16_t* x, int64_t R, int64_t C, int64_t ldx, uint8_t* codes, uint8_t* scales,
                            float* tensor_scale, const uint32_t* amax_word, int mode, int scale_given, int sr,
                            uint64_t seed, uint64_t offset, cudaStream_t stream) {
  const int64_t tiles = ((C + kColThreads - 1) / kColThreads) * ((R + kColRows - 1) / kColRows);
  if (tiles == 0) return 0;
  int64_t grid = tiles < num_sms() * 4 ? tiles : num_sms() * 4;
  cudaError_t e;
#define MIXFP4_LAUNCH_C(MODE, SR)                                                                            \
  e = launch_pdl(quantize_colwise_kernel<MODE, SR>, (unsigned)grid, kColThreads, 0, stream, x, R, C, ldx, codes, \
                 scales, tensor_scale, amax_word, scale_given, seed, offset)
  switch (mode) {
    case MIXFP4_MODE_MIX:
      if (sr) MIXFP4_LAUNCH_C(MIXFP4_MODE_MIX, true); else MIXFP4_LAUNCH_C(MIXFP4_MODE_MIX, false);
      break;
    case MIXFP4_MODE_E2M1_ONLY:
      if (sr) MIXFP4_LAUNCH_C(MIXFP4_MODE_E2M1_ONLY, true); else MIXFP4_LAUNCH_C(MIXFP4_MODE_E2M1_ONLY, false);
      break;
    default:
      if (sr) MIXFP4_LAUNCH_C(MIXFP4_MODE_E1M2_ONLY, true); else MIXFP4_LAUNCH_C(MIXFP4_MODE_E1M2_ONLY, false);
      break;
  }
#undef MIXFP4_LAUNCH_C
  return e == cudaSuccess ? 0 : -1;
}

int launch_quantize_sr(const uint16_t* x, int64_t rows, int64_t K, int64_t ldx, uint8_t* codes, uint8_t* scales,
                       float* tensor_scale, const uint32_t* amax_word, int mode, int scale_given, uint64_t seed,
                       uint64_t offset, cudaStream_t stream) {
  const int64_t kblocks = K / 16, nblocks = rows * kblocks;
  if (nblocks == 0) return 0;
  int64_t grid = (nblocks + 255) / 256;
  if (grid > num_sms() * 3) grid = num_sms() * 3;
  cudaError_t e;
#define MIXFP4_LAUNCH_S(MODE)                                                                               \
  e = (ldx == K) ? launch_pdl(quantize_sr_kernel<MODE, true>, (unsigned)grid, 256, 0, stream, x, nblocks, kblocks, \
                              ldx, codes, scales, tensor_scale, amax_word, scale_given, seed, offset)          \
                 : launch_pdl(quantize_sr_kernel<MODE, false>, (unsigned)grid, 256, 0, stream, x, nblocks,       \
                              kblocks, ldx, codes, scales, tensor_scale, amax_word, scale_given, seed, offset)
  switch (mode) {
    case MIXFP4_MODE_MIX: MIXFP4_LAUNCH_S(MIXFP4_MODE_MIX); break;
    case MIXFP4_MODE_E2M1_ONLY: MIXFP4_LAUNCH_S(MIXFP4_MODE_E2M1_ONLY); break;
    default: MIXFP4_LAUNCH_S(MIXFP4_MODE_E1M2_ONLY); break;
  }
#undef MIXFP4_LAUNCH_S
  return e == cudaSuccess ? 0 : -1;
}

int launch_quantize_2d(const uint16_t* x, int64_t rows, int64_t K, int64_t ldx, uint8_t* codes, uint8_t* scales,
                       float* tensor_scale, const uint32_t* amax_word, int mode, int scale_given,
                       cudaStream_t stream) {
  const int64_t units = ((rows + 15) / 16) * ((K / 16 + 1) / 2);
  if (units == 0) return 0;
  int64_t grid = (units + k2dThreads / 32 - 1) / (k2dThreads / 32);
  if (grid > num_sms() * 4) grid = num_sms() * 4;
  cudaError_t e;
  switch (mode) {
    case MIXFP4_MODE_MIX:
      e = launch_pdl(quantize_2d_kernel<MIXFP4_MODE_MIX>, (unsigned)grid, k2dThreads, 0, stream, x, rows, K, ldx,
                     codes, scales, tensor_scale, amax_word, scale_given);
      break;
    case MIXFP4_MODE_E2M1_ONLY:
      e = launch_pdl(quantize_2d_kernel<MIXFP4_MODE_E2M1_ONLY>, (unsigned)grid, k2dThreads, 0, stream, x, rows, K,
                     ldx, codes, scales, tensor_scale, amax_word, scale_given);
      break;
    default:
      e = launch_pdl(quantize_2d_kernel<MIXFP4_MODE_E1M2_ONLY>, (unsigned)grid, k2dThreads, 0, stream, x, rows, K,
                     ldx, codes, scales, tensor_scale, amax_word, scale_given);
      break;
  }
  return e == cudaSuccess ? 0 : -1;
}

int launch_quantize_colwise_rht(const uint16_t* x, int64_t R, int64_t C, int64_t ldx, const uint8_t* signs,
                                uint8_t* codes, uint8_t* scales, float* tensor_scale, uint32_t* amax_word, int mode,
                                int scale_given, int amax_pass, cudaStream_t stream) {
  const int64_t ctas = (C / kCrCols * (R / kCrRows) + kCrWarps - 1) / kCrWarps;  // C is a multiple of 16
  if (ctas == 0) return 0;
  const int64_t cap = num_sms() * 4;
  const int64_t grid = ctas < cap ? ctas : cap;
  cudaError_t e;
#define MIXFP4_LAUNCH_CR(MODE, AMAX)                                                                           \
  e = launch_pdl(quantize_colwise_rht_kernel<MODE, AMAX>, (unsigned)grid, 32 * kCrWarps, 0, stream, x, R, C, ldx, signs, \
                 codes, scales, tensor_scale, amax_word, scale_given)
  if (amax_pass) {
    if (launch_zero_word(amax_word, stream) != 0) return -1;
    MIXFP4_LAUNCH_CR(MIXFP4_MODE_MIX, true);
  } else {
    switch (mode) {
      case MIXFP4_MODE_MIX: MIXFP4_LAUNCH_CR(MIXFP4_MODE_MIX, false); break;
      case MIXFP4_MODE_E2M1_ONLY: MIXFP4_LAUNCH_CR(MIXFP4_MODE_E2M1_ONLY, false); break;
      default: MIXFP4_LAUNCH_CR(MIXFP4_MODE_E1M2_ONLY, false); break;
    }
  }
#undef MIXFP4_LAUNCH_CR
  return e == cudaSuccess ? 0 : -1;
}

int launch_transpose_2d(const uint8_t* codes, const uint8_t* scales, int64_t rows, int64_t K, uint8_t* codes_t,
                        uint8_t* scales_t, cudaStream_t stream) {
  const int64_t units = ((K + kTrUnitCols - 1) / kTrUnitCols) * ((rows + kTrUnitRows - 1) / kTrUnitRows);
  if (units == 0) return 0;
  const int64_t blocks = (units + 7) / 8;  // 8 warps per CTA, one unit each per pass
  const int64_t grid = blocks < num_sms() * 8 ? blocks : num_sms() * 8;
  transpose_2d_kernel<<<(unsigned)grid, 256, 0, stream>>>(codes, scales, rows, K, codes_t, scales_t);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace mixfp4
