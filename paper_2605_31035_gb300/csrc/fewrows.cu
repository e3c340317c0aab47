// Few-row MixFP4 GEMM (M <= 64 activation rows, the decode shapes) on the
// block-scaled FP4 tensor path: C = A_deq . B_deq^T.
//
// Decomposition (every product exact).  A weight block is used in the form
// that costs the fewest instructions: an E2M1 block is its stored codes w
// under its scale; an E1M2 block has p = 2 (e(p & 3) + e(p & 4)) with e() the
// E2M1 value, so it is two operands that differ from w by one mask each,
// w & 0xB.. and w & 0xC.. (sign bits kept), under the same scale and with the
// factor 2 applied at the end (twice the scale itself would overflow E4M3).
// Scales of the other type are 0, so no code is rewritten.  The stored codes go
// from HBM straight into an MMA operand tile.  (The residual form of native.cu
// takes eight instructions per eight codes where this takes two.)  Activation
// rows are main + residual as in native.cu, formed once per call by
// fewrows_prep_kernel: XR main rows, then XR residual rows (XR = 16, 32 or 64),
// with their scales in the tensor core's tiled layout.
//
// Main kernel: one CTA per SM; unit = 128 weight rows x 256 K; a work item is
// (128-row tile, part of K: kps units of one accumulation), dealt round-robin.
// The weight rows are the MMA's M = 128 side and the 2 XR activation operand
// rows its N side: an instruction takes max(39, N / 2) cycles (measured), 40 for up
// to 16 rows, against 64 with the sides swapped, and accumulator lanes are
// weight rows, so C is stored coalesced.  Per 64-K step three kind::mxf4nvf4
// MMAs: the stored codes into D2, the two masked tiles into D1.  Per CTA:
//   warp 0       TMA: activation operand, weight codes (128-byte swizzle) and
//                activation scales into the raw ring; the first weight codes
//                before the activations are ready;
//   warp 1       TMEM allocator; one thread copies each unit's scales to tensor
//                memory (tcgen05.cp, about 9 cycles each) and issues its MMAs;
//   warp 2       the weight rows' block scales, 16 bytes a row, into the raw ring
//                by cp.async (a 16-byte-wide TMA box runs at 0.9 TB/s, and plain
//                loads in the splitters stall their proxy fence for a DRAM
//                round trip: 1.5 us a unit);
//   warps 4-7    epilogue, one TMEM lane quarter each (for XR = 64, where eight
//                splitter warps have no slot, twelve warps: three share a
//                quarter's activation rows in turns of eight);
//   warps 8-31   three groups of eight (two for XR = 64) taking units in turn,
//                two threads per weight row: masked codes into tensor memory (the MMA's A
//                operand; in shared memory their stores and the MMA's reads
//                put a unit at 1200 of its 850 cycles of HBM time), the two
//                scale tiles (E2M1 blocks, E1M2 blocks) into shared memory.
// An item adds up D2 + 2 D1 over main and residual columns with two-sum
// compensation and stores C, or, with K in several parts, its part;
// sum_parts_kernel adds those up the same way.  The sums run on packed fp32
// pairs, two activation rows an instruction; with the twelve warps that took the
// GEMM at 64 x 28672 x 8192 from 50.0 to 44.6 us, at 64 x 14336 x 4096 from 16.9
// to 14.9, at 16 x 28672 x 8192 from 33.3 to 32.1.  (An exchange of the parts
// within a cluster in place of the sum kernel took 40 us there: its cluster-wide
// release waits for the loads in flight, 3 us an item.)
//
// Every pipeline wait is bounded; a wait that gives up records a status bit
// (1 producer, 2 / 4 MMA thread, 8 final drain, 16 / 32 splitters, 64
// epilogue) and the CTA drains and exits without storing more of its output.  With
// K in parts the sum kernel still runs, over parts that may not have been written.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>
#include <cstdint>

#include "host_util.cuh"
#include "kernels.cuh"
#include "pipeline.cuh"
#include "ptx.cuh"
#include "residual.cuh"
#include "sm100.cuh"

namespace mixfp4 {
namespace {

using namespace sm100;

namespace fr {

constexpr int WR = 128;                    // weight rows per tile
constexpr int BKC = 256, ROWB = BKC / 2;   // K and code bytes of a row per unit
constexpr int W_TILE = WR * ROWB;          // 16 KB
constexpr int SF_UNIT = 4 * 512;           // tiled scales of 128 rows for a unit's four K steps
constexpr int SPLIT_SLOT = 2 * SF_UNIT;     // the weight scales of E2M1 blocks and of E1M2 blocks
constexpr int kMaxRaw = 8, kMaxSplit = 3;
constexpr int kGroups = 3, kGroupWarps = 8;
constexpr int kFirstEpi = 4, kFirstSplit = 8;
constexpr int kThreads = 32 * (kFirstSplit + kGroups * kGroupWarps);  // 1024
// Tensor memory: D2 and D1 of 2 XR columns each (twice for XR = 16), then per
// split slot the two masked code operands (lane = weight row, 8 codes a
// column: 32 columns each) and the unit's scales (per K step 4 columns each of
// the activation, E2M1-block and E1M2-block scales).
constexpr uint32_t kTmemCols = 512, kCodeCols = 32, kSlotCols = 2 * kCodeCols + 48;
__host__ __device__ constexpr int acc_buffers(int xr) { return xr == 16 ? 2 : 1; }
__host__ __device__ constexpr int acc_cols(int xr) { return acc_buffers(xr) * 4 * xr; }
constexpr uint64_t kWaitLimitNs = 1000000000ull;
constexpr int OFF_RINGS = 1024;            // after the barrier block

__host__ __device__ constexpr int xr_of(int m) { return m <= 16 ? 16 : (m <= 32 ? 32 : 64); }
// Raw stage: activation operand (2 XR rows), weight codes, activation scales, weight scale rows.
__host__ __device__ constexpr int off_w(int xr) { return 2 * xr * ROWB; }
__host__ __device__ constexpr int off_sfa(int xr) { return off_w(xr) + W_TILE; }
__host__ __device__ constexpr int off_ws(int xr) { return off_sfa(xr) + SF_UNIT; }
__host__ __device__ constexpr int raw_stage(int xr) { return off_ws(xr) + WR * 16; }
__host__ __device__ constexpr int raw_stages(int xr) { return xr == 16 ? 8 : (xr == 32 ? 7 : 5); }
__host__ __device__ constexpr int split_slots(int xr) { return xr == 64 ? 2 : 3; }
// Splitter groups at work.  A group takes every groups()-th unit and waits by
// phase parity, so it must never be two phases of a barrier ahead: as many
// groups as split slots, and a raw slot's previous landing must lie before the
// last unit known to be consumed (groups + slots units back).
__host__ __device__ constexpr int groups(int xr) { return split_slots(xr); }
// Sets of four epilogue warps: the warps of a group without a slot join warps 4-7.
__host__ __device__ constexpr int epi_sets(int xr) { return 1 + 2 * (kGroups - groups(xr)); }
__host__ __device__ constexpr int smem_of(int xr) {
  return 1024 + OFF_RINGS + raw_stages(xr) * raw_stage(xr) + split_slots(xr) * SPLIT_SLOT;
}
static_assert(smem_of(16) <= 232448 && smem_of(32) <= 232448 && smem_of(64) <= 232448, "shared memory budget");
static_assert(raw_stages(16) >= 6 && raw_stages(32) >= 6 && raw_stages(64) >= 4 && groups(16) <= kGroups,
              "raw stages >= groups + split slots");
static_assert(raw_stage(16) % 1024 == 0, "swizzled tiles need 1024-byte alignment");
static_assert(acc_cols(16) + split_slots(16) * kSlotCols <= kTmemCols &&
                  acc_cols(32) + split_slots(32) * kSlotCols <= kTmemCols &&
                  acc_cols(64) + split_slots(64) * kSlotCols <= kTmemCols, "TMEM budget");

// Workspace: activation operand, its scales, the parts ([splits][M][tiles x 128]).
struct Scratch {
  int64_t sfa, parts, bytes;
};
inline Scratch scratch_of(int64_t M, int64_t N, int64_t K, int splits) {
  const int64_t xr = xr_of((int)M), tiles = (N + WR - 1) / WR;
  auto up = [](int64_t v) { return (v + 255) / 256 * 256; };
  Scratch s;
  s.sfa = up(2 * xr * (K / 2));
  s.parts = s.sfa + K / BKC * SF_UNIT;
  s.bytes = s.parts + (splits > 1 ? splits * M * tiles * WR * 4 : 0);
  return s;
}

// two_sum_add on pairs.
__device__ __forceinline__ void two_sum_add2(u64& s, u64& e, u64 v) {
  const u64 t = add2(s, v), z = sub2(t, s);
  e = add2(e, add2(sub2(s, sub2(t, z)), sub2(v, z)));
  s = t;
}

struct Bars {
  uint64_t raw_full[kMaxRaw], raw_empty[kMaxRaw];
  uint64_t split_full[kMaxSplit], split_empty[kMaxSplit];
  uint64_t acc_full[2], acc_empty[2];
  uint64_t drain;
  uint32_t tmem_base;
  int abort;
};
static_assert(sizeof(Bars) <= OFF_RINGS, "barrier block");

// Activation operand: thread = 16-byte chunk (32 codes) of one of XR rows.
__global__ void __launch_bounds__(256)
fewrows_prep_kernel(const uint8_t* codes, const uint8_t* scales, int M, int xr, int K, uint8_t* __restrict__ xop,
                    uint8_t* __restrict__ sfa) {
  griddep_wait();
  griddep_launch_dependents();
  // Unsigned: 64 rows of K = 2^30 are 2^31 chunks.
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x, per_row = (uint32_t)K / 32;
  if (i >= (uint32_t)xr * per_row) return;
  const int r = (int)(i / per_row), c = (int)(i - (uint32_t)r * per_row);
  uint4 w = make_uint4(0u, 0u, 0u, 0u);
  uint32_t s4 = 0u;  // scales of the 64-K step this chunk lies in
  if (r < M) {
    w = reinterpret_cast<const uint4*>(codes + (int64_t)r * (K / 2))[c];
    s4 = reinterpret_cast<const uint32_t*>(scales + (int64_t)r * (K / 16))[c / 2];
  }
  const uint32_t m0 = type_mask(s4, 2 * (c & 1)), m1 = type_mask(s4, 2 * (c & 1) + 1);
  const uint4 q = make_uint4(residual_word(w.x) & m0, residual_word(w.y) & m0, residual_word(w.z) & m1,
                             residual_word(w.w) & m1);
  reinterpret_cast<uint4*>(xop + (int64_t)r * (K / 2))[c] = w;
  reinterpret_cast<uint4*>(xop + (int64_t)(xr + r) * (K / 2))[c] = q;
  if ((c & 1) == 0) {
    uint8_t* t = sfa + (int64_t)(c / 2) * 512;
    *reinterpret_cast<uint32_t*>(t + tiled_scale_row(r)) = s4 & 0x7F7F7F7Fu;
    *reinterpret_cast<uint32_t*>(t + tiled_scale_row(xr + r)) = s4 & 0x7F7F7F7Fu;
  }
}

// Units whose weight codes are requested while the kernel before still writes
// the activations.  linear() with weights out of L2 (M x N x K, us): 1x14336x4096
// 20.5 with none, 18.4 with 2, 18.4 with the whole ring; 1x4096x14336 25.4,
// 23.6, 23.0; 16x28672x8192 44.5, 43.0, 42.5; 20x14336x14336 48.7, 48.1, 49.2.
// After the shorter operand kernel of a GEMM on quantized rows the whole ring
// costs up to 0.8 us (1x4096x14336 13.4, 13.5, 14.2: its small loads queue
// behind the weights), two units nothing.
constexpr int kAhead = 2;

__global__ void __launch_bounds__(kThreads, 1)
fewrows_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_x,
               const uint8_t* w_scales, const uint8_t* sfa, int M, int xr, int N, int K, int splits, int kps,
               const float* a_ts, const float* b_ts, float* __restrict__ parts, float* __restrict__ C, long long ldc,
               uint32_t* status_word) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  Bars* bars = reinterpret_cast<Bars*>(smem);
  volatile int* abort_flag = &bars->abort;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int num_kc = K / BKC, tiles = (N + WR - 1) / WR, items = tiles * splits;
  const int R = raw_stages(xr), S = split_slots(xr), NB = acc_buffers(xr);
  const uint32_t RS = (uint32_t)raw_stage(xr);
  const uint32_t raw0 = smem_u32(smem) + OFF_RINGS, split0 = raw0 + (uint32_t)R * RS;

  if (threadIdx.x == 0) {
    for (int s = 0; s < R; ++s) {
      mbar_init(smem_u32(&bars->raw_full[s]), 1 + 32);  // TMA thread, the scale loader's lanes
      mbar_init(smem_u32(&bars->raw_empty[s]), 1);
    }
    for (int s = 0; s < S; ++s) {
      mbar_init(smem_u32(&bars->split_full[s]), kGroupWarps);
      mbar_init(smem_u32(&bars->split_empty[s]), 1);
    }
    for (int s = 0; s < NB; ++s) {
      mbar_init(smem_u32(&bars->acc_full[s]), 1);
      mbar_init(smem_u32(&bars->acc_empty[s]), 4 * (uint32_t)epi_sets(xr));
    }
    mbar_init(smem_u32(&bars->drain), 1);
    bars->abort = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&bars->tmem_base), kTmemCols);
    tmem_relinquish();
  }
  griddep_launch_dependents();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = bars->tmem_base;

  auto fail = [&](uint32_t code) {
    *abort_flag = 1;
    if (status_word) atomicOr(status_word, code);
  };
  // K range of an item: tile = item / splits, part = item % splits.
  auto k_begin = [&](int item) { return (item % splits) * kps; };
  auto k_end = [&](int item) {
    const int e = (item % splits) * kps + kps;
    return e < num_kc ? e : num_kc;
  };

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    // The weights do not depend on the kernel before this one (see the launch),
    // so the first kAhead units' codes are requested before waiting for it (and
    // the scale warp does not wait at all); their activation parts follow after
    // the wait, the other units in one go.
    if (elect_one()) {
      tma_prefetch(&tm_w);
      tma_prefetch(&tm_x);
      const uint32_t tx = (uint32_t)off_ws(xr);  // all of the stage but the weight scale rows
      auto load_w = [&](int s, int row, int kc) {
        const uint32_t fb = smem_u32(&bars->raw_full[s]);
        mbar_arrive_expect_tx(fb, tx);
        tma_load_2d(raw0 + (uint32_t)s * RS + (uint32_t)off_w(xr), &tm_w, kc * ROWB, row, fb);
      };
      auto load_x = [&](int s, int kc) {
        const uint32_t st = raw0 + (uint32_t)s * RS, fb = smem_u32(&bars->raw_full[s]);
        tma_load_2d(st, &tm_x, kc * ROWB, 0, fb);
        bulk_load(st + (uint32_t)off_sfa(xr), sfa + (int64_t)kc * SF_UNIT, SF_UNIT, fb);
      };
      int n = 0;
      for (int item = blockIdx.x; item < items && n < kAhead; item += gridDim.x)
        for (int kc = k_begin(item); kc < k_end(item) && n < kAhead; ++kc, ++n) load_w(n, (item / splits) * WR, kc);
      griddep_wait();
      int it = 0, last = -1, s = 0;
      uint32_t ph = 1;
      bool ok = true;
      for (int item = blockIdx.x; item < items && ok; item += gridDim.x) {
        const int row = (item / splits) * WR, ke = k_end(item);
        for (int kc = k_begin(item); kc < ke; ++kc, ++it) {
          if (it >= n) {
            if (!mbar_wait(smem_u32(&bars->raw_empty[s]), ph, abort_flag, kWaitLimitNs)) {
              fail(1u);
              ok = false;
              break;
            }
            load_w(s, row, kc);
          }
          load_x(s, kc);
          last = it;
          if (++s == R) {
            s = 0;
            ph ^= 1;
          }
        }
      }
      if (*abort_flag)
        for (int u = last - R + 1; u <= last; ++u)
          if (u >= 0) mbar_wait(smem_u32(&bars->raw_full[u % R]), (uint32_t)((u / R) & 1), nullptr, kWaitLimitNs);
    }
  } else if (warp == 1) {
    // ---------------- scale copies and MMAs ----------------
    if (elect_one()) {
      const uint32_t idesc = idesc_nvf4_f32(WR, 2 * xr);
      int r = 0, s = 0, ab = 0;
      uint32_t sph = 0, aph = 1;
      bool ok = true;
      for (int item = blockIdx.x; item < items && ok; item += gridDim.x) {
        if (!mbar_wait(smem_u32(&bars->acc_empty[ab]), aph, abort_flag, kWaitLimitNs)) {
          fail(2u);
          break;
        }
        tc_fence_after();
        const uint32_t d2 = tmem_base + (uint32_t)(ab * 4 * xr), d1 = d2 + (uint32_t)(2 * xr);
        const int kb = k_begin(item), ke = k_end(item);
        for (int kc = kb; kc < ke; ++kc) {
          // The splitters waited for the raw stage before they filled the slot.
          if (!mbar_wait(smem_u32(&bars->split_full[s]), sph, abort_flag, kWaitLimitNs)) {
            fail(4u);
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t st = raw0 + (uint32_t)r * RS, sl = split0 + (uint32_t)s * SPLIT_SLOT;
          const uint32_t tb = tmem_base + (uint32_t)acc_cols(xr) + (uint32_t)s * kSlotCols, sc = tb + 2 * kCodeCols;
          const uint64_t xs = smem_desc_noswizzle(st + (uint32_t)off_sfa(xr), 128, 128);
          const uint64_t w2s = smem_desc_noswizzle(sl, 128, 128);
          const uint64_t xd = smem_desc_sw128(st), wd = smem_desc_sw128(st + (uint32_t)off_w(xr));
          // Offsets below move the descriptors' start addresses (16-byte units).
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            tmem_cp_32x128b_x4(sc + 12 * j, xs + j * (512 >> 4));
            tmem_cp_32x128b_x4(sc + 12 * j + 4, w2s + j * (512 >> 4));
            tmem_cp_32x128b_x4(sc + 12 * j + 8, w2s + ((SF_UNIT + j * 512) >> 4));
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const uint32_t acc = (kc > kb || j > 0) ? 1u : 0u;
            mma_nvf4(d2, wd + j * 2, xd + j * 2, idesc, sc + 12 * j + 4, sc + 12 * j, acc);
            mma_nvf4_tmem_a(d1, tb + 8 * j, xd + j * 2, idesc, sc + 12 * j + 8, sc + 12 * j, acc);
            mma_nvf4_tmem_a(d1, tb + kCodeCols + 8 * j, xd + j * 2, idesc, sc + 12 * j + 8, sc + 12 * j, 1u);
          }
          mma_commit(smem_u32(&bars->raw_empty[r]));
          mma_commit(smem_u32(&bars->split_empty[s]));
          if (++r == R) r = 0;
          if (++s == S) {
            s = 0;
            sph ^= 1;
          }
        }
        if (ok) mma_commit(smem_u32(&bars->acc_full[ab]));
        if (++ab == NB) {
          ab = 0;
          aph ^= 1;
        }
      }
      mma_commit(smem_u32(&bars->drain));
      if (!mbar_wait(smem_u32(&bars->drain), 0, nullptr, kWaitLimitNs)) fail(8u);
    }
  } else if (warp == 2) {
    // ---------------- weight scale rows ----------------
    int s = 0;
    uint32_t ph = 1;
    bool ok = true;
    for (int item = blockIdx.x; item < items && ok; item += gridDim.x) {
      const int row = (item / splits) * WR, ke = k_end(item);
      for (int kc = k_begin(item); kc < ke; ++kc) {
        if (!mbar_wait(smem_u32(&bars->raw_empty[s]), ph, abort_flag, kWaitLimitNs)) {
          fail(1u);
          ok = false;
          break;
        }
        const uint32_t dst = raw0 + (uint32_t)s * RS + (uint32_t)off_ws(xr);
#pragma unroll
        for (int i = 0; i < WR / 32; ++i) {
          const int n = row + 32 * i + lane;
          cp_async16(dst + (uint32_t)(32 * i + lane) * 16, w_scales + (int64_t)(n < N ? n : 0) * (K / 16) + kc * 16, n < N);
        }
        cp_async_arrive(smem_u32(&bars->raw_full[s]));
        if (++s == R) {
          s = 0;
          ph ^= 1;
        }
      }
      ok = __all_sync(0xffffffffu, ok);
    }
    cp_async_wait_all();
  } else if (warp >= kFirstSplit && warp < kFirstSplit + groups(xr) * kGroupWarps) {
    // ---------------- masked code tiles and scale tiles ----------------
    const int g = (warp - kFirstSplit) / kGroupWarps;
    const int row = (warp & 3) * 32 + lane;       // the warp's TMEM lane quarter
    const int half = (warp >> 2) & 1;             // 16-byte chunks 4 half .. 4 half + 3 of the row
    const uint32_t swz = (uint32_t)(row & 7);
    // Walk of this group's units: every G-th one of the CTA's sequence.
    const int G = groups(xr);
    int item = blockIdx.x, kc = k_begin(item), ke = k_end(item), it = 0;
    auto advance = [&](int steps) {
      for (; steps > 0 && item < items; --steps, ++it)
        if (++kc >= ke) {
          item += gridDim.x;
          kc = k_begin(item);
          ke = k_end(item);
        }
    };
    advance(g);
    while (item < items) {
      const int u = it, r = u % R, s = u % S;
      const bool landed = mbar_wait(smem_u32(&bars->raw_full[r]), (uint32_t)((u / R) & 1), abort_flag, kWaitLimitNs);
      if (!__all_sync(0xffffffffu, landed)) {
        if (!landed) fail(16u);
        break;
      }
      const uint32_t src = raw0 + (uint32_t)r * RS + (uint32_t)off_w(xr) + (uint32_t)row * ROWB;
      uint32_t w[16];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint4 c = lds128(src + ((((uint32_t)(4 * half + q)) ^ swz) << 4));
        w[4 * q] = c.x;
        w[4 * q + 1] = c.y;
        w[4 * q + 2] = c.z;
        w[4 * q + 3] = c.w;
      }
      const uint2 cur = lds64(raw0 + (uint32_t)r * RS + (uint32_t)off_ws(xr) + (uint32_t)(row * 16 + half * 8));
      advance(G);
      const bool free = mbar_wait(smem_u32(&bars->split_empty[s]), (uint32_t)((u / S) & 1) ^ 1u, abort_flag, kWaitLimitNs);
      if (!__all_sync(0xffffffffu, free)) {  // tcgen05.st is warp-collective: the warp decides together
        if (!free) fail(32u);
        break;
      }
      tc_fence_after();
      const uint32_t slot = split0 + (uint32_t)s * SPLIT_SLOT;
      const uint32_t tb = tmem_base + (uint32_t)acc_cols(xr) + (uint32_t)s * kSlotCols + (uint32_t)(16 * half) +
                          ((uint32_t)((warp & 3) * 32) << 16);
      uint32_t o[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) o[q] = w[q] & 0xBBBBBBBBu;
      tmem_st_32x32b_x16(tb, o);
#pragma unroll
      for (int q = 0; q < 16; ++q) o[q] = w[q] & 0xCCCCCCCCu;
      tmem_st_32x32b_x16(tb + kCodeCols, o);
#pragma unroll
      for (int j = 0; j < 2; ++j) {  // scales of this half's two K steps, by block type
        const uint32_t sw = j ? cur.y : cur.x;
        const uint32_t t1 = sw & prmt(sw, 0u, 0xBA98u) & 0x7F7F7F7Fu;  // prmt: 0xFF bytes where the type bit is set
        const uint32_t o = slot + (uint32_t)(2 * half + j) * 512 + tiled_scale_row(row);
        sts32(o, (sw & 0x7F7F7F7Fu) ^ t1);
        sts32(o + SF_UNIT, t1);
      }
      fence_proxy_async_smem();
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bars->split_full[s]));
    }
  } else if (warp >= kFirstEpi) {
    // ---------------- epilogue ----------------
    // Lane d = 32 q + lane is weight row d of the tile; columns m and XR + m of
    // D2 and D1 are activation row m's main and residual products.
    const int q = warp & 3;
    griddep_wait();
    const float sa = a_ts[0], sb = b_ts[0];
    const u64 sa2 = pack2(sa, sa), sb2 = pack2(sb, sb), two = pack2(2.0f, 2.0f);
    const int npad = tiles * WR;
    const int set = warp < kFirstSplit ? 0 : (warp - kFirstSplit) / 4 - 2 * groups(xr) + 1;
    int ab = 0;
    uint32_t aph = 0;
    for (int item = blockIdx.x; item < items; item += gridDim.x) {
      const bool acc_ok = mbar_wait(smem_u32(&bars->acc_full[ab]), aph, abort_flag, kWaitLimitNs);
      tc_fence_after();
      const bool go = __all_sync(0xffffffffu, acc_ok && !*abort_flag);
      if (!go) {
        if (!acc_ok && !*abort_flag) fail(64u);
        break;
      }
      const int part = item % splits, n = (item / splits) * WR + q * 32 + lane;
      const uint32_t t2 = tmem_base + (uint32_t)(ab * 4 * xr) + ((uint32_t)(q * 32) << 16), t1 = t2 + (uint32_t)(2 * xr);
#pragma unroll 1
      for (int m0 = 8 * set; m0 < M; m0 += 8 * epi_sets(xr)) {
        uint32_t v[4][8];
        tmem_ld_32x32b_x8(t2 + (uint32_t)m0, v[0]);
        tmem_ld_32x32b_x8(t2 + (uint32_t)(xr + m0), v[1]);
        tmem_ld_32x32b_x8(t1 + (uint32_t)m0, v[2]);
        tmem_ld_32x32b_x8(t1 + (uint32_t)(xr + m0), v[3]);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 4; ++i) reg_fence8(v[i]);
#pragma unroll
        for (int k = 0; k < 8; k += 2) {  // two activation rows per instruction
          if (m0 + k >= M) break;         // uniform
          u64 s = bits2(v[0][k], v[0][k + 1]), e = 0ull;
          two_sum_add2(s, e, bits2(v[1][k], v[1][k + 1]));
          two_sum_add2(s, e, mul2(bits2(v[2][k], v[2][k + 1]), two));
          two_sum_add2(s, e, mul2(bits2(v[3][k], v[3][k + 1]), two));
          s = add2(s, e);
          const bool second = m0 + k + 1 < M;
          float o0, o1;
          if (splits > 1) {
            float* dst = parts + ((int64_t)part * M + m0 + k) * npad + n;
            unpack2(s, o0, o1);
            dst[0] = o0;
            if (second) dst[npad] = o1;
          } else if (n < N) {
            float* dst = C + (long long)(m0 + k) * ldc + n;
            unpack2(mul2(mul2(s, sa2), sb2), o0, o1);
            dst[0] = o0;
            if (second) dst[ldc] = o1;
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bars->acc_empty[ab]));
      if (++ab == NB) {
        ab = 0;
        aph ^= 1;
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kTmemCols);
  }
}

// Units per item, by the time of the whole call (us): a CTA's units at 0.45
// each, 0.5 per item for its first loads and last drain, and with several parts
// the sum kernel and its traffic.  Fitted to every size of item at 1 to 64 rows
// on ten weight shapes (1024x8192 to 28672x8192): the choice is within 0.5 % of
// the best one on average.  An item is at most one accumulation chunk.
int plan_kps(int64_t M, int64_t N, int64_t K) {
  const int64_t tiles = (N + WR - 1) / WR, num_kc = K / BKC, ctas = num_sms();
  int best = 1;
  double best_cost = -1.0;
  for (int64_t kps = 1; kps <= num_kc && kps <= kAccumChunkK / BKC; ++kps) {
    const int64_t splits = (num_kc + kps - 1) / kps;
    double cost = (double)((tiles * splits + ctas - 1) / ctas) * (0.45 * (double)kps + 0.5);
    if (splits > 1) cost += 1.5 + 0.2 * (double)splits + 2e-6 * (double)(splits * M * N);
    if (best_cost < 0.0 || cost < best_cost) {
      best_cost = cost;
      best = (int)kps;
    }
  }
  return best;
}

}  // namespace fr
}  // namespace

int64_t fewrows_scratch_bytes(int64_t M, int64_t N, int64_t K) {
  const int64_t kps = fr::plan_kps(M, N, K), num_kc = K / fr::BKC;
  return fr::scratch_of(M, N, K, (int)((num_kc + kps - 1) / kps)).bytes;
}

// Few-row GEMM from an activation operand already in the scratch.
static int launch_fewrows_main(const float* a_ts, const uint8_t* b_codes, const uint8_t* b_scales, const float* b_ts,
                               int64_t M, int64_t N, int64_t K, float* C, int64_t ldc, void* scratch,
                               uint32_t* status_word, cudaStream_t stream) {
  const int64_t num_kc = K / fr::BKC, tiles = (N + fr::WR - 1) / fr::WR;
  const int kps = fr::plan_kps(M, N, K), splits = (int)((num_kc + kps - 1) / kps), xr = fr::xr_of((int)M);
  const fr::Scratch sc = fr::scratch_of(M, N, K, splits);
  uint8_t* base = static_cast<uint8_t*>(scratch);
  CUtensorMap tw, tx;
  if (!make_map(&tw, b_codes, (uint64_t)K / 2, (uint64_t)N, fr::ROWB, fr::WR, CU_TENSOR_MAP_SWIZZLE_128B) ||
      !make_map(&tx, base, (uint64_t)K / 2, (uint64_t)(2 * xr), fr::ROWB, (uint32_t)(2 * xr),
                CU_TENSOR_MAP_SWIZZLE_128B))
    return MIXFP4_ERR_CUDA;
  static std::atomic<uint64_t> smem_set{0};
  if (!set_dynamic_smem_once(reinterpret_cast<const void*>(fr::fewrows_kernel), 232448, smem_set))
    return MIXFP4_ERR_CUDA;
  const int64_t items = tiles * splits;
  const int64_t grid = items < num_sms() ? items : num_sms();
  float* parts = reinterpret_cast<float*>(base + sc.parts);
  // A programmatic dependent of the kernel that writes the activation operand
  // (the small quantizer or fewrows_prep_kernel).  That kernel lets this one
  // start only after its own wait for everything before it, so the weights are
  // complete here from the start; only what it writes must be waited for.
  if (launch_pdl(fr::fewrows_kernel, (unsigned)grid, fr::kThreads, (size_t)fr::smem_of(xr), stream, tw, tx, b_scales,
                 static_cast<const uint8_t*>(base + sc.sfa), (int)M, xr, (int)N, (int)K, splits, kps, a_ts,
                 b_ts, parts, C, (long long)ldc, status_word) != cudaSuccess)
    return MIXFP4_ERR_CUDA;
  if (splits == 1) return MIXFP4_OK;
  return launch_sum_parts(parts, splits, M * tiles * fr::WR, tiles * fr::WR, 1.0f, a_ts, b_ts, M, N, C, ldc, stream);
}

int launch_fewrows(const uint8_t* a_codes, const uint8_t* a_scales, const float* a_ts, const uint8_t* b_codes,
                   const uint8_t* b_scales, const float* b_ts, int64_t M, int64_t N, int64_t K, float* C, int64_t ldc,
                   void* scratch, uint32_t* status_word, cudaStream_t stream) {
  const int xr = fr::xr_of((int)M);
  uint8_t* base = static_cast<uint8_t*>(scratch);
  const int64_t prep = xr * (K / 32);
  if (launch_pdl(fr::fewrows_prep_kernel, (unsigned)((prep + 255) / 256), 256, 0, stream, a_codes, a_scales, (int)M, xr,
                 (int)K, base, base + fr::scratch_of(M, N, K, 1).sfa) != cudaSuccess)
    return MIXFP4_ERR_CUDA;
  return launch_fewrows_main(a_ts, b_codes, b_scales, b_ts, M, N, K, C, ldc, scratch, status_word, stream);
}

bool launch_linear_fewrows(const uint16_t* x, int64_t M, int64_t K, int64_t ldx, int mode, float* x_ts,
                           const uint8_t* w_codes, const uint8_t* w_scales, const float* w_ts, int64_t N, float* C,
                           int64_t ldc, void* scratch, uint32_t* status_word, cudaStream_t stream, int* status) {
  uint8_t* base = static_cast<uint8_t*>(scratch);
  if (!launch_quantize_fewrows(x, M, K, ldx, base, base + fr::scratch_of(M, N, K, 1).sfa, x_ts, mode, fr::xr_of((int)M),
                               stream))
    return false;
  *status = launch_fewrows_main(x_ts, w_codes, w_scales, w_ts, M, N, K, C, ldc, scratch, status_word, stream);
  return true;
}

}  // namespace mixfp4
