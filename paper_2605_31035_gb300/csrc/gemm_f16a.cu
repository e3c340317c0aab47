// MixFP4 x MixFP4 GEMM with the A operand decoded beforehand:
// C = A_deq . B_deq^T from A as exact f16 values u * s8 ([M][K], see
// decode.cuh; written by decode_f16_kernel or straight by the quantizer) and
// B as MixFP4 codes, decoded in the main loop.  Same products, same
// accumulation chunks and same epilogue scaling as the kernel of gemm.cu.
//
// Why a decoded A: with 256-row tiles every A row is decoded once per output
// tile column (18 times for N = 4096) and that work, done by the CUDA cores
// into tensor memory, was what bounded the main loop (A decoders busy 36 of
// 45 us on 2048 x 4096 x 4096).  Decoded once, A costs 2 bytes per element of
// L2-resident traffic, arrives by TMA in the MMA's own layout, and leaves the
// decoders only the B rows of the tile and all of tensor memory to two
// accumulators, so a tile's drain overlaps the next tile's main loop.
//
// Persistent CTA pairs (cta_group::2), pair tiles of 256 x tile_n (tile_n a
// multiple of 32 up to 256, chosen by launch_gemm_f16a).  Per CTA:
//   warp 0       TMA: A stages, 128 rows x 64 K f16 (128-byte swizzle, the
//                layout the MMA reads);
//   warp 1       TMEM allocator; in the leader the MMA-issuing thread;
//   warp 2       TMA: B codes and scales, tile_n / 2 rows x 256 K per stage;
//   warp 3       in the peer: passes landed A stages on to the leader;
//   warps 4-11   epilogue: two warps per TMEM lane quarter, alternating
//                16-column steps: tcgen05.ld -> x s32A s32B / 4 -> swizzled
//                staging tile -> TMA store (or add) of the 32 x 16 box;
//   warps 12-27  B decoders, one thread per row, 64 K at a time (f16 in the
//                canonical K-major no-swizzle layout): four groups of four
//                warps take the four 64-K stages of a code stage.  A group's
//                round (wait, decode, proxy fence, remote arrival) is about
//                0.45 us whatever its share of a stage, so groups side by side
//                and not threads per stage set the rate: two groups held a
//                stage at 0.28 us on every tile width, four at 0.20 to 0.27.
// Measured against the in-loop decode of gemm.cu (warm L2, batches, with the
// decode pass of A): 2048 x 4096 x 4096 51.5 -> 43.3 us, 4096 x 14336 x 4096
// 279 -> 241, 4096 x 4096 x 14336 298 -> 262, 8192^3 643 -> 557 us (1.97
// PFLOP/s).  Bound: the tensor pipe on many waves (83.6 % of active cycles at
// 4096^3); on two (74.7 % at 2048 x 4096 x 4096) a stage's waits, commits and
// decoder round beside it, and the launch, first loads and last drain, about 8 us.
// Every pipeline wait is bounded; a wait that gives up records a status bit
// (1 producers, 2 / 4 MMA waiting for an accumulator / a stage, 8 final drain,
// 16 / 32 decoders, 64 epilogue, 128 forwarder) and the CTA drains and exits.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>
#include <cstdint>
#include <cstring>

#include "decode.cuh"
#include "host_util.cuh"
#include "kernels.cuh"
#include "pipeline.cuh"
#include "ptx.cuh"
#include "sm100.cuh"

namespace mixfp4 {
namespace {

using namespace sm100;

// ------------------------------------------------------------ operand decode
// Thread per 16-byte chunk (32 codes of one row): 16 + 2 bytes in, 64 out.
__global__ void __launch_bounds__(256)
decode_f16_kernel(const uint8_t* codes, const uint8_t* scales, int64_t nchunks, uint8_t* __restrict__ out) {
  griddep_wait();
  griddep_launch_dependents();
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nchunks; i += (int64_t)gridDim.x * blockDim.x) {
    const uint4 c = reinterpret_cast<const uint4*>(codes)[i];
    const uint32_t s = reinterpret_cast<const uint16_t*>(scales)[i];
    uint32_t o[16];
    decode_chunk(c, s, o);
    stg256(out + i * 64, o);
    stg256(out + i * 64 + 32, o + 8);
  }
}

// ---------------------------------------------------------------------- GEMM
namespace fa {

constexpr int BM = 128, TILE_M = 256, TILE_N = 256;   // TILE_N: the widest tile
constexpr int BKC = 256;                              // K per code stage
constexpr int BKS = 64;                               // K per A / decoded-B stage
constexpr int kSub = BKC / BKS;
constexpr int A_STAGE = BM * BKS * 2;                 // 16 KB
constexpr int B_STAGE = (TILE_N / 2) * BKS * 2;       // 16 KB
constexpr int kAStages = 6, kBStages = 4;             // ring slots of A and of decoded B
static_assert(kAStages >= kBStages, "the barriers of a stage are indexed by its A slot");
constexpr int kCodeStages = 2;
constexpr int B_CODE = (TILE_N / 2) * BKC / 2, B_SCALE = (TILE_N / 2) * BKC / 16;
constexpr int CODE_STAGE = B_CODE + B_SCALE;          // 18 KB
constexpr int kEpiWarps = 8, kDecWarps = 16;           // four decoder groups of four
constexpr int kFirstEpi = 4, kFirstDec = kFirstEpi + kEpiWarps;
constexpr int kThreads = 32 * (kFirstDec + kDecWarps);  // 896
static_assert(kFirstEpi % 4 == 0 && kFirstDec % 4 == 0, "warp w covers TMEM lane quarter w % 4");
constexpr int EPI_CHUNK = 16;
constexpr int EPI_BYTES = 32 * EPI_CHUNK * 4;         // one staging tile per warp
constexpr int OFF_B = kAStages * A_STAGE;
constexpr int OFF_CODE = OFF_B + kBStages * B_STAGE;
constexpr int OFF_EPI = OFF_CODE + kCodeStages * CODE_STAGE;
constexpr int OFF_BAR = OFF_EPI + kEpiWarps * EPI_BYTES;
constexpr int SMEM_ALLOC = OFF_BAR + 512 + 1024;
static_assert(CODE_STAGE % 1024 == 0 && SMEM_ALLOC <= 232448, "shared memory layout");
constexpr uint32_t kAccCols = TILE_N, kTmemCols = 512;
constexpr uint32_t kLBO = 128, kSBO = (BKS / 8) * 128;  // decoded B: next 8 K / next 8 rows
constexpr uint64_t kWaitLimitNs = 1000000000ull;

// Stage n (64 K) uses A slot n % kAStages and B slot n % kBStages; both of its
// barriers are the A slot's.  One full barrier collects everything the MMAs of
// a stage wait for and one commit frees both slots: the MMA thread's waits and
// commits (about 40 ns each, three and two per stage with separate barriers
// for A and B) were what bounded narrow tiles.
struct Bars {
  uint64_t full[kAStages];         // leader: own A bytes, the peer's A (forwarded), the stage's decoder warps
  uint64_t peer_full[kAStages];    // peer: own A bytes
  uint64_t empty[kAStages];        // MMA commit (multicast)
  uint64_t code_full[kCodeStages];
  uint64_t code_empty[kCodeStages];
  uint64_t acc_full[2];            // MMA commit (multicast)
  uint64_t acc_empty[2];           // leader: 2 x kEpiWarps arrivals
  uint64_t drain;
  uint32_t tmem_base;
  int abort;
};
static_assert(sizeof(Bars) <= 512, "barrier block");

// The pair's work: Sched over (tile, part of K) units.  With splits > 1 a
// tile's K is cut into `splits` parts of kps 256-K slices (the last one may be
// shorter), each accumulated on its own into its copy of C.
struct Work {
  Sched sched;
  int splits, kps, num_kc, part;
  __device__ Work(int cluster, int ncl, int dp, int ntiles, int nkc, int chunk_kc, int splits_, int kps_)
      : sched(cluster, ncl, dp * splits_, ntiles * splits_, kps_, chunk_kc), splits(splits_), kps(kps_), num_kc(nkc),
        part(0) {}
  __device__ bool next(int& tile, int& k0, int& k1) {
    int tt, a, b;
    while (sched.next(tt, a, b)) {
      tile = tt / splits;
      part = tt - tile * splits;
      k0 = part * kps + a;
      k1 = part * kps + b < num_kc ? part * kps + b : num_kc;
      if (k0 < k1) return true;
    }
    return false;
  }
};

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
gemm_f16a_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_bc,
                 const __grid_constant__ CUtensorMap tm_bs, const __grid_constant__ CUtensorMap tm_c, int c_tma,
                 const float* a_ts, const float* b_ts, int M, int N, int K,
                 float* __restrict__ C, long long ldc, int tile_n, int dp_tiles, int chunk_kc, int splits, int kps,
                 int after_zero, uint32_t* status_word) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  Bars* bars = reinterpret_cast<Bars*>(smem + OFF_BAR);
  volatile int* abort_flag = &bars->abort;
  const uint32_t sbase = smem_u32(smem);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const bool leader = rank == 0;
  const int num_kc = K / BKC;
  const int b_rows = tile_n / 2;  // B rows of this CTA
  const int mtiles = (M + TILE_M - 1) / TILE_M, ntiles_n = (N + tile_n - 1) / tile_n;
  const int ntiles = mtiles * ntiles_n;
  const int cluster_id = blockIdx.x >> 1, nclusters = gridDim.x >> 1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kAStages; ++s) {
      mbar_init(smem_u32(&bars->full[s]), 2 + 2 * kDecWarps / kSub);  // producer, forwarder, one decoder group of each CTA
      mbar_init(smem_u32(&bars->peer_full[s]), 1);
      mbar_init(smem_u32(&bars->empty[s]), 1);
    }
    for (int s = 0; s < kCodeStages; ++s) {
      mbar_init(smem_u32(&bars->code_full[s]), 1);
      mbar_init(smem_u32(&bars->code_empty[s]), kDecWarps);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(smem_u32(&bars->acc_full[s]), 1);
      mbar_init(smem_u32(&bars->acc_empty[s]), 2 * kEpiWarps);
    }
    mbar_init(smem_u32(&bars->drain), 1);
    bars->abort = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc_pair(smem_u32(&bars->tmem_base), kTmemCols);
    tmem_relinquish_pair();
  }
  griddep_launch_dependents();
  tc_fence_before();
  cluster_sync();
  tc_fence_after();
  const uint32_t tmem_base = bars->tmem_base;

  auto fail = [&](uint32_t code) {
    *abort_flag = 1;
    if (status_word) atomicOr(status_word, code);
  };
  Work work(cluster_id, nclusters, dp_tiles, ntiles, num_kc, chunk_kc, splits, kps);
  int t, k0, k1;

  if (warp == 0) {
    // ---------------- TMA producer: A ----------------
    if (elect_one()) {
      tma_prefetch(&tm_a);
      if (!after_zero) griddep_wait();  // launch_zero_rows has waited for the operands
      int it = 0, last = -1;
      bool ok = true;
      while (ok && work.next(t, k0, k1)) {
        const int ma = (t / ntiles_n) * TILE_M + (int)rank * BM;
        for (int k = k0 * kSub; k < k1 * kSub; ++k, ++it) {
          const int s = it % kAStages;
          if (!mbar_wait(smem_u32(&bars->empty[s]), ((it / kAStages) & 1) ^ 1, abort_flag, kWaitLimitNs)) {
            fail(1u);
            ok = false;
            break;
          }
          const uint32_t fb = smem_u32(leader ? &bars->full[s] : &bars->peer_full[s]);
          mbar_arrive_expect_tx(fb, A_STAGE);
          tma_load_2d(sbase + s * A_STAGE, &tm_a, k * BKS, ma, fb);
          last = it;
        }
      }
      if (*abort_flag)
        for (int u = last - kAStages + 1; u <= last; ++u)
          if (u >= 0)
            mbar_wait(smem_u32(leader ? &bars->full[u % kAStages] : &bars->peer_full[u % kAStages]),
                      (uint32_t)((u / kAStages) & 1), nullptr, kWaitLimitNs);
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer (leader CTA) ----------------
    if (leader && elect_one()) {
      const uint32_t idesc = idesc_f16_f32(TILE_M, tile_n);
      const uint64_t adesc0 = smem_desc_sw128(sbase), bdesc0 = smem_desc_noswizzle(sbase + OFF_B, kLBO, kSBO);
      int s = 0, bs = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int i = 0; ok && work.next(t, k0, k1); ++i) {
        const int ab = i & 1;
        if (!mbar_wait_cluster(smem_u32(&bars->acc_empty[ab]), ((i >> 1) & 1) ^ 1, abort_flag, kWaitLimitNs)) {
          fail(2u);
          break;
        }
        tc_fence_after();
        const uint32_t acc = tmem_base + (uint32_t)ab * kAccCols;
        for (int k = k0 * kSub; k < k1 * kSub; ++k) {
          if (!mbar_wait_cluster(smem_u32(&bars->full[s]), ph, abort_flag, kWaitLimitNs)) {
            fail(4u);
            ok = false;
            break;
          }
          tc_fence_after();
          // Start addresses are the descriptors' low 14 bits, in 16-byte units (no carry out of them).
          const uint64_t ad = adesc0 + (uint64_t)((s * A_STAGE) >> 4), bd = bdesc0 + (uint64_t)((bs * B_STAGE) >> 4);
          mma_f16_pair(acc, ad, bd, idesc, k > k0 * kSub ? 1u : 0u);
#pragma unroll
          for (int j = 1; j < BKS / 16; ++j)
            mma_f16_pair(acc, ad + (uint64_t)(j * 2), bd + (uint64_t)(j * 16), idesc, 1u);
          mma_commit_pair(smem_u32(&bars->empty[s]), 3);
          if (++s == kAStages) {
            s = 0;
            ph ^= 1;
          }
          if (++bs == kBStages) bs = 0;
        }
        if (ok) mma_commit_pair(smem_u32(&bars->acc_full[ab]), 3);
      }
      mma_commit_pair(smem_u32(&bars->drain), 1);
      if (!mbar_wait_cluster(smem_u32(&bars->drain), 0, nullptr, kWaitLimitNs)) fail(8u);
    }
  } else if (warp == 2) {
    // ---------------- TMA producer: B codes and scales ----------------
    if (elect_one()) {
      tma_prefetch(&tm_bc);
      tma_prefetch(&tm_bs);
      if (!after_zero) griddep_wait();
      const uint32_t tx = (uint32_t)b_rows * (BKC / 2 + BKC / 16);
      int it = 0, last = -1;
      bool ok = true;
      while (ok && work.next(t, k0, k1)) {
        const int nb = (t % ntiles_n) * tile_n + (int)rank * b_rows;
        for (int kc = k0; kc < k1; ++kc, ++it) {
          const int s = it % kCodeStages;
          if (!mbar_wait(smem_u32(&bars->code_empty[s]), ((it / kCodeStages) & 1) ^ 1, abort_flag, kWaitLimitNs)) {
            fail(1u);
            ok = false;
            break;
          }
          const uint32_t st = sbase + OFF_CODE + s * CODE_STAGE;
          const uint32_t fb = smem_u32(&bars->code_full[s]);
          mbar_arrive_expect_tx(fb, tx);
          tma_load_2d(st, &tm_bc, kc * (BKC / 2), nb, fb);
          tma_load_2d(st + B_CODE, &tm_bs, kc * (BKC / 16), nb, fb);
          last = it;
        }
      }
      if (*abort_flag)
        for (int u = last - kCodeStages + 1; u <= last; ++u)
          if (u >= 0)
            mbar_wait(smem_u32(&bars->code_full[u % kCodeStages]), (uint32_t)((u / kCodeStages) & 1), nullptr,
                      kWaitLimitNs);
    }
  } else if (warp == 3) {
    // ---------------- forwarder (peer CTA) ----------------
    if (!leader && elect_one()) {
      const uint32_t ready0 = mapa_shared(smem_u32(&bars->full[0]), 0);
      int s = 0;
      uint32_t ph = 0;
      bool ok = true;
      while (ok && work.next(t, k0, k1)) {
        for (int k = k0 * kSub; k < k1 * kSub; ++k) {
          if (!mbar_wait(smem_u32(&bars->peer_full[s]), ph, abort_flag, kWaitLimitNs)) {
            fail(128u);
            ok = false;
            break;
          }
          mbar_arrive_cluster(ready0 + 8u * (uint32_t)s);
          if (++s == kAStages) {
            s = 0;
            ph ^= 1;
          }
        }
      }
    }
  } else if (warp >= kFirstDec) {
    // ---------------- B decoders ----------------
    const int sub = (warp - kFirstDec) >> 2;      // the 64-K stage of every code stage this group decodes
    const int rl = (warp & 3) * 32 + lane;        // B row of this thread
    const bool active = rl < b_rows;
    const uint32_t dst_row = sbase + OFF_B + (uint32_t)(rl >> 3) * kSBO + (uint32_t)(rl & 7) * 16;
    const uint32_t swz = (uint32_t)(rl & 7);
    const uint32_t full0 = mapa_shared(smem_u32(&bars->full[0]), 0);
    int it = 0;
    bool ok = true;
    while (ok && work.next(t, k0, k1)) {
      for (int kc = k0; kc < k1 && ok; ++kc, ++it) {
        const int s = it % kCodeStages;
        if (!mbar_wait(smem_u32(&bars->code_full[s]), (uint32_t)((it / kCodeStages) & 1), abort_flag, kWaitLimitNs)) {
          fail(16u);
          break;
        }
        const uint32_t st = sbase + OFF_CODE + s * CODE_STAGE;
        const uint32_t crow = st + (uint32_t)rl * (BKC / 2);
        uint4 c[2];
        uint32_t s4 = 0u;  // the stage's four block scales of the row
        if (active) {
          s4 = lds32(st + B_CODE + (uint32_t)rl * (BKC / 16) + (uint32_t)sub * 4);
#pragma unroll
          for (int j = 0; j < 2; ++j) c[j] = lds128(crow + (((uint32_t)(2 * sub + j) ^ swz) << 4));
        }
        const int n = it * kSub + sub, prev = n - kBStages;  // the stage that last used this stage's B slot
        if (prev >= 0 && !mbar_wait_cluster(smem_u32(&bars->empty[prev % kAStages]),
                                            (uint32_t)(prev / kAStages) & 1u, abort_flag, kWaitLimitNs)) {
          fail(32u);
          ok = false;
          break;
        }
        if (active) {
          const uint32_t dst = dst_row + (uint32_t)(n % kBStages) * B_STAGE;
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            uint32_t o[16];
            decode_chunk(c[j], j ? (s4 >> 16) : (s4 & 0xFFFFu), o);
#pragma unroll
            for (int q = 0; q < 4; ++q)
              sts128(dst + (uint32_t)(j * 4 + q) * kLBO, o[4 * q], o[4 * q + 1], o[4 * q + 2], o[4 * q + 3]);
          }
          fence_proxy_async_smem();
        }
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(full0 + 8u * (uint32_t)(n % kAStages));
        // Every value loaded from the code stage has been consumed.
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bars->code_empty[s]));
      }
      if (*abort_flag) ok = false;
    }
  } else {
    // ---------------- epilogue ----------------
    const int q = warp & 3;                      // TMEM lane quarter
    const int ew = warp - kFirstEpi, half = ew >> 2;
    const bool elected = elect_one();
    griddep_wait();
    // Parts of a split K are stored unscaled: sum_parts_kernel scales their sum.
    const float sa = splits > 1 ? 1.0f : 0.25f * a_ts[0], sb = splits > 1 ? 1.0f : b_ts[0];
    const u64 sa2 = pack2(sa, sa), sb2 = pack2(sb, sb);
    const uint32_t acc_empty0 = mapa_shared(smem_u32(&bars->acc_empty[0]), 0);
    const uint32_t stage = sbase + OFF_EPI + (uint32_t)ew * EPI_BYTES;
    const uint32_t wr_off = (uint32_t)lane * 64u, wr_swz = (uint32_t)(lane >> 1) & 3u;
    const int steps = tile_n / EPI_CHUNK;        // even; this warp takes every second one
    for (int i = 0; work.next(t, k0, k1); ++i) {
      const bool whole = work.sched.store;       // first chunk of a whole tile: stored, else added
      // An add into C must follow the earlier segments' stores into the tile.
      if (!whole && c_tma && elected) bulk_wait_all();
      const int ab = i & 1;
      const bool acc_ok =
          mbar_wait_cluster(smem_u32(&bars->acc_full[ab]), (uint32_t)(i >> 1) & 1u, abort_flag, kWaitLimitNs);
      tc_fence_after();
      const bool go = __all_sync(0xffffffffu, acc_ok && !*abort_flag);
      if (!go) {
        if (!acc_ok && !*abort_flag) fail(64u);
        break;
      }
      const int row0 = (t / ntiles_n) * TILE_M + (int)rank * BM + q * 32;
      const int out0 = row0 + work.part * ((M + 31) & ~31);  // row in the output of this part of K
      const int n0 = (t % ntiles_n) * tile_n;
      const uint32_t tbase = tmem_base + (uint32_t)ab * kAccCols + ((uint32_t)(q * 32) << 16);
#pragma unroll 1
      for (int cc = half; cc < steps; cc += 2) {
        uint32_t o[EPI_CHUNK];
        tmem_ld_32x32b_x16(tbase + (uint32_t)(cc * EPI_CHUNK), o);
        tmem_ld_wait_x16(o);
        if (cc + 2 >= steps) {
          // This warp's share of the accumulator sits in registers.
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(acc_empty0 + 8u * (uint32_t)ab);
        }
#pragma unroll
        for (int k = 0; k < EPI_CHUNK; k += 2) {  // (acc x sa) x sb, two columns per instruction
          const u64 v = mul2(mul2(bits2(o[k], o[k + 1]), sa2), sb2);
          o[k] = (uint32_t)v;
          o[k + 1] = (uint32_t)(v >> 32);
        }
        const int col = n0 + cc * EPI_CHUNK;
        if (c_tma) {
          if (elected) bulk_wait_read_all();  // the previous step's store has read the tile
          __syncwarp();
#pragma unroll
          for (int j = 0; j < 4; ++j)
            sts128(stage + wr_off + (((uint32_t)j ^ wr_swz) << 4), o[4 * j], o[4 * j + 1], o[4 * j + 2],
                   o[4 * j + 3]);
          fence_proxy_async_smem();
          __syncwarp();
          if (elected) {
            if (row0 < M && col < N) {
              if (whole) tma_store_2d(&tm_c, stage, col, out0);
              else tma_reduce_add_2d(&tm_c, stage, col, out0);
            }
            bulk_commit_group();
          }
        } else if (row0 + lane < M) {
          float* crow = C + (long long)(row0 + lane) * ldc + col;
          for (int k = 0; k < EPI_CHUNK; ++k)
            if (col + k < N) {
              if (whole) crow[k] = __uint_as_float(o[k]);
              else atomicAdd(crow + k, __uint_as_float(o[k]));
            }
        }
      }
    }
    if (c_tma && elected) bulk_wait_all();
  }

  tc_fence_before();
  cluster_sync();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, kTmemCols);
  }
}

// C = factor x s32A x s32B x the sum of the parts of a split product (part_stride
// floats apart, rows of ldp floats), four columns per thread.  The sum carries its rounding errors along
// (Knuth's two-sum), so splitting K costs no accuracy: on 100 x 512 x 14336 the
// parts added into C one by one in fp32 left twice the error of one pass.
__global__ void __launch_bounds__(256)
sum_parts_kernel(const float* parts, int splits, long long part_stride, int ldp, float factor, const float* a_ts,
                 const float* b_ts, int M, int N, float* __restrict__ C, long long ldc, int vec) {
  griddep_wait();
  griddep_launch_dependents();
  const float sa = factor * a_ts[0], sb = b_ts[0];  // factor: a power of two
  const int q_n = (N + 3) / 4;
  const long long n = (long long)M * q_n;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const int m = (int)(i / q_n), c = (int)(i - (long long)m * q_n) * 4;
    const float* p = parts + (long long)m * ldp + c;
    float s[4] = {0.0f, 0.0f, 0.0f, 0.0f}, e[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 8
    for (int j = 0; j < splits; ++j) {
      const float4 v4 = *reinterpret_cast<const float4*>(p + j * part_stride);
      const float v[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
      for (int k = 0; k < 4; ++k) two_sum_add(s[k], e[k], v[k]);
    }
    float o[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) o[k] = __fmul_rn(__fmul_rn(__fadd_rn(s[k], e[k]), sa), sb);
    float* dst = C + m * ldc + c;
    if (vec && c + 4 <= N) {
      *reinterpret_cast<float4*>(dst) = make_float4(o[0], o[1], o[2], o[3]);
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (c + k < N) dst[k] = o[k];
    }
  }
}

}  // namespace fa
}  // namespace

int launch_decode_f16(const uint8_t* codes, const uint8_t* scales, int64_t rows, int64_t K, void* out,
                      cudaStream_t stream) {
  const int64_t nchunks = rows * (K / 32);
  int64_t grid = (nchunks + 255) / 256;
  if (grid > num_sms() * 8) grid = num_sms() * 8;
  if (grid == 0) return 0;
  return launch_pdl(decode_f16_kernel, (unsigned)grid, 256, 0, stream, codes, scales, nchunks,
                    static_cast<uint8_t*>(out)) == cudaSuccess ? 0 : -1;
}

// Whether decoding A in a pass of its own pays against decoding it in the main
// loop (gemm.cu).  A 64-K stage of the main loop is about 0.07 us shorter with
// A decoded (0.335 -> 0.265 us on 2048 x 4096 x 4096), and the pass costs about
// 1.8 us plus 0.45 us per million elements of A.  Both sides measured: 2048 x 4096
// x 4096 51.5 -> 43.3 us, 1500 x 5000 x 2560 36.0 -> 31.5, 777 x 3000 x 2816
// 20.4 -> 19.4; against it 663 x 5056 x 1792 17.0 -> 18.2, 3000 x 500 x 1024
// 12.3 -> 13.3, 8000 x 300 x 8192 47 -> 68 us.
bool gemm_predecode_pays(int64_t M, int64_t N, int64_t K) {
  const int64_t pairs = num_sms() / 2, tiles = (M + 255) / 256 * ((N + 255) / 256);
  const double stages = (double)((tiles + pairs - 1) / pairs) * (double)(K / 64);
  return 0.07 * stages > 1.8 + 0.45e-6 * (double)M * (double)K;
}

// The same for the layer (M > 64): whether the quantizer writes f16 values, 2 bytes
// an element, for this GEMM, or codes and scales, 0.56 bytes, for gemm.cu's.  Here
// no pass is saved by the codes, only bytes, so this GEMM is the rule.  With one
// column of tiles (N <= 256) gemm.cu decodes A only once as well, and this GEMM has
// nothing over it but its split of K, for up to half a wave of tiles.  f16 / codes,
// L2 flushed, us: 32768 x 64 x 4096 209 / 190, 32768 x 256 x 8192 409 / 363, 16384 x 256 x
// 2560 79 / 75; with K split or below 2^25 elements 8192 x 64 x 14336 190 / 203,
// 20000 x 64 x 1024 46 / 48, 65536 x 64 x 256 42 / 46; with two columns 32768 x 300 x 8192
// 429 / 437, 16384 x 384 x 4096 130 / 126.
bool linear_predecode_pays(int64_t M, int64_t N, int64_t K) {
  const int64_t pairs = num_sms() / 2, tiles = (M + 255) / 256;
  return N > 256 || 2 * tiles <= pairs || M * K < (1ll << 25);
}

namespace {

struct Plan {
  int tile_n, splits, kps;  // kps: 256-K slices per part (all of them when splits is 1)
  int64_t dp_tiles, tiles;
};

int64_t parts_bytes(int64_t M, int64_t N, int splits) {
  return splits > 1 ? (int64_t)splits * ((M + 31) / 32 * 32) * ((N + 3) / 4 * 4) * 4 : 0;
}

// Tile width and K split.  A 64-K stage takes about 340 + 7 n / 8 cycles at
// width n (measured over 2048 x 4096 x 4096 at every width: 560 at 256, 520 at
// 224, 450 at 160, 415 at 96; the tensor pipe alone is 2 n), so a width costs
// its waves times that.  Two ways to use pairs that would idle:
// - a partial last wave's K slices shared out over all pairs (stream-K: C rows
//   zeroed, partial sums added), about 17000 cycles (the zeroing kernel, one more
//   drain and the adds: 7.5 to 10 us over ten shapes.  256-wide tiles whole / split,
//   L2 flushed, us: 2560 x 4096 x 4096 71.7 / 62.9, 3072 x 4096 x 4096 72.9 / 72.6,
//   4096 x 4096 x 2304 59.5 / 61.5; at 4096^3 93.3 / 89.4, and 85.1 as whole 224-wide
//   tiles, which the plan takes);
// - where the tiles do not fill one wave, K cut into parts that are summed by
//   sum_parts_kernel, if the caller's workspace holds the parts: about 8000
//   cycles plus the parts' traffic.
Plan make_plan(int64_t M, int64_t N, int64_t K, int64_t parts_room) {
  constexpr int64_t kStreamKCycles = 17000, kPartsCycles = 8000, kBytesPerCycle = 2400;
  const int64_t mtiles = (M + fa::TILE_M - 1) / fa::TILE_M, num_kc = K / fa::BKC, pairs = num_sms() / 2;
  Plan best{};
  int64_t best_cost = -1;
  auto consider = [&](int64_t cost, int n, int splits, int64_t kps, int64_t dp, int64_t t) {
    if (best_cost < 0 || cost < best_cost) {
      best_cost = cost;
      best = Plan{n, splits, (int)kps, dp, t};
    }
  };
  for (int n = 256; n >= 96; n -= 32) {
    const int64_t t = mtiles * ((N + n - 1) / n), full = t / pairs * pairs, rem = t - full;
    const int64_t slice = fa::kSub * (340 + 7 * n / 8);
    consider((t + pairs - 1) / pairs * num_kc * slice, n, 1, num_kc, t, t);
    if (full > 0 && rem > 0)
      consider((full / pairs * num_kc + (rem * num_kc + pairs - 1) / pairs) * slice + kStreamKCycles, n, 1, num_kc, full,
               t);
    if (2 * t > pairs) continue;
    for (int64_t want = 2; want <= 16 && want <= num_kc; ++want) {
      const int64_t kps = (num_kc + want - 1) / want, splits = (num_kc + kps - 1) / kps;
      const int64_t bytes = parts_bytes(M, N, (int)splits);
      if (bytes > parts_room) break;
      consider((t * splits + pairs - 1) / pairs * kps * slice + kPartsCycles + 2 * bytes / kBytesPerCycle, n, (int)splits,
               kps, t, t);
    }
  }
  return best;
}

}  // namespace

// Scratch for the parts of a split K, beside the decoded A (0: K is not split).
int64_t gemm_f16a_parts_bytes(int64_t M, int64_t N, int64_t K) {
  return parts_bytes(M, N, make_plan(M, N, K, INT64_MAX).splits);
}

int launch_sum_parts(const float* parts, int splits, int64_t part_stride, int64_t ldp, float factor, const float* a_ts,
                     const float* b_ts, int64_t M, int64_t N, float* C, int64_t ldc, cudaStream_t stream) {
  const int vec = ((ldc & 3) == 0) && ((reinterpret_cast<uintptr_t>(C) & 15) == 0);
  int64_t grid = (M * ((N + 3) / 4) + 255) / 256;
  if (grid > num_sms() * 8) grid = num_sms() * 8;
  return launch_pdl(fa::sum_parts_kernel, (unsigned)grid, 256, 0, stream, parts, splits, (long long)part_stride,
                    (int)ldp, factor, a_ts, b_ts, (int)M, (int)N, C, (long long)ldc, vec) == cudaSuccess
             ? MIXFP4_OK
             : MIXFP4_ERR_CUDA;
}

int launch_gemm_f16a(const void* a_f16, const float* a_ts, const uint8_t* b_codes, const uint8_t* b_scales,
                     const float* b_ts, int64_t M, int64_t N, int64_t K, float* C, int64_t ldc, void* parts,
                     int64_t parts_room, uint32_t* status_word, cudaStream_t stream) {
  if (M > (1 << 30) || N > (1 << 30) || K > (1 << 30)) return MIXFP4_ERR_SHAPE;
  const int64_t num_kc = K / fa::BKC, pairs = num_sms() / 2;
  const Plan p = make_plan(M, N, K, parts ? parts_room : 0);
  const int64_t ntiles_n = (N + p.tile_n - 1) / p.tile_n;
  const int64_t units = p.dp_tiles < p.tiles ? p.tiles * num_kc : p.tiles * p.splits;
  const int64_t clusters = units < pairs ? units : pairs;
  CUtensorMap ta, tbc, tbs, tmc;
  if (!make_map_f16(&ta, a_f16, (uint64_t)K, (uint64_t)M, fa::BKS, fa::BM, CU_TENSOR_MAP_SWIZZLE_128B) ||
      !make_map(&tbc, b_codes, (uint64_t)K / 2, (uint64_t)N, fa::BKC / 2, (uint32_t)p.tile_n / 2,
                CU_TENSOR_MAP_SWIZZLE_128B) ||
      !make_map(&tbs, b_scales, (uint64_t)K / 16, (uint64_t)N, fa::BKC / 16, (uint32_t)p.tile_n / 2,
                CU_TENSOR_MAP_SWIZZLE_NONE))
    return MIXFP4_ERR_CUDA;
  memset(&tmc, 0, sizeof(tmc));
  const int c_vec = ((ldc & 3) == 0) && ((reinterpret_cast<uintptr_t>(C) & 15) == 0);
  const int64_t m_pad = (M + 31) / 32 * 32, ldp = (N + 3) / 4 * 4;
  int c_tma = c_vec;
  if (p.splits > 1) {
    c_tma = 1;
    if (!make_map_f32(&tmc, static_cast<float*>(parts), (uint64_t)N, (uint64_t)(p.splits * m_pad), (uint64_t)ldp,
                      fa::EPI_CHUNK, 32, CU_TENSOR_MAP_SWIZZLE_64B))
      return MIXFP4_ERR_CUDA;
  } else if (c_tma && !make_map_f32(&tmc, C, (uint64_t)N, (uint64_t)M, (uint64_t)ldc, fa::EPI_CHUNK, 32,
                                    CU_TENSOR_MAP_SWIZZLE_64B)) {
    return MIXFP4_ERR_CUDA;
  }
  static std::atomic<uint64_t> smem_set{0};
  if (!set_dynamic_smem_once(reinterpret_cast<const void*>(fa::gemm_f16a_kernel), fa::SMEM_ALLOC, smem_set))
    return MIXFP4_ERR_CUDA;
  if (p.dp_tiles < p.tiles) {
    // Zero C from the first split tile's row band down (whole tiles among those
    // rows are overwritten by plain stores after this).
    const int64_t r0 = (p.dp_tiles / ntiles_n) * fa::TILE_M;
    if (launch_zero_rows(C + r0 * ldc, M - r0, N, ldc, stream) != 0) return MIXFP4_ERR_CUDA;
  }
  if (launch_pdl(fa::gemm_f16a_kernel, (unsigned)(2 * clusters), fa::kThreads, fa::SMEM_ALLOC, stream, ta, tbc, tbs,
                 tmc, c_tma, a_ts, b_ts, (int)M, (int)N, (int)K, C, (long long)ldc, p.tile_n, (int)p.dp_tiles,
                 kAccumChunkK / fa::BKC, p.splits, p.kps, p.dp_tiles < p.tiles ? 1 : 0, status_word) != cudaSuccess)
    return MIXFP4_ERR_CUDA;
  if (p.splits > 1)
    return launch_sum_parts(static_cast<const float*>(parts), p.splits, m_pad * ldp, ldp, 0.25f, a_ts, b_ts, M, N, C,
                            ldc, stream);
  return MIXFP4_OK;
}

}  // namespace mixfp4
