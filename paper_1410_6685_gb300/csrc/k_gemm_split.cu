// k_gemm_split.cu -- the binary32 matrix product (Sec. 3.4 `multiply`,
// SG_PREC_F32_SIMT) of larger sizes on the 5th-generation tensor cores
// (sm_103a): C = A B (or C = C - A B, the elimination's update).
//
// Every binary32 operand is split exactly into three bf16 pieces, x = x1 +
// x2 + x3 (24 = 8 + 8 + 8 significant bits; x2 and x3 round to nearest what
// is left), and the product is the sum of the six piece products that matter
// -- x1 y1, x1 y2, x2 y1, x2 y2, x1 y3, x3 y1 -- each exact in binary32.  What
// is left out, x2 y3 + x3 y2 + x3 y3, is at most 2^-24 of |x y| (|x2| <= 2^-8
// |x|, |x3| <= 2^-17 |x|), one binary32 rounding, and 2^-27.4 by its mean square.
//
// The tensor core does not round its sums: it aligns the 16 products of a step
// and the accumulator to the largest, keeps two bits below binary32's, and
// truncates (measured).  A long sum kept there drifts toward zero, and a
// single product that meets its smaller ones there is not rounded to nearest.
// Hence two accumulators:
//   x1 y1          : TK = 32 consecutive k, two truncations; the epilogue warps
//                    take each chunk's sum out of tensor memory and add it,
//                    rounding to nearest, to a running sum in registers while the
//                    tensor core goes on with the next chunk;
//   the other five : some 2^-7 of the whole at most, so that their truncations weigh
//                    as much less, and their signs are x2's and y2's, not the
//                    products'; kept for 2048 k (a pair: 8192), then added.
// Per entry the error is within (24 + K / 16) 2^-24 of sum |a b| (2^-20 + 2^-22 for
// the truncations of x1 y1, 2^-24 for what is left out, K / 32 roundings, and
// K 2^-29 for the truncations of the other five); the CUDA cores' chain of K
// roundings K 2^-24.  Norm of the error against the product's, CUDA cores / here:
// N(0,1) at 1000 5.7e-7 / 1.2e-7, at 4096 1.15e-6 / 2.2e-7; U[0,1) at 4096 8.4e-7 /
// 1.6e-7; 64 / 16 / 4 / 2 non-zeros per row of A 14 / 7.4 / 4.0 / 3.1e-8 against 5.6 /
// 3.4 / 2.7 / 2.6e-8; one 2.53e-8 (each entry rounded once) against 2.59e-8; exp(4 N(0,1))
// at 1000 4.4e-8 against 5.1e-8 (of sum |a b|, entry by entry, 2.5e-7 against 0.9e-7),
// at 2048 4.6 and 4.6e-8.  With all six products in one accumulator, no
// faster, the sparse ones were 11-14 / 8.6 / 6.0 / 5.2e-8 and 4.5e-8.
//
// The tensor pipe bounds it: six bf16 multiply-adds per binary32 one, so a
// sixth of the bf16 rate, about 317 TFLOP/s of measured, where the CUDA
// cores' form (k_gemm_simt.cu) reaches 44-49.
//
// Range: pieces and piece products stay normal numbers for |x| = 0 or
// 2^-50 <= |x| < 2^55.  The cast kernels raise a flag for any other value
// (subnormals, infinities, NaN, extreme scales); then this kernel does
// nothing and the CUDA-core form, queued behind it, computes the product.
#include <cuda.h>

#include <algorithm>

#include "sg_linalg_kernels.h"
#include "sg_tcgen05.cuh"

namespace sgk {
namespace {

using namespace tc;

constexpr int TK = 32;        // k per pipeline stage and per accumulation of x1 y1
constexpr int kEpiWarps = 8;
constexpr int kThreads = 96 + 32 * kEpiWarps;   // producer, two MMA issuers, epilogue
constexpr int T_BYTES = kEpiWarps * 16 * 32 * 4;

// Tile forms.  PAIR: a CTA pair computes 256 x TN (each CTA 128 rows of A and
// TN / 2 rows of B^T per stage); else one CTA computes 128 x TN.  Each MMA issuer
// has 2 TN columns of tensor memory: an accumulator for x1 y1, one for the other
// products.
template <bool PAIR, int TN>
struct Form {
  static constexpr int kBRows = PAIR ? TN / 2 : TN;
  static constexpr int kAPiece = 128 * TK * 2;
  static constexpr int kBPiece = kBRows * TK * 2;
  static constexpr int kStageBytes = 3 * (kAPiece + kBPiece);
  static constexpr int kTileM = PAIR ? 256 : 128;
  // (one issuer's 256-column accumulators fill the tensor memory)
  static constexpr int kIssuers = TN == 256 ? 1 : 2;
  static constexpr int kColumns = kIssuers * 2 * TN;
  // chunks of an issuer per accumulation of the other products
  static constexpr int kLong = (kIssuers == 1 ? 8192 : 2048) / TK / kIssuers;
  static constexpr int kStages = (232448 - 1024 - 256 - T_BYTES) / kStageBytes;   // 4 or 5
  static constexpr int kSmem = kStages * kStageBytes + 1024 + 256 + T_BYTES;
  // kind::f16, D f32, A / B bf16, both K-major
  static constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) |
                                     ((uint32_t)(TN >> 3) << 17) |
                                     ((uint32_t)(kTileM >> 4) << 24);
};

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y,
                                            int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const CUtensorMap* map, int x,
                                                 int y, int z, uint32_t bar_cl) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar_cl)
      : "memory");
}

// 16 columns of the warp's 32 tensor-memory lanes (16, not 32: the running
// sums already hold up to 128 registers)
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
        "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// shared-memory descriptor of a K-major tile in the 64-byte swizzle layout
// (rows of 64 B, 8-row groups 512 B apart)
__device__ __forceinline__ uint64_t sdesc64(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);   // start address >> 4
  d |= (uint64_t)1 << 16;                      // leading byte offset (unused here)
  d |= (uint64_t)(512 >> 4) << 32;             // stride byte offset: 8 rows x 64 B
  d |= (uint64_t)1 << 46;                      // descriptor version
  d |= (uint64_t)4 << 61;                      // 64-byte swizzle
  return d;
}

// Persistent, roles as in k_gemm_tc / k_gemm_tc2: warp 0 TMA producer, warps 1
// and (one-CTA forms) 10 MMA issuers, warps 2..9 epilogue (lane quarter warp % 4,
// column half (warp - 2) / 4).  Chunks of all tiles are numbered in one sequence;
// with two issuers chunk it uses the accumulators of issuer it & 1.  gate[0] != 0 or
// skip[0] != 0 (each written by earlier launches): nothing is done.
template <bool PAIR, int TN, bool SUB>
__global__ void __launch_bounds__(kThreads, 1)
    k_gemm_split(const __grid_constant__ CUtensorMap ma, const __grid_constant__ CUtensorMap mb,
                 float* __restrict__ C, int ldc, int M, int N, int KB, const int* gate, const int* skip,
                 int* err) {
  using F = Form<PAIR, TN>;
  constexpr int HN = TN / 2;                  // columns per epilogue warp
  constexpr int NC = HN / 32;                 // 32-column groups of the store
  constexpr int kStages = F::kStages;
  if (*gate != 0 || (skip && *skip != 0)) return;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kStages * F::kStageBytes);
  // bars[0..S): stage full, [S..2S): stage done (its MMAs have completed),
  // [2S, 2S+2): an issuer's accumulators empty (one issuer: that of x1 y1, that of
  // the other products), [2S+2]: drain
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kStages + 3);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  float* s_t = reinterpret_cast<float*>(smem + kStages * F::kStageBytes + 256);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = PAIR ? cluster_rank() : 0;
  const int unit = PAIR ? blockIdx.x >> 1 : blockIdx.x;
  const int nunits = PAIR ? gridDim.x >> 1 : gridDim.x;
  const int nN = (N + TN - 1) / TN, nM = (M + F::kTileM - 1) / F::kTileM;
  const int ntiles = nN * nM;
  const uint32_t stage0 = smem_u32(smem), full0 = smem_u32(bars), done0 = full0 + 8 * kStages;
  const uint32_t tempty0 = done0 + 8 * kStages, drain_bar = tempty0 + 16;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(full0 + 8 * s, PAIR ? 2 : 1);
      mbar_init(done0 + 8 * s, 1);
    }
    mbar_init(tempty0, (PAIR ? 2 : 1) * kEpiWarps);
    mbar_init(tempty0 + 8, (PAIR ? 2 : 1) * kEpiWarps);
    mbar_init(drain_bar, F::kIssuers);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 2) {
    if (PAIR) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                       smem_u32(tmem_slot)), "r"(F::kColumns) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                       smem_u32(tmem_slot)), "r"(F::kColumns) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  if (PAIR) cluster_sync(); else __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      int it = 0;
      bool ok = true;
      for (int t = unit; t < ntiles && ok; t += nunits) {
        int bm, bn;
        tile_coords(t, nM, nN, &bm, &bn, SUB);
        const int m0 = bm * F::kTileM + (int)rank * 128;
        const int n0 = bn * TN + (int)rank * F::kBRows;
        for (int kb = 0; kb < KB; ++kb, ++it) {
          const int s = it % kStages;
          const uint32_t ph = (uint32_t)(it / kStages) & 1u;
          if (it >= kStages &&
              !mbar_wait_ab(done0 + 8 * s, ph ^ 1u, err, abort_flag)) {
            ok = false;
            break;
          }
          const uint32_t dst = stage0 + (uint32_t)(s * F::kStageBytes);
          if (PAIR) {
            const uint32_t full = map_rank(full0 + 8 * s, 0);
            mbar_expect_tx_cl(full, F::kStageBytes);
#pragma unroll
            for (int p = 0; p < 3; ++p) {
              tma_load_3d_pair(dst + p * F::kAPiece, &ma, kb * TK, m0, p, full);
              tma_load_3d_pair(dst + 3 * F::kAPiece + p * F::kBPiece, &mb, kb * TK, n0, p, full);
            }
          } else {
            const uint32_t full = full0 + 8 * s;
            mbar_expect_tx(full, F::kStageBytes);
#pragma unroll
            for (int p = 0; p < 3; ++p) {
              tma_load_3d(dst + p * F::kAPiece, &ma, kb * TK, m0, p, full);
              tma_load_3d(dst + 3 * F::kAPiece + p * F::kBPiece, &mb, kb * TK, n0, p, full);
            }
          }
        }
      }
    }
  } else if (warp == 1 || warp == 2 + kEpiWarps) {
    // Per chunk the five smaller products into their accumulator, which goes on
    // for kLong chunks, then x1 y1 into its own.  One-CTA forms: two issuer warps,
    // taking turns by chunk, each with its accumulators, since a chunk's two waits
    // and its commit take about 470 clocks, in which the tensor pipe ran dry behind
    // a single issuer.  A pair's chunk runs for 1536 clocks: one issuer suffices,
    // and x1 y1 is drained while the next chunk's other products run.  The whole
    // warp runs the loop and one elected lane issues, so that the descriptors stay
    // in uniform registers: with a lone diverged lane each tcgen05.mma took 68
    // clocks to issue, more than a 64-column one takes to run.  A chunk's commit
    // releases its stage to the producer and hands its accumulators to the
    // epilogue (both wait on it).
    if (rank == 0 && (F::kIssuers == 2 || warp == 1)) {
      const int acc = warp == 1 ? 0 : 1;
      const uint32_t dbig = tmem + (uint32_t)(acc * 2 * TN), dsmall = dbig + TN;
      int it = 0, s = 0, longs = 0;
      uint32_t ph = 0;
      bool ok = true, full = false;   // full: this chunk's stage is known to be
      auto mma = [&](uint32_t d, int pa, int pb, int k, uint64_t da0, uint64_t db0, bool add) {
        // 16 elements (32 bytes) along K inside the swizzled rows
        const uint64_t da = da0 + (uint64_t)((pa * F::kAPiece >> 4) + 2 * k);
        const uint64_t db = db0 + (uint64_t)((pb * F::kBPiece >> 4) + 2 * k);
        if (PAIR)
          umma2(d, da, db, F::kIdesc, add);
        else
          umma(d, da, db, F::kIdesc, add);
      };
      // the lanes give up together
      auto wait = [&](uint32_t bar, uint32_t parity) {
        return __all_sync(0xffffffffu, mbar_wait_ab(bar, parity, err, abort_flag)) != 0;
      };
      for (int t = unit; t < ntiles && ok; t += nunits) {
        for (int kb = 0; kb < KB; ++kb, ++it) {
          if (F::kIssuers == 2 && (it & 1) != acc) {   // the other issuer's chunk
            if (++s == kStages) {
              s = 0;
              ph ^= 1u;
            }
            continue;
          }
          const bool fresh = kb / F::kIssuers % F::kLong == 0;
          if (!full) ok = wait(full0 + 8 * s, ph);
          full = false;
          if (F::kIssuers == 2) {
            if (ok && it >= 2) ok = wait(tempty0 + 8 * acc, (uint32_t)((it >> 1) - 1) & 1u);
          } else if (fresh) {
            if (ok && longs > 0) ok = wait(tempty0 + 8, (uint32_t)(longs - 1) & 1u);
            ++longs;
          }
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint64_t da0 = sdesc64(stage0 + (uint32_t)(s * F::kStageBytes));
          const uint64_t db0 = da0 + (uint64_t)(3 * F::kAPiece >> 4);
          if (elect_one()) {
            constexpr int pa[5] = {2, 0, 1, 1, 0}, pb[5] = {0, 2, 1, 0, 1};
#pragma unroll
            for (int p = 0; p < 5; ++p)
#pragma unroll
              for (int k = 0; k < TK / 16; ++k)
                mma(dsmall, pa[p], pb[p], k, da0, db0, !fresh || (p | k) != 0);
          }
          __syncwarp();
          if (F::kIssuers == 1) {
            // the next stage first: between the wait for the accumulator and the
            // next chunk's products there is then none (4096^3: 477 -> 455 us)
            if (kb + 1 < KB || t + nunits < ntiles)
              ok = full = wait(full0 + 8 * (s + 1 == kStages ? 0 : s + 1),
                               s + 1 == kStages ? ph ^ 1u : ph);
            if (ok && it >= 1) ok = wait(tempty0, (uint32_t)(it - 1) & 1u);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          }
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < TK / 16; ++k) mma(dbig, 0, 0, k, da0, db0, k != 0);
            if (PAIR) umma_commit_pair(done0 + 8 * s);
            else umma_commit(done0 + 8 * s);
          }
          __syncwarp();
          if (++s == kStages) {
            s = 0;
            ph ^= 1u;
          }
        }
      }
      // completes when every MMA issued above has finished
      if (elect_one()) {
        if (PAIR) umma_commit_pair(drain_bar);
        else umma_commit(drain_bar);
      }
      __syncwarp();
    }
  } else {
    const int q = warp & 3, hh = (warp - 2) >> 2;
    float* s_tw = s_t + (warp - 2) * 16 * 32;
    const uint32_t tempty_cl = PAIR ? map_rank(tempty0, 0) : 0;
    const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(hh * HN);
    int ch = 0, s = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int t = unit; t < ntiles && ok; t += nunits) {
      int bm, bn;
      tile_coords(t, nM, nN, &bm, &bn, SUB);
      const int m0q = bm * F::kTileM + (int)rank * 128 + q * 32, c0 = bn * TN + hh * HN;
      if (SUB) prefetch_c_row(C, ldc, M, N, m0q + lane, c0, HN);
      // of x1 y1, and of the other products, which a pair (its sums already take
      // 128 registers) adds to the same at the end
      constexpr int HS = F::kIssuers == 2 ? HN : 1;
      float sum[HN], small[HS];
#pragma unroll
      for (int j = 0; j < HN; ++j) sum[j] = 0.0f;
#pragma unroll
      for (int j = 0; j < HS; ++j) small[j] = 0.0f;
      // adds this warp's part of an accumulator; once it is drained, the warp
      // arrives on `bar` (no bar: 0)
      auto drain = [&](float* to, uint32_t col, uint32_t bar, uint32_t bar_cl) {
#pragma unroll
        for (int c = 0; c < HN / 16; ++c) {
          uint32_t r[16];
          tmem_ld16(lane_addr + col + (uint32_t)(c * 16), r);
          if (bar && c == HN / 16 - 1) {
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) {
              if (PAIR) mbar_arrive_cl(bar_cl);
              else mbar_arrive(bar);
            }
          }
#pragma unroll
          for (int j = 0; j < 16; ++j) to[c * 16 + j] += __uint_as_float(r[j]);
        }
      };
#pragma unroll 1
      for (int i = 0; i < KB; ++i, ++ch) {
        const int acc = F::kIssuers == 2 ? ch & 1 : 0;
        if (!mbar_wait_ab(done0 + 8 * s, ph, err, abort_flag)) {
          ok = false;
          break;
        }
        if (++s == kStages) {
          s = 0;
          ph ^= 1u;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t col = (uint32_t)(acc * 2 * TN);
        // the issuer's last chunk of the tile, or of a long accumulation
        const bool both = i + F::kIssuers >= KB || i / F::kIssuers % F::kLong == F::kLong - 1;
        if (F::kIssuers == 2 && both) drain(small, col + TN, 0u, 0u);
        drain(sum, col, tempty0 + 8 * acc, tempty_cl + 8 * acc);
        if (F::kIssuers == 1 && both) drain(sum, col + TN, tempty0 + 8, tempty_cl + 8);
      }
      if (!ok) break;
      if (F::kIssuers == 2) {
#pragma unroll
        for (int j = 0; j < HS; ++j) sum[j] += small[j];
      }
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        float4 cv[8];
        if (SUB) load_c(C, ldc, M, N, m0q, c0 + c * 32, lane, cv);
        uint32_t r[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) r[j] = __float_as_uint(sum[c * 32 + j]);
        store_chunk<SUB>(C, ldc, M, N, m0q, c0 + c * 32, r, s_tw, lane, cv);
      }
    }
  }
  __syncthreads();
  if (warp == 2) {
    // every MMA has completed before the tensor memory is released
    mbar_wait(drain_bar, 0, err);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (PAIR)
      asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                   "r"(F::kColumns) : "memory");
    else
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                   "r"(F::kColumns) : "memory");
  }
  // neither CTA leaves while the other may still signal its barriers
  if (PAIR) cluster_sync();
}

// the pieces [3][rows][Kp], boxes of TK x box_rows of one piece; rows past
// the end read as zero
bool make_map3(CUtensorMap* m, const void* base, int rows, int Kp, int box_rows) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[3] = {(cuuint64_t)Kp, (cuuint64_t)rows, 3};
  cuuint64_t strides[2] = {(cuuint64_t)Kp * 2, (cuuint64_t)rows * Kp * 2};
  cuuint32_t box[3] = {(cuuint32_t)TK, (cuuint32_t)box_rows, 1};
  cuuint32_t es[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box,
            es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <bool PAIR, int TN, bool SUB>
cudaError_t launch_form(const uint16_t* a3, const uint16_t* b3, int Kp, float* C, int ldc, int M,
                        int N, int K, const int* gate, const int* skip, int* err, cudaStream_t s) {
  using F = Form<PAIR, TN>;
  CUtensorMap ma, mb;
  if (!make_map3(&ma, a3, M, Kp, 128) || !make_map3(&mb, b3, N, Kp, F::kBRows))
    return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(k_gemm_split<PAIR, TN, SUB>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, F::kSmem);
  if (e != cudaSuccess) return e;
  const long long tiles = (long long)((M + F::kTileM - 1) / F::kTileM) * ((N + TN - 1) / TN);
  const int units = (int)std::min<long long>(tiles, PAIR ? sm_count() / 2 : sm_count());
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((PAIR ? 2 : 1) * units);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = F::kSmem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  if (PAIR) {
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
  }
  return cudaLaunchKernelEx(&cfg, k_gemm_split<PAIR, TN, SUB>, ma, mb, C, ldc, M, N, (K + TK - 1) / TK,
                            gate, skip, err);
}

template <bool SUB>
cudaError_t launch_split(int form, const uint16_t* a3, const uint16_t* b3, int Kp, float* C,
                         int ldc, int M, int N, int K, const int* gate, const int* skip, int* err,
                         cudaStream_t s) {
  if constexpr (!SUB)
    if (form == 2) return launch_form<true, 256, SUB>(a3, b3, Kp, C, ldc, M, N, K, gate, skip, err, s);
  return form ? launch_form<false, 128, SUB>(a3, b3, Kp, C, ldc, M, N, K, gate, skip, err, s)
              : launch_form<false, 64, SUB>(a3, b3, Kp, C, ldc, M, N, K, gate, skip, err, s);
}

// Estimated microseconds of the product in each tile form, and the form with
// the least: waves of tiles times (chunks of 32 k, and the tile's start and
// store).  Measured per chunk: 0.40 us (128 x 64), 0.48 us (128 x 128), 0.84 us
// (a pair's 256 x 256), so the larger tiles win once they fill the chip: at
// 1000^3 20.1 / 22.1 / 37.5 us, at 2048^3 110 / 65.1 / 63.8 us, at 8192^3 5487 /
// 3660 / 3150 us (349 TFLOP/s; the CUDA cores 22400 us).  Not a pair for the
// elimination's updates, whose K is 128 and whose C is read and written: between
// two tiles nothing is in flight in its accumulators (a determinant of n = 8192,
// binary32 updates, 6.79 ms by 128 x 128 tiles, 7.93 by pairs).
int choose_form(int M, int N, int K, bool subtract, double* us) {
  const double c = (K + TK - 1) / TK;
  auto waves = [&](int tm, int tn, int slots) {
    const long long t = (long long)((M + tm - 1) / tm) * ((N + tn - 1) / tn);
    return (double)((t + slots - 1) / slots);
  };
  const int sms = sm_count();
  const double t[3] = {6.5 + waves(128, 64, sms) * (0.40 * c + 1.5),
                       6.5 + waves(128, 128, sms) * (0.48 * c + 3.0),
                       !subtract && gemm_pair_available()
                           ? 7.0 + waves(256, 256, std::max(1, sms / 2)) * (0.84 * c + 5.0)
                           : 1e300};
  const int f = (int)(std::min_element(t, t + 3) - t);
  if (us) *us = t[f];
  return f;
}

}  // namespace

// Where the split product gains over the CUDA cores' form, by estimates of
// both: the casts stream 10 bytes per operand entry and cost two launches,
// the CUDA cores take 0.145 us per k up to one 128 x 128 tile per SM and 0.71
// ns per k and tile beyond (1000 x 1000 x 100: 20.3 us on the CUDA cores, 24 us
// split; 200^3: 34 against 26 us).  Not for K <= 64, where the CUDA cores'
// sum rounds as rarely, nor where the pieces would take more than 16 GB of
// scratch.
bool gemm_split_wanted(int M, int N, int K) {
  if (M <= 0 || N <= 0 || K <= 64) return false;
  if (gemm_split_scratch_bytes(M, N, K) > ((size_t)16 << 30)) return false;
  double split = 0.0;
  choose_form(M, N, K, false, &split);
  split += 11.0 + 10.0 * K * ((double)M + N) / 6.0e6;
  const double tiles = (double)((M + 127) / 128) * ((N + 127) / 128);
  const double simt = 3.0 + K * std::max(0.145, 0.00071 * tiles) + 4.0 * M * (double)N / 2.5e6;
  return split < simt;
}

size_t gemm_split_scratch_bytes(int M, int N, int K) {
  const size_t Kp = (size_t)((K + 63) / 64) * 64;
  return 256 + align256((size_t)M * Kp * 6) + align256((size_t)N * Kp * 6);
}

cudaError_t launch_gemm_split(const float* A, int lda, const float* B, int ldb, float* C, int ldc,
                              int M, int N, int K, bool subtract, void* scratch, cudaStream_t s,
                              Prof* prof, int64_t* kernels, int* err) {
  const int Kp = ((K + 63) / 64) * 64;
  char* p = static_cast<char*>(scratch);
  int* gate = reinterpret_cast<int*>(p);   // [0] out of range, [1] a wait gave up
  if (!err) err = gate + 1;
  uint16_t* a3 = reinterpret_cast<uint16_t*>(p + 256);
  uint16_t* b3 = reinterpret_cast<uint16_t*>(p + 256 + align256((size_t)M * Kp * 6));
  prof_begin(prof, "split_operands", s);
  cudaError_t e = cudaMemsetAsync(gate, 0, 8, s);
  if (e == cudaSuccess)
    e = launch_cast_operands<SG_PREC_F32_SIMT>(A, lda, B, ldb, M, N, K, Kp, a3, b3, gate, s);
  if (e != cudaSuccess) return e;
  prof_end(prof, s);
  prof_begin(prof, "gemm_f32_split", s);
  const int form = choose_form(M, N, K, subtract, nullptr);
  e = subtract ? launch_split<true>(form, a3, b3, Kp, C, ldc, M, N, K, gate, nullptr, err, s)
               : launch_split<false>(form, a3, b3, Kp, C, ldc, M, N, K, gate, nullptr, err, s);
  prof_end(prof, s);
  if (e != cudaSuccess) return e;
  *kernels += 3;
  return launch_gemm_f32(A, lda, B, ldb, C, ldc, M, N, K, subtract, s, prof, gate);
}

cudaError_t launch_gemm_split_operands(const uint16_t* a3, const uint16_t* b3, const float* A,
                                       int lda, const float* B, int ldb, float* C, int ldc, int M,
                                       int N, int K, const int* gate, const int* skip, int* err,
                                       cudaStream_t s, int64_t* kernels) {
  cudaError_t e = launch_split<true>(choose_form(M, N, K, true, nullptr), a3, b3, K, C, ldc, M, N, K,
                                     gate, skip, err, s);
  if (e != cudaSuccess) return e;
  *kernels += 2;
  return launch_gemm_f32(A, lda, B, ldb, C, ldc, M, N, K, true, s, nullptr, gate);
}

}  // namespace sgk
