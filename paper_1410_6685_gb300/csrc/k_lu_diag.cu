// k_lu_diag.cu -- elimination with partial pivoting where every pivot already
// stands on the diagonal (sm_103a).
//
// The general elimination (k_lu.cu) finds each column's pivot by an exchange
// between the CTAs of a cluster, one microsecond per column whatever the
// matrix: 154 of the 235 us that a 128-column outer block took at n = 8192.
// When no interchange will be needed, as for diagonally dominant matrices,
// the outer block is three launches instead of about eleven, on average 85 us
// at n = 8192 (28 + 18 + 43 by kernel; the factorisation 14.8 -> 5.4 ms), and
// 64 us with the next diagonal block beside the update (4.1 ms; 16-bit updates):
//   k_lu_diag_block : the 128 x 128 diagonal block, in one CTA's shared memory;
//   k_lu_border     : L21 = A21 U11^-1 and U12 = L11^-1 A12, 64 rows or columns
//                     per CTA, which also writes the trailing update's
//                     operands (bf16, fp16 or three bf16 pieces);
//   the trailing update A22 -= L21 U12 (k_gemm_tc.cu, k_gemm_split.cu).
// Every entry goes through the same operations in the same order as in the
// general form (a -= l_ik u_kj for increasing k, l = a (1 / u)), so the factors are
// the same bits, but for binary32 updates of trailing blocks that the general form
// leaves to the CUDA cores (gemm_split_wanted: order 1537 to 1792 on 152 SMs); here
// the border has written their pieces already.  Every candidate a_ik is compared
// with its pivot before it is scaled: one that is larger in magnitude (or NaN), or a
// zero pivot, raises `fail`; what is queued behind then does nothing and the caller
// factors the matrix by the general form.  k_anorm (k_lu.cu) chooses the form
// beforehand.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "sg_linalg_kernels.h"
#include "sg_lu.h"
#include "sg_lu_tri.cuh"
#include "sg_tcgen05.cuh"

namespace sgk {
namespace {

constexpr int kNB = kLuOuter;     // 128
constexpr int kP = kLuPanel;      // 32
constexpr int kS = kNB + 4;       // row stride of a 128-wide tile: 16-byte loads, conflict-free
constexpr int kDiagThreads = 768;   // three groups of eight warps, one per 32 rows left

// x := x U^-1 for one row of 32 entries (U: 32 x 32 upper, row stride kS,
// 16-byte aligned; rd its diagonal's reciprocals), by substitution in
// registers; bad: an entry larger than its pivot.
__device__ __forceinline__ bool upper_solve_row(const float* U, const float* rd, float (&x)[kP]) {
  bool bad = false;
#pragma unroll
  for (int j = 0; j < kP; ++j) {
    const float4* Uj = reinterpret_cast<const float4*>(U + j * kS);
    bad |= !(fabsf(x[j]) <= fabsf(U[j * kS + j]));
    const float l = x[j] * rd[j];
    x[j] = l;
#pragma unroll
    for (int g = (j + 1) / 4; g < kP / 4; ++g) {
      const float4 u = Uj[g];
      if (4 * g > j) x[4 * g] = fmaf(-l, u.x, x[4 * g]);
      if (4 * g + 1 > j) x[4 * g + 1] = fmaf(-l, u.y, x[4 * g + 1]);
      if (4 * g + 2 > j) x[4 * g + 2] = fmaf(-l, u.z, x[4 * g + 2]);
      if (4 * g + 3 > j) x[4 * g + 3] = fmaf(-l, u.w, x[4 * g + 3]);
    }
  }
  return bad;
}

// C(32 x 32 G) -= P(32 x 32) Q(32 x 32 G), q increasing; 8 warps: warp w takes
// rows w, w + 8, w + 16, w + 24, lane the column of each of the G groups.
template <int G>
__device__ __forceinline__ void update32(float* C, int cs, const float* P, int ps, const float* Q,
                                         int qs, int w, int lane) {
  float acc[4][G];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int u = 0; u < G; ++u) acc[i][u] = C[(w + 8 * i) * cs + lane + 32 * u];
#pragma unroll 2
  for (int q = 0; q < kP; q += 4) {
    float4 p[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) p[i] = *reinterpret_cast<const float4*>(P + (w + 8 * i) * ps + q);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      float v[G];
#pragma unroll
      for (int u = 0; u < G; ++u) v[u] = Q[(q + e) * qs + lane + 32 * u];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float pe = e == 0 ? p[i].x : e == 1 ? p[i].y : e == 2 ? p[i].z : p[i].w;
#pragma unroll
        for (int u = 0; u < G; ++u) acc[i][u] = fmaf(-pe, v[u], acc[i][u]);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int u = 0; u < G; ++u) C[(w + 8 * i) * cs + lane + 32 * u] = acc[i][u];
}

__device__ __forceinline__ void update32_any(int g, float* C, int cs, const float* P, int ps,
                                             const float* Q, int qs, int w, int lane) {
  if (g == 3) update32<3>(C, cs, P, ps, Q, qs, w, lane);
  else if (g == 2) update32<2>(C, cs, P, ps, Q, qs, w, lane);
  else update32<1>(C, cs, P, ps, Q, qs, w, lane);
}

// The KB x KB diagonal block at (K, K), in place.  A serial chain bounds it:
// per 32 columns the 32 x 32 factorisation in one warp's registers (lane =
// row), the rows below and the columns to the right
// one per thread, and the rest of the block by all.
__global__ void __launch_bounds__(kDiagThreads) k_lu_diag_block(float* __restrict__ LU, int n, int K,
                                                                int KB, int* __restrict__ piv,
                                                                const int* prev, const int* err,
                                                                int* fail) {
  if (__syncthreads_or(threadIdx.x == 0 && prev && (*prev | *err))) {
    if (threadIdx.x == 0) *fail = 1;
    return;
  }
  extern __shared__ __align__(16) float S[];   // [kNB][kS]
  float* rd = S + kNB * kS;                    // [kNB] reciprocal pivots
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  // (past KB: the identity) every load of a thread in flight at once
  {
    constexpr int kPer = (kNB * kNB + kDiagThreads - 1) / kDiagThreads;
    float v[kPer];
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int t = tid + i * kDiagThreads, r = t / kNB, c = t % kNB;
      v[i] = r < KB && c < KB ? __ldcg(LU + (size_t)(K + r) * n + K + c) : (r == c ? 1.0f : 0.0f);
    }
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int t = tid + i * kDiagThreads, r = t / kNB, c = t % kNB;
      if (r < kNB) S[r * kS + c] = v[i];
    }
  }
  __syncthreads();
  bool bad = false;
  for (int o = 0; o < kNB; o += kP) {
    float* D = S + o * kS + o;
    if (w == 0) {
      float x[kP];
      float4* row = reinterpret_cast<float4*>(D + lane * kS);
#pragma unroll
      for (int g = 0; g < kP / 4; ++g) {
        const float4 v = row[g];
        x[4 * g] = v.x; x[4 * g + 1] = v.y; x[4 * g + 2] = v.z; x[4 * g + 3] = v.w;
      }
      // Lane j's row is final at step j: it goes back to shared memory, which
      // is also how the other lanes read it.  What happens to a lane's
      // registers after its own step does not matter, so no lane is masked
      // (masking each update by lane made the compiler branch around every
      // one: 4700 clocks a column).
#pragma unroll
      for (int j = 0; j < kP; ++j) {
        const float d = __shfl_sync(0xffffffffu, x[j], j);
        if (lane == j)
#pragma unroll
          for (int g = 0; g < kP / 4; ++g)
            row[g] = make_float4(x[4 * g], x[4 * g + 1], x[4 * g + 2], x[4 * g + 3]);
        const float r = 1.0f / d;
        bad |= lane > j ? !(fabsf(x[j]) <= fabsf(d)) : !(fabsf(d) > 0.0f);
        const float l = x[j] * r;
        x[j] = l;
        if (lane == j) rd[o + j] = r;
        __syncwarp();
        const float4* Uj = reinterpret_cast<const float4*>(D + j * kS);
#pragma unroll
        for (int g = (j + 1) / 4; g < kP / 4; ++g) {
          const float4 u = Uj[g];
          if (4 * g > j) x[4 * g] = fmaf(-l, u.x, x[4 * g]);
          if (4 * g + 1 > j) x[4 * g + 1] = fmaf(-l, u.y, x[4 * g + 1]);
          if (4 * g + 2 > j) x[4 * g + 2] = fmaf(-l, u.z, x[4 * g + 2]);
          if (4 * g + 3 > j) x[4 * g + 3] = fmaf(-l, u.w, x[4 * g + 3]);
        }
      }
    }
    __syncthreads();
    const int rest = kNB - o - kP;
    if (tid < rest) {
      // one row below: l = a U^-1
      float4* row = reinterpret_cast<float4*>(S + (o + kP + tid) * kS + o);
      float x[kP];
#pragma unroll
      for (int g = 0; g < kP / 4; ++g) {
        const float4 v = row[g];
        x[4 * g] = v.x; x[4 * g + 1] = v.y; x[4 * g + 2] = v.z; x[4 * g + 3] = v.w;
      }
      bad |= upper_solve_row(D, rd + o, x);
#pragma unroll
      for (int g = 0; g < kP / 4; ++g)
        row[g] = make_float4(x[4 * g], x[4 * g + 1], x[4 * g + 2], x[4 * g + 3]);
    } else if (tid >= 128 && tid - 128 < rest) {
      // one column to the right: u = L^-1 a
      unit_lower_solve_col4(D, kS, S + o * kS + o + kP + tid - 128, kS);
    }
    __syncthreads();
    const int rb = o + kP + (w / 8) * kP;
    if (rb < kNB)
      update32_any(rest / kP, S + rb * kS + o + kP, kS, S + rb * kS + o, kS, S + o * kS + o + kP, kS,
                   w % 8, lane);
    __syncthreads();
  }
  for (int t = tid; t < KB * kNB; t += kDiagThreads) {
    const int r = t / kNB, c = t % kNB;
    if (c < KB) LU[(size_t)(K + r) * n + K + c] = S[r * kS + c];
  }
  if (tid < KB) piv[K + tid] = K + tid;
  if (bad) *fail = 1;
}

// The outer block's border.  The first CTAs take 64 rows each of A21 (L21 =
// A21 U11^-1), the others 64 columns each of A12 (U12 = L11^-1 A12); both hold
// the whole factored diagonal block in shared memory and go through it by 32
// columns (rows): one thread solves one row (column) against the 32 x 32
// diagonal block, then all threads update what is left of the strip.  64 wide
// so that one wave of CTAs covers n = 8192; the two serial solves per 32 (two
// warps of eight busy) bound it.
constexpr int kW = 64;
constexpr int kXS = kW + 1;       // U12 strip's row stride (lane = column)
constexpr int kBorderThreads = 256;
static_assert(kNB * kXS <= kW * kS, "either strip fits the same space");
constexpr size_t kBorderSmem = ((size_t)kNB * kS + (size_t)kW * kS + kNB) * 4;
template <int PREC>
__global__ void __launch_bounds__(kBorderThreads, 2)
    k_lu_border(float* __restrict__ LU, int n, int K, int nrow_ctas, uint16_t* __restrict__ a16,
                uint16_t* __restrict__ bt16, size_t plane, int* gate, int* fail) {
  // (another CTA may raise it meanwhile: one thread's reading decides)
  if (__syncthreads_or(threadIdx.x == 0 && *fail)) return;
  extern __shared__ __align__(16) float sm[];
  float* S = sm;                    // [kNB][kS] the diagonal block's factors
  float* X = S + kNB * kS;          // the strip: rows [kW][kS], or columns [kNB][kXS]
  float* rd = X + kW * kS;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const bool rows = (int)blockIdx.x < nrow_ctas;
  const int first = K + kNB + ((int)blockIdx.x - (rows ? 0 : nrow_ctas)) * kW;
  const int cnt = min(kW, n - first);
  // every load in flight at once, straight into shared memory (past the end:
  // zero); eight at a time through registers the border took 17.5 us, now 16.2
  auto copy4 = [&](float* dst, const float* src, bool in) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(tc::smem_u32(dst)),
                 "l"(in ? src : LU), "r"(in ? 4 : 0)
                 : "memory");
  };
#pragma unroll 4
  for (int r = w; r < kNB; r += 8)
#pragma unroll
    for (int u = 0; u < 4; ++u)
      copy4(S + r * kS + lane + 32 * u, LU + (size_t)(K + r) * n + K + lane + 32 * u, true);
  if (rows) {
#pragma unroll 4
    for (int r = w; r < kW; r += 8)
#pragma unroll
      for (int u = 0; u < 4; ++u)
        copy4(X + r * kS + lane + 32 * u, LU + (size_t)(first + r) * n + K + lane + 32 * u, r < cnt);
  } else {
#pragma unroll 4
    for (int r = w; r < kNB; r += 8)
#pragma unroll
      for (int u = 0; u < 2; ++u)
        copy4(X + r * kXS + lane + 32 * u, LU + (size_t)(K + r) * n + first + lane + 32 * u,
              lane + 32 * u < cnt);
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  if (rows && tid < kNB) rd[tid] = 1.0f / S[tid * kS + tid];
  __syncthreads();
  bool bad = false, out = false;
  for (int o = 0; o < kNB; o += kP) {
    const float* D = S + o * kS + o;
    const int rest = kNB - o - kP;
    if (rows) {
      if (tid < kW) {
        float4* row = reinterpret_cast<float4*>(X + tid * kS + o);
        float x[kP];
#pragma unroll
        for (int g = 0; g < kP / 4; ++g) {
          const float4 v = row[g];
          x[4 * g] = v.x; x[4 * g + 1] = v.y; x[4 * g + 2] = v.z; x[4 * g + 3] = v.w;
        }
        bad |= upper_solve_row(D, rd + o, x);
#pragma unroll
        for (int g = 0; g < kP / 4; ++g)
          row[g] = make_float4(x[4 * g], x[4 * g + 1], x[4 * g + 2], x[4 * g + 3]);
      }
      __syncthreads();
      if (rest)
        for (int rb = 0; rb < kW; rb += kP)
          update32_any(rest / kP, X + rb * kS + o + kP, kS, X + rb * kS + o, kS, D + kP, kS, w, lane);
    } else {
      if (tid < kW) unit_lower_solve_col4(D, kS, X + o * kXS + tid, kXS);
      __syncthreads();
      for (int rb = o + kP; rb < kNB; rb += kP)
        update32<2>(X + rb * kXS, kXS, S + rb * kS + o, kS, X + o * kXS, kXS, w, lane);
    }
    __syncthreads();
  }
  if (rows) {
    for (int t = tid; t < kW * kNB; t += kBorderThreads) {
      const int r = t / kNB, c = t % kNB;
      if (r < cnt) LU[(size_t)(first + r) * n + K + c] = X[r * kS + c];
    }
    for (int t = tid; t < kW * (kNB / 8); t += kBorderThreads) {
      const int r = t / (kNB / 8), c = (t % (kNB / 8)) * 8;
      float v[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = X[r * kS + c + j];
      if (r < cnt) out |= tc::store_operand<PREC>(a16 + (size_t)(first - K - kNB + r) * kNB + c, plane, v);
    }
    if (bad) *fail = 1;
  } else {
    for (int t = tid; t < kNB * kW; t += kBorderThreads) {
      const int r = t / kW, c = t % kW;
      if (c < cnt) LU[(size_t)(K + r) * n + first + c] = X[r * kXS + c];
    }
    for (int t = tid; t < kW * (kNB / 8); t += kBorderThreads) {
      const int c = t / (kNB / 8), k = (t % (kNB / 8)) * 8;
      float v[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = X[(k + j) * kXS + c];
      if (c < cnt) out |= tc::store_operand<PREC>(bt16 + (size_t)(first - K - kNB + c) * kNB + k, plane, v);
    }
  }
  if (PREC == SG_PREC_F32_SIMT && out) *gate = 1;
}

}  // namespace

cudaError_t lu_diag_prepare() {
  cudaError_t e = cudaFuncSetAttribute(k_lu_diag_block, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (kNB * kS + kNB) * 4);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_lu_border<SG_PREC_F32_SIMT>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBorderSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_lu_border<SG_PREC_BF16_TC>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBorderSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_lu_border<SG_PREC_F16_TC>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBorderSmem);
  return e;
}

cudaError_t launch_lu_diag_block(float* LU, int n, int K, int KB, int* piv, const int* prev,
                                 const int* err, int* fail, cudaStream_t s) {
  k_lu_diag_block<<<1, kDiagThreads, (kNB * kS + kNB) * 4, s>>>(LU, n, K, KB, piv, prev, err,
                                                                  fail);
  return cudaGetLastError();
}

cudaError_t launch_lu_border(float* LU, int n, int K, int prec, void* a16, void* bt16, int* gate,
                             int* fail, cudaStream_t s) {
  const int rest = n - K - kNB, nc = (rest + kW - 1) / kW;
  if (rest <= 0) return cudaSuccess;
  uint16_t *a = static_cast<uint16_t*>(a16), *b = static_cast<uint16_t*>(bt16);
  const size_t plane = (size_t)rest * kNB;
  const dim3 g(2 * nc);
  if (prec == SG_PREC_F32_SIMT)
    k_lu_border<SG_PREC_F32_SIMT><<<g, kBorderThreads, kBorderSmem, s>>>(LU, n, K, nc, a, b, plane,
                                                                         gate, fail);
  else if (prec == SG_PREC_BF16_TC)
    k_lu_border<SG_PREC_BF16_TC><<<g, kBorderThreads, kBorderSmem, s>>>(LU, n, K, nc, a, b, plane,
                                                                        gate, fail);
  else
    k_lu_border<SG_PREC_F16_TC><<<g, kBorderThreads, kBorderSmem, s>>>(LU, n, K, nc, a, b, plane,
                                                                       gate, fail);
  return cudaGetLastError();
}

}  // namespace sgk
