// sg_tcgen05.cuh -- device helpers of the tensor-core products
// (k_gemm_tc.cu, k_gemm_split.cu): mbarriers with bounded waits, TMA loads,
// tcgen05 instructions, and the epilogue's accesses to C.
#pragma once
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "safegpu.h"

namespace sgk {
namespace tc {

constexpr unsigned kWaitLimit = 1u << 26;

// the driver's encoder of tensor maps (null where there is none; asked once)
inline PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static const PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      p = nullptr;
    return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }();
  return fn;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}

// bounded wait for the phase with the given parity to complete
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int* err) {
  for (unsigned i = 0; i < kWaitLimit; ++i) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  atomicExch(err, 1);
  return false;
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y,
                                            uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}

// UMMA shared-memory descriptor: K-major tile in the 128-byte swizzle
// layout (rows of 128 B, 8-row groups 1024 B apart).
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);   // start address >> 4
  d |= (uint64_t)1 << 16;                      // leading byte offset (unused here)
  d |= (uint64_t)(1024 >> 4) << 32;            // stride byte offset: 8 rows x 128 B
  d |= (uint64_t)1 << 46;                      // descriptor version
  d |= (uint64_t)2 << 61;                      // 128-byte swizzle
  return d;
}

__device__ __forceinline__ void umma(uint32_t tmem, uint64_t a, uint64_t b, uint32_t id,
                                     uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
      "l"(a), "l"(b), "r"(id), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
      : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
        "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
        "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
        "=r"(r[31])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// bounded wait that also gives up as soon as another role of the CTA has
// raised the abort flag (so one failed wait cannot leave the others spinning
// through every remaining tile)
__device__ __forceinline__ bool mbar_wait_ab(uint32_t bar, uint32_t parity, int* err,
                                             volatile int* abort_flag) {
  for (unsigned i = 0; i < kWaitLimit; ++i) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
    if ((i & 255) == 255 && *abort_flag) return false;
  }
  atomicExch(err, 1);
  *abort_flag = 1;
  return false;
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// arrive on a barrier anywhere in the cluster
__device__ __forceinline__ void mbar_arrive_cl(uint32_t bar_cl) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(bar_cl) : "memory");
}

// An update's 32 x 32 chunk that lies inside M x N with 16-byte aligned rows, as
// almost all do, is loaded and stored without a test or an address of its own
// per access: with them a chunk took some 440 instructions of a warp, and the
// updates, most of whose time the epilogue takes, were 7% slower.  (Products only
// store; a second path cost them 5% at 1537 x 2049 x 1023.)
__device__ __forceinline__ bool whole_chunk(const float* C, int ldc, int M, int N, int m0q,
                                            int col0) {
  return m0q + 32 <= M && col0 + 32 <= N &&
         ((reinterpret_cast<uintptr_t>(C) | ((size_t)ldc * 4)) & 15) == 0;
}

// C rows m0q .. m0q + 31, columns col0 .. col0 + 31, as the epilogue's
// stores take them: access it, lane l: row m0q + 4 it + l / 8, columns
// col0 + 4 (l % 8) .. + 3 (zero outside M x N)
__device__ __forceinline__ void load_c(const float* __restrict__ C, int ldc, int M, int N, int m0q,
                                       int col0, int lane, float4 (&cv)[8]) {
  if (whole_chunk(C, ldc, M, N, m0q, col0)) {
    const float* p = C + (size_t)(m0q + (lane >> 3)) * ldc + col0 + (lane & 7) * 4;
#pragma unroll
    for (int it = 0; it < 8; ++it) cv[it] = *reinterpret_cast<const float4*>(p + (size_t)it * 4 * ldc);
    return;
  }
#pragma unroll
  for (int it = 0; it < 8; ++it) {
    const int grow = m0q + it * 4 + (lane >> 3), gcol = col0 + (lane & 7) * 4;
    const float* cp = C + (size_t)grow * ldc + gcol;
    if (grow < M && gcol + 4 <= N && ((reinterpret_cast<uintptr_t>(cp) & 15) == 0)) {
      cv[it] = *reinterpret_cast<const float4*>(cp);
    } else {
      float e[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) e[u] = grow < M && gcol + u < N ? cp[u] : 0.0f;
      cv[it] = make_float4(e[0], e[1], e[2], e[3]);
    }
  }
}

// Row `row`, columns c0 .. c0 + w - 1 of C (clipped to N) into L2: the
// subtracting product's epilogue reads them a tile later
__device__ __forceinline__ void prefetch_c_row(const float* C, int ldc, int M, int N, int row,
                                               int c0, int w) {
  if (row >= M || c0 >= N) return;
  const float* p = C + (size_t)row * ldc + c0;
  const unsigned bytes = (unsigned)(min(w, N - c0) * 4) & ~15u;
  if ((reinterpret_cast<uintptr_t>(p) & 15) == 0 && bytes)
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// One 32 x 32 chunk of the epilogue: lane l holds row m0q + l, columns
// col0 .. col0 + 31 (r); C := chunk, or C := cv - chunk when SUB (cv from
// load_c), through the warp's transpose buffer s_tw (16 x 32 floats,
// rows 16 h .. 16 h + 15 in turn); rows outside M and columns outside N are
// left alone.
template <bool SUB>
__device__ __forceinline__ void store_chunk(float* __restrict__ C, int ldc, int M, int N, int m0q,
                                            int col0, const uint32_t (&r)[32], float* s_tw,
                                            int lane, const float4 (&cv)[8]) {
  const bool whole = SUB && whole_chunk(C, ldc, M, N, m0q, col0);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    if ((lane >> 4) == h) {
      const int rw = lane & 15;
      float4* dst = reinterpret_cast<float4*>(s_tw + rw * 32);
#pragma unroll
      for (int j = 0; j < 8; ++j)
        dst[j ^ (rw & 7)] = make_float4(__uint_as_float(r[4 * j]), __uint_as_float(r[4 * j + 1]),
                                        __uint_as_float(r[4 * j + 2]),
                                        __uint_as_float(r[4 * j + 3]));
    }
    __syncwarp();
    if (whole) {
      float* const p = C + (size_t)(m0q + 16 * h + (lane >> 3)) * ldc + col0 + (lane & 7) * 4;
#pragma unroll
      for (int it = 0; it < 4; ++it) {
        const int rr = it * 4 + (lane >> 3);
        const float4 v = reinterpret_cast<const float4*>(s_tw + rr * 32)[(lane & 7) ^ (rr & 7)];
        const float4 c4 = cv[4 * h + it];
        // an update's results are not needed again soon: they leave L2 first,
        // which keeps the prefetched C there (4% of an update at n = 8192)
        __stcs(reinterpret_cast<float4*>(p + (size_t)it * 4 * ldc),
               make_float4(c4.x - v.x, c4.y - v.y, c4.z - v.z, c4.w - v.w));
      }
      __syncwarp();
      continue;
    }
#pragma unroll
    for (int it = 0; it < 4; ++it) {
      const int rr = it * 4 + (lane >> 3), g = lane & 7;
      const float4 v = reinterpret_cast<const float4*>(s_tw + rr * 32)[g ^ (rr & 7)];
      const int grow = m0q + 16 * h + rr, gcol = col0 + 4 * g;
      if (grow >= M) continue;
      const float4 c4 = cv[4 * h + it];
      const float4 o = SUB ? make_float4(c4.x - v.x, c4.y - v.y, c4.z - v.z, c4.w - v.w) : v;
      float* cp = C + (size_t)grow * ldc + gcol;
      if (gcol + 4 <= N && ((reinterpret_cast<uintptr_t>(cp) & 15) == 0)) {
        *reinterpret_cast<float4*>(cp) = o;
      } else {
        const float oe[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (gcol + u < N) cp[u] = oe[u];
      }
    }
    __syncwarp();
  }
}

// Tile t of the persistent order: groups of kGroupM row blocks; inside a
// group the row block varies fastest.  The 76 pairs' concurrent 256 x 256
// tiles then span 8 row blocks x about 10 column blocks, whose A and B
// slices (some 75 MB at K = 8192) stay in L2 instead of all of B (groups of
// 8 measured 0.7% faster than 16, and 32 4% slower).  by_rows: the
// elimination's updates, whose operands are narrow and whose traffic is C, go
// along the rows of C (n = 8192: 1.5% faster than in groups).
constexpr int kGroupM = 8;
__device__ __forceinline__ void tile_coords(int t, int nM, int nN, int* mb, int* nb,
                                            bool by_rows = false) {
  if (by_rows) {
    *mb = t / nN;
    *nb = t - *mb * nN;
    return;
  }
  const int per_group = kGroupM * nN;
  const int g = t / per_group;
  const int first = g * kGroupM;
  const int gm = min(kGroupM, nM - first);
  const int r = t - g * per_group;
  *mb = first + r % gm;
  *nb = r / gm;
}

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t map_rank(uint32_t local, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;"
               ::: "memory");
}
// arrive (with a byte count to expect) on a barrier anywhere in the cluster;
// CTA-scope release: a cluster-scope one would wait for every earlier global
// store of the thread
__device__ __forceinline__ void mbar_expect_tx_cl(uint32_t bar_cl, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cluster.b64 _, [%0], %1;" ::"r"(bar_cl),
               "r"(bytes) : "memory");
}
// TMA load into this CTA's shared memory completing on a barrier of either CTA of the pair
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, int x,
                                                 int y, uint32_t bar_cl) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar_cl)
      : "memory");
}
__device__ __forceinline__ void umma2(uint32_t tmem, uint64_t a, uint64_t b, uint32_t id,
                                      uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
      "l"(a), "l"(b), "r"(id), "r"(accumulate)
      : "memory");
}
// arrives once on the barrier at this offset in both CTAs of the pair when
// every MMA issued before it has completed
__device__ __forceinline__ void umma_commit_pair(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64"
      " [%0], %1;" ::"r"(bar), "h"((unsigned short)3)
      : "memory");
}

__device__ __forceinline__ uint16_t to16(float v, bool fp16) {
  if (fp16) {
    const __half x = __float2half_rn(v);
    return *reinterpret_cast<const uint16_t*>(&x);
  }
  const __nv_bfloat16 x = __float2bfloat16_rn(v);
  return *reinterpret_cast<const uint16_t*>(&x);
}

// true in one lane of a converged warp
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(p));
  return p != 0;
}

// x = p[0] + p[1] + p[2], each a bf16 (nearest to what is left); true when x
// is outside the range in which the pieces and their products are exact
__device__ __forceinline__ bool split3(float x, uint16_t (&p)[3]) {
  const uint32_t e = (__float_as_uint(x) >> 23) & 0xFFu;
  const __nv_bfloat16 h = __float2bfloat16_rn(x);
  const float r1 = x - __bfloat162float(h);
  const __nv_bfloat16 m = __float2bfloat16_rn(r1);
  const float r2 = r1 - __bfloat162float(m);
  const __nv_bfloat16 l = __float2bfloat16_rn(r2);
  p[0] = *reinterpret_cast<const uint16_t*>(&h);
  p[1] = *reinterpret_cast<const uint16_t*>(&m);
  p[2] = *reinterpret_cast<const uint16_t*>(&l);
  return x != 0.0f && (e < 127u - 50u || e > 127u + 54u);
}

// eight consecutive entries as a product's operands (PREC: an sg_precision):
// bf16, fp16, or the three bf16 pieces in planes `plane` apart (true: an entry they do not take)
template <int PREC>
__device__ __forceinline__ bool store_operand(uint16_t* dst, size_t plane, const float (&v)[8]) {
  bool bad = false;
  uint32_t h[3][4];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    uint16_t p[3];
    if (PREC == SG_PREC_F32_SIMT)
      bad |= split3(v[j], p);
    else
      p[0] = to16(v[j], PREC == SG_PREC_F16_TC);
#pragma unroll
    for (int z = 0; z < (PREC == SG_PREC_F32_SIMT ? 3 : 1); ++z)
      h[z][j >> 1] = (j & 1) ? h[z][j >> 1] | ((uint32_t)p[z] << 16) : (uint32_t)p[z];
  }
#pragma unroll
  for (int z = 0; z < (PREC == SG_PREC_F32_SIMT ? 3 : 1); ++z)
    *reinterpret_cast<uint4*>(dst + z * plane) = make_uint4(h[z][0], h[z][1], h[z][2], h[z][3]);
  return bad;
}


// Both operands of a product in one launch: A (M x K, leading dimension lda) ->
// a16 (M x Kp) and B (K x N) -> b16 (N x Kp), K-major 16-bit copies (PREC: bf16,
// fp16, or three bf16 planes), zero padded to Kp, a multiple of 64.  The first
// na CTAs take A, eight entries a thread; the others 64 x 64 tiles of B, turned
// around in shared memory: 16-byte loads along n, 16-byte stores along k.
// *gate = 1: an entry the pieces do not take.
template <int PREC>
__global__ void __launch_bounds__(256) k_cast_operands(const float* __restrict__ A, int lda, int M,
                                                       const float* __restrict__ B, int ldb, int N,
                                                       int K, int Kp, uint16_t* __restrict__ a16,
                                                       uint16_t* __restrict__ b16, int* gate,
                                                       unsigned na, int va, int vb) {
  __shared__ float t[64][65];
  bool bad = false;
  if (blockIdx.x < na) {
    const long long u = blockIdx.x * 256LL + threadIdx.x, r = u / (Kp / 8);
    const int c0 = (int)(u % (Kp / 8)) * 8;
    if (r >= M) return;
    const float* src = A + r * lda + c0;
    float x[8];
    if (va && c0 + 8 <= K) {
      const float4 p = __ldcs(reinterpret_cast<const float4*>(src));
      const float4 q = __ldcs(reinterpret_cast<const float4*>(src) + 1);
      x[0] = p.x; x[1] = p.y; x[2] = p.z; x[3] = p.w;
      x[4] = q.x; x[5] = q.y; x[6] = q.z; x[7] = q.w;
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j) x[j] = c0 + j < K ? __ldcs(src + j) : 0.0f;
    }
    bad = store_operand<PREC>(a16 + r * Kp + c0, (size_t)M * Kp, x);
  } else {
    const unsigned b = blockIdx.x - na, nt = (unsigned)(N + 63) / 64;
    const int k0 = (int)(b / nt) * 64, n0 = (int)(b % nt) * 64;
    float4 v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int e = threadIdx.x + 256 * i, k = k0 + (e >> 4), n = n0 + (e & 15) * 4;
      const float* src = B + (size_t)k * ldb + n;
      if (vb && k < K && n + 4 <= N) {
        v[i] = __ldcs(reinterpret_cast<const float4*>(src));
      } else {
        float x[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) x[j] = k < K && n + j < N ? __ldcs(src + j) : 0.0f;
        v[i] = make_float4(x[0], x[1], x[2], x[3]);
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int e = threadIdx.x + 256 * i, r = e >> 4, c = (e & 15) * 4;
      t[r][c] = v[i].x; t[r][c + 1] = v[i].y; t[r][c + 2] = v[i].z; t[r][c + 3] = v[i].w;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int e = threadIdx.x + 256 * i, nn = e >> 3, kc = (e & 7) * 8;
      if (n0 + nn >= N) continue;
      float x[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) x[j] = t[kc + j][nn];
      bad |= store_operand<PREC>(b16 + (size_t)(n0 + nn) * Kp + k0 + kc, (size_t)N * Kp, x);
    }
  }
  if (PREC == SG_PREC_F32_SIMT && bad) *gate = 1;
}

template <int PREC>
cudaError_t launch_cast_operands(const float* A, int lda, const float* B, int ldb, int M, int N,
                                 int K, int Kp, uint16_t* a16, uint16_t* b16, int* gate,
                                 cudaStream_t s) {
  const long long na = ((long long)M * (Kp / 8) + 255) / 256;
  const long long nb = (long long)((N + 63) / 64) * (Kp / 64);
  k_cast_operands<PREC><<<(unsigned)(na + nb), 256, 0, s>>>(
      A, lda, M, B, ldb, N, K, Kp, a16, b16, gate, (unsigned)na,
      lda % 4 == 0 && (uintptr_t)A % 16 == 0, ldb % 4 == 0 && (uintptr_t)B % 16 == 0);
  return cudaGetLastError();
}

}  // namespace tc
}  // namespace sgk
