// sg_solve.cpp -- Gaussian elimination with partial pivoting and the solve
// with iterative refinement (Sec. 5, Listing 6; the mixed-precision form
// and the residual postcondition are the library's).
//
//   1. P A = L U in binary32 storage: panels of 32 columns factored by a
//      thread-block cluster, trailing updates A22 -= L21 U12 on the tensor
//      cores (bf16 / fp16 operands, binary32 accumulation) or in binary32
//      (three bf16 pieces per operand there, or the CUDA cores).
//   2. x0 = U^-1 L^-1 P b (binary32 substitution of b rounded to binary32).
//   3. repeat: r = b - A x in binary64 (A widened exactly), d = LU \ r in
//      binary32, x += d in binary64, until max|d| <= refine_tol max|x|, or
//      the correction stops shrinking (max|d| > max|d_prev| / 2: the
//      binary64 residual limits what refinement can reach), or max_iter
//      steps (SG_ERR_NOT_CONVERGED).
//   4. postcondition (mode >= PRE_POST): max|b - A x| <= residual_tol
//      (|A|_inf max|x| + max|b|), evaluated in binary64; the first row over
//      the bound is reported.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>

#include "sg_linalg_kernels.h"
#include "sg_lu.h"
#include "sg_runtime.h"

struct sg_matrix : public sg_vector {};

namespace {

sg_status err(sg_ctx* c, sg_status s, const char* m) {
  if (c) c->err = m;
  return s;
}

size_t al(size_t x) { return (x + 255) & ~(size_t)255; }

struct SolveWork {
  float* lu;
  int* piv;
  float* y;
  double* r;
  unsigned long long* words;   // the substitutions' exchange
  unsigned* tickets;
  int* dev_err;
  int* info;
  double* norms;          // [0] max|r| [1] max|d| [2] max|x| [3] |A|_inf [4] max|b|
  unsigned long long* viol;
};

// Blocked elimination with partial pivoting of the n x n binary32 matrix in
// `lu` (row-major), in place: L (unit lower) and U overwrite it, piv[k] is
// the row interchanged with row k at step k, *info = k+1 at an exactly zero
// pivot.  moves: ceil(n / kLuPanel) * kLuMoveInts ints, zero on entry.
// gemm: tensor-core scratch (gemm_tc_scratch_bytes or, for binary32 updates,
// gemm_split_scratch_bytes of (n, n, kLuOuter)).  info[2] = 1: a wait of a
// trailing update gave up, and the factors are worthless.
cudaError_t factor_in_place(sg_ctx* c, float* lu, int n, int* piv, int* perm, int* info,
                            int* moves, unsigned* counters, void* gemm, sg_precision prec,
                            cudaStream_t s, sgk::Prof* prof) {
  cudaError_t e = cudaSuccess;
  // two levels: 32-column panels inside 128-column outer blocks.  Inside an
  // outer block each panel applies its interchanges to the block's other
  // columns and one fused kernel updates the block's columns to its right;
  // per outer block one launch applies its interchanges everywhere else, one
  // solves U12 for its 128 rows, and the trailing matrix is updated with
  // K = 128 (tensor cores, or in binary32 where the pieces do not gain on them
  // the CUDA cores)
  const bool tc = prec != SG_PREC_F32_SIMT;
  auto at = [&](int r, int col) { return lu + (size_t)r * n + col; };
  for (int K = 0; K < n && e == cudaSuccess; K += sgk::kLuOuter) {
    const int KB = std::min(sgk::kLuOuter, n - K);
    int* mv0 = moves + (size_t)(K / sgk::kLuPanel) * sgk::kLuMoveInts;
    int np = 0;
    for (int j = K; j < K + KB && e == cudaSuccess; j += sgk::kLuPanel, ++np) {
      const int jb = std::min(sgk::kLuPanel, K + KB - j);
      int* mv = moves + (size_t)(j / sgk::kLuPanel) * sgk::kLuMoveInts;
      e = sgk::launch_lu_panel(lu, n, j, jb, piv, info, mv, K, K + KB, s, prof);
      c->kernels += 1;
      if (e == cudaSuccess && j + jb < K + KB) {
        e = sgk::launch_lu_inner(lu, n, j, j + jb, K + KB, counters + j / sgk::kLuPanel, s, prof);
        c->kernels += 1;
      }
    }
    if (e == cudaSuccess) {
      e = sgk::launch_lu_laswp_outer(lu, n, mv0, np, K, KB, perm, s, prof);
      c->kernels += 1;
    }
    const int rest = n - K - KB;
    if (rest > 0 && e == cudaSuccess) {
      e = sgk::launch_lu_trsm_outer(lu, n, K, KB, K + KB, n, s, prof);
      c->kernels += 1;
      if (e == cudaSuccess && tc) {
        e = sgk::launch_gemm_tc(at(K + KB, K), n, at(K, K + KB), n, at(K + KB, K + KB), n, rest,
                                rest, KB, prec == SG_PREC_F16_TC, true, gemm, s, prof,
                                &c->kernels, -1, -1, 0.0f, 0, info + 2);
      } else if (e == cudaSuccess && sgk::gemm_split_wanted(rest, rest, KB)) {
        e = sgk::launch_gemm_split(at(K + KB, K), n, at(K, K + KB), n, at(K + KB, K + KB), n, rest,
                                   rest, KB, true, gemm, s, prof, &c->kernels, info + 2);
      } else if (e == cudaSuccess) {
        e = sgk::launch_gemm_f32(at(K + KB, K), n, at(K, K + KB), n, at(K + KB, K + KB), n, rest,
                                 rest, KB, true, s, prof);
        c->kernels += 1;
      }
    }
  }
  return e;
}

// The same factors where no interchange is needed: three launches per
// 128-column outer block (k_lu_diag.cu).  info[1] != 0 afterwards: a pivot did
// not stand on the diagonal, and the factors are worthless.
// With 16-bit updates the next diagonal block, one CTA's serial chain, runs
// beside the update: its 128 x 128 entries are updated first by a launch of
// their own, and the update of the rest leaves them and two SMs alone (the whole
// solve at n = 8192 7.39 -> 6.47 ms, at 2048 1.26 -> 1.19 ms).
cudaError_t factor_diag(sg_ctx* c, LuCache& L, int n, sg_precision prec, cudaStream_t s) {
  cudaError_t e = cudaSuccess;
  auto at = [&](int r, int col) { return L.lu + (size_t)r * n + col; };
  const bool f32 = prec == SG_PREC_F32_SIMT, fp16 = prec == SG_PREC_F16_TC;
  const int pieces = f32 ? 3 : 1;
  const int nb = (n + sgk::kLuOuter - 1) / sgk::kLuOuter;
  uint16_t* a16 = reinterpret_cast<uint16_t*>(L.operands);
  uint16_t* b16 = a16 + (size_t)n * sgk::kLuOuter * pieces;
  int* err_word = L.info + 2;
  // one word per outer block, so that no launch writes what another beside it reads
  auto fail = [&](int q) { return q == nb - 1 ? L.info + 1 : L.gates + nb + q; };
  auto diag = [&](int q, cudaStream_t st) {
    const int K = q * sgk::kLuOuter;
    c->kernels += 1;
    return sgk::launch_lu_diag_block(L.lu, n, K, std::min(sgk::kLuOuter, n - K), L.piv,
                                     q ? fail(q - 1) : nullptr, err_word, fail(q), st);
  };
  e = diag(0, s);
  for (int q = 0; q + 1 < nb && e == cudaSuccess; ++q) {
    const int K = q * sgk::kLuOuter, next = K + sgk::kLuOuter, rest = n - next;
    e = sgk::launch_lu_border(L.lu, n, K, prec, a16, b16, L.gates + q, fail(q), s);
    c->kernels += 1;
    if (e != cudaSuccess) break;
    if (f32) {
      e = sgk::launch_gemm_split_operands(a16, b16, at(next, K), n, at(K, next), n, at(next, next),
                                          n, rest, rest, sgk::kLuOuter, L.gates + q, fail(q),
                                          err_word, s, &c->kernels);
      if (e == cudaSuccess) e = diag(q + 1, s);
      continue;
    }
    auto update = [&](int m, int form, bool corner, cudaStream_t st) {
      return sgk::launch_gemm_tc_operands(a16, b16, sgk::kLuOuter, fp16, at(next, next), n, m, m,
                                          err_word, fail(q), st, &c->kernels, form, corner);
    };
    e = cudaEventRecord(L.fork, s);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(L.side, L.fork, 0);
    if (e == cudaSuccess) e = update(std::min(sgk::kLuOuter, rest), 1, false, L.side);
    if (e == cudaSuccess) e = diag(q + 1, L.side);
    if (e == cudaSuccess) e = cudaEventRecord(L.join, L.side);
    if (e == cudaSuccess && rest > sgk::kLuOuter) e = update(rest, 0, true, s);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(s, L.join, 0);
  }
  return e;
}

// Captures `body` (which launches on L.cap) into an executable graph and
// counts its kernels.
template <class F>
cudaError_t capture(sg_ctx* c, LuCache& L, cudaGraphExec_t* exec, int64_t* kernels, F&& body) {
  const int64_t k0 = c->kernels;
  cudaGraph_t g = nullptr;
  cudaError_t e = cudaStreamBeginCapture(L.cap, cudaStreamCaptureModeThreadLocal);
  if (e == cudaSuccess) {
    const cudaError_t le = body();
    e = cudaStreamEndCapture(L.cap, &g);
    if (e == cudaSuccess) e = le;
  }
  if (e == cudaSuccess) e = cudaGraphInstantiate(exec, g, 0);
  if (g) cudaGraphDestroy(g);
  *kernels = c->kernels - k0;
  c->kernels = k0;
  if (e != cudaSuccess) *exec = nullptr;
  return e;
}

// Factors A (n x n binary32) into the context's cached workspace: the first
// call for a size and precision allocates it and captures the blocked
// elimination (memsets and about 7 n / 32 kernels, or 3 n / 128 without
// interchanges) as a CUDA graph on a private stream; every call copies A in
// (the pass that forms its norms, all zero on entry, does so: a copy of its own took
// 80 us at n = 8192) and replays a graph on the context's stream.  A matrix of
// more than one panel whose rows are all diagonally dominant is factored without
// interchanges first (each pivot is verified on the device);
// when that fails, or for any other matrix, the general elimination runs (and
// SG_ERR_TIMEOUT is returned when one of its updates gave up a wait).
// The choice costs one read-back of 8 bytes (about 15 us: a determinant of n = 8
// 97 us with it, 84 without); where it applies it
// takes the factorisation at n = 8192 from 14.8 to 4.1 ms (binary32 updates: 21.8
// to 6.5 ms), at 2048 from 2.82 to 0.70 ms.  Waits for the stream.  Afterwards
// c->lu.lu holds L\U, c->lu.piv the interchanges and *hinfo the zero-pivot
// report.
sg_status lu_factor(sg_ctx* c, const float* A, int n, sg_precision prec, double* norms,
                    int* hinfo) {
  LuCache& L = c->lu;
  const int np = (n + sgk::kLuPanel - 1) / sgk::kLuPanel;
  if (L.n != n || L.prec != (int)prec || !L.base) {
    L.clear();
    size_t off = 0;
    auto take = [&](size_t bytes) {
      const size_t o2 = off;
      off = al(off + bytes);
      return o2;
    };
    const size_t o_lu = take((size_t)n * n * 4);
    const size_t o_piv = take((size_t)n * 4);
    const size_t o_perm = take((size_t)n * 4);
    const size_t o_inv = take(sgk::lu_diag_inv_bytes(n));
    const size_t o_info = take(64);
    const size_t o_moves = take((size_t)np * sgk::kLuMoveInts * 4 + (size_t)np * 4);
    const size_t o_gates = take((size_t)np * 8);
    // the operand copies of either form: M x 128 and N x 128, 16 bits each,
    // three of each for binary32 updates
    const size_t o_gemm =
        take((prec == SG_PREC_F32_SIMT ? sgk::gemm_split_scratch_bytes(n, n, sgk::kLuOuter)
                                       : sgk::gemm_tc_scratch_bytes(n, n, sgk::kLuOuter)) + 256);
    if (cudaMalloc(&L.base, off) != cudaSuccess ||
        cudaStreamCreateWithFlags(&L.cap, cudaStreamNonBlocking) != cudaSuccess ||
        cudaStreamCreateWithFlags(&L.side, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&L.fork, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&L.join, cudaEventDisableTiming) != cudaSuccess) {
      cudaGetLastError();
      L.clear();
      return err(c, SG_ERR_OOM, "factorisation workspace allocation failed");
    }
    char* base = static_cast<char*>(L.base);
    L.lu = reinterpret_cast<float*>(base + o_lu);
    L.piv = reinterpret_cast<int*>(base + o_piv);
    L.perm = reinterpret_cast<int*>(base + o_perm);
    L.inv = reinterpret_cast<float*>(base + o_inv);
    L.info = reinterpret_cast<int*>(base + o_info);
    L.moves = reinterpret_cast<int*>(base + o_moves);
    L.gates = reinterpret_cast<int*>(base + o_gates);
    L.operands = base + o_gemm;
    if (cudaMallocHost(&L.host, 128) != cudaSuccess) {
      cudaGetLastError();
      L.clear();
      return err(c, SG_ERR_OOM, "pinned result buffer allocation failed");
    }
    L.n = n;
    L.prec = (int)prec;
  }
  cudaStream_t s = c->stream;
  auto run = [&](bool diag) -> sg_status {
    cudaGraphExec_t& exec = diag ? L.exec_diag : L.exec;
    int64_t& kernels = diag ? L.kernels_diag : L.kernels;
    if (!exec) {
      cudaError_t e = sgk::lu_prepare(n);
      if (e == cudaSuccess) e = capture(c, L, &exec, &kernels, [&]() {
        cudaError_t le = cudaMemsetAsync(L.info, 0, 64, L.cap);
        if (le == cudaSuccess) le = sgk::launch_lu_iota(L.perm, n, L.cap);
        if (diag) {
          if (le == cudaSuccess) le = cudaMemsetAsync(L.gates, 0, (size_t)np * 8, L.cap);
          if (le == cudaSuccess) le = factor_diag(c, L, n, prec, L.cap);
        } else {
          const size_t counters = (size_t)np * sgk::kLuMoveInts;
          if (le == cudaSuccess)
            le = cudaMemsetAsync(L.moves, 0, (counters + (size_t)np) * 4, L.cap);
          if (le == cudaSuccess)
            le = factor_in_place(c, L.lu, n, L.piv, L.perm, L.info, L.moves,
                                 reinterpret_cast<unsigned*>(L.moves + counters), L.operands, prec,
                                 L.cap, nullptr);
        }
        if (le == cudaSuccess) le = sgk::launch_lu_diag_inv(L.lu, n, L.inv, L.cap);
        if (le == cudaSuccess) c->kernels += 2;
        return le;
      });
      if (e != cudaSuccess) {
        cudaGetLastError();
        L.clear();
        return err(c, SG_ERR_CUDA, "factorisation graph capture failed");
      }
    }
    int hi[3] = {0, 0, 0};
    sgk::prof_begin(&c->prof, "lu_factor_graph", s);
    cudaError_t e = cudaGraphLaunch(exec, s);
    sgk::prof_end(&c->prof, s);
    c->kernels += kernels;
    if (e == cudaSuccess && !diag && c->inject_update_timeout) {
      c->inject_update_timeout = false;
      e = cudaMemsetAsync(L.info + 2, 1, sizeof(int), s);
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(L.host, L.info, sizeof hi, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
      cudaGetLastError();
      return err(c, SG_ERR_CUDA, cudaGetErrorString(e));
    }
    memcpy(hi, L.host, sizeof hi);
    *hinfo = hi[0];
    if (diag) return hi[1] || hi[2] ? SG_ERR_NOT_CONVERGED : SG_OK;   // only seen below
    return hi[2] ? err(c, SG_ERR_TIMEOUT, "trailing update's wait gave up") : SG_OK;
  };
  const size_t bytes = (size_t)n * n * 4;
  cudaError_t e = sgk::launch_anorm(A, n, norms, L.lu, s);
  int not_dominant = 1;
  if (n > sgk::kLuPanel) {   // (one panel: the general form is as short)
    if (e == cudaSuccess) e = cudaMemcpyAsync(L.host, norms + 6, 8, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    memcpy(&not_dominant, L.host, sizeof not_dominant);
  }
  if (e == cudaSuccess && !not_dominant) {
    const sg_status st = run(true);
    if (st != SG_ERR_NOT_CONVERGED) return st;
    e = cudaMemcpyAsync(L.lu, A, bytes, cudaMemcpyDeviceToDevice, s);
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    return err(c, SG_ERR_CUDA, cudaGetErrorString(e));
  }
  return run(false);
}

}  // namespace

extern "C" sg_status sg_solve(sg_ctx* c, sg_matrix* A, sg_vector* b, const sg_solve_opts* opts,
                              sg_vector** xout, sg_solve_info* info) {
  if (!c || !A || !b || !xout || !A->v || !b->v) return err(c, SG_ERR_INVALID_ARG, "bad solve arguments");
  if (c->planning_only) return err(c, SG_ERR_UNSUPPORTED, "planning-only context");
  const int64_t n64 = A->v->rows;
  if (A->v->cols != n64 || b->v->n != n64)
    return err(c, SG_ERR_SHAPE, "solve needs a square matrix and a right-hand side of its size");
  if (A->v->dt != SG_F32 || b->v->dt != SG_F64)
    return err(c, SG_ERR_DTYPE, "solve needs SG_F32 A and SG_F64 b");
  if (n64 > sgk::kLuMaxN) return err(c, SG_ERR_SHAPE, "solve supports n <= 9216");
  sg_solve_opts o{SG_PREC_BF16_TC, 30, 1e-14, 1e-12, 0};
  if (opts) {
    o = *opts;
    if (o.max_iter <= 0) o.max_iter = 30;
    if (o.refine_tol <= 0) o.refine_tol = 1e-14;
    if (o.residual_tol <= 0) o.residual_tol = 1e-12;
  }
  if (o.precision < SG_PREC_F32_SIMT || o.precision > SG_PREC_F16_TC)
    return err(c, SG_ERR_INVALID_ARG, "bad precision");
  // queued work that produces A or b runs first
  sg_status st = sg_flush(c);
  if (st && st != SG_ERR_PRECONDITION && st != SG_ERR_POSTCONDITION) return st;
  if (A->v->poisoned || b->v->poisoned) return err(c, SG_ERR_POISONED, "input depends on a failed contract");
  const int n = (int)n64;
  if (n == 0) {
    auto v = std::make_shared<Value>();
    v->dt = SG_F64;
    v->n = 0;
    v->rows = 0;
    v->st = std::make_shared<Storage>();
    auto* h = new sg_vector;
    h->ctx = c;
    h->v = v;
    v->handles = 1;
    *xout = h;
    if (info) *info = sg_solve_info{0, 0, 0.0, 0.0};
    return SG_OK;
  }

  // workspace (one allocation, freed at the end of the call)
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o2 = off;
    off = al(off + bytes);
    return o2;
  };
  const size_t o_y = take((size_t)n * 4);
  const size_t o_r = take((size_t)n * 8);
  const size_t o_words = take((size_t)n * 8);
  const size_t o_tk = take(64);
  const size_t o_norms = take(8 * 8 + 16);   // norms, then viol and dev_err: read back together
  char* base = nullptr;
  cudaError_t e = cudaMallocAsync((void**)&base, off, c->stream);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return err(c, SG_ERR_OOM, "solve workspace allocation failed");
  }
  SolveWork w;
  w.y = reinterpret_cast<float*>(base + o_y);
  w.r = reinterpret_cast<double*>(base + o_r);
  w.words = reinterpret_cast<unsigned long long*>(base + o_words);
  w.tickets = reinterpret_cast<unsigned*>(base + o_tk);
  w.norms = reinterpret_cast<double*>(base + o_norms);
  w.viol = reinterpret_cast<unsigned long long*>(w.norms + 8);
  w.dev_err = reinterpret_cast<int*>(w.norms + 9);

  // the solution vector (owned by the returned handle)
  auto xv = std::make_shared<Value>();
  xv->dt = SG_F64;
  xv->n = n;
  xv->rows = n;
  xv->st = std::make_shared<Storage>();
  xv->st->bytes = (size_t)n * 8;
  xv->st->stream = c->stream;
  e = cudaMallocAsync(&xv->st->ptr, xv->st->bytes, c->stream);
  if (e != cudaSuccess) {
    cudaGetLastError();
    cudaFreeAsync(base, c->stream);
    return err(c, SG_ERR_OOM, "solution allocation failed");
  }
  xv->st->owned = true;
  double* x = static_cast<double*>(xv->st->ptr);
  join_transfers(c, A->v->st.get());
  join_transfers(c, b->v->st.get());
  const float* a = static_cast<const float*>(A->v->st->ptr);
  const double* bb = static_cast<const double*>(b->v->st->ptr);
  sgk::Prof* prof = &c->prof;
  cudaStream_t s = c->stream;

  sg_solve_info inf{0, 0, 0.0, 0.0};
  sg_status status = SG_OK;
  double hn[10] = {};
  unsigned long long hviol = 0;
  int hinfo = 0, herr = 0;
  unsigned epoch = 0;
  // One copy to pinned memory brings norms, violation and error: with three to
  // pageable memory, and memsets between the steps, a solve of n = 1000 took
  // 1756 us against 1552.
  auto sync_read = [&]() -> bool {
    e = cudaMemcpyAsync(c->lu.host, w.norms, sizeof hn, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return false;
    memcpy(hn, c->lu.host, sizeof hn);
    memcpy(&hviol, &hn[8], sizeof hviol);
    memcpy(&herr, &hn[9], sizeof herr);
    return true;
  };

  // 1. factorisation of a copy of A (the context's cached graph)
  e = cudaMemsetAsync(base + o_words, 0, o_norms + sizeof hn - o_words, s);
  if (e == cudaSuccess) {
    status = lu_factor(c, a, n, o.precision, w.norms, &hinfo);
    if (status) {
      cudaFreeAsync(base, s);
      return status;
    }
  }
  w.lu = c->lu.lu;
  w.piv = c->lu.piv;
  w.info = c->lu.info;
  if (e != cudaSuccess) {
    status = err(c, SG_ERR_CUDA, cudaGetErrorString(e));
    cudaGetLastError();
  } else if (hinfo < 0) {
    status = err(c, SG_ERR_TIMEOUT, "panel exchange wait gave up");
  } else if (hinfo) {
    inf.info = hinfo;
    status = err(c, SG_ERR_SINGULAR, "exactly zero pivot");
  }

  // 2. initial solve, 3. refinement
  bool converged = false;
  if (!status) {
    e = sgk::launch_lu_solve(w.lu, c->lu.inv, n, c->lu.perm, bb, w.y, w.words, ++epoch, w.tickets,
                             w.norms, w.dev_err, s, prof);
    if (e == cudaSuccess) e = sgk::launch_update(x, w.y, bb, n, true, w.norms, s);
    c->kernels += 4;
    double prev = -1.0;
    for (int it = 0; it < o.max_iter && e == cudaSuccess; ++it) {
      e = sgk::launch_residual(a, n, bb, x, w.r, w.norms, 0.0, nullptr, s, prof);
      if (e == cudaSuccess)
        e = sgk::launch_lu_solve(w.lu, c->lu.inv, n, c->lu.perm, w.r, w.y, w.words, ++epoch,
                                 w.tickets, w.norms, w.dev_err, s, prof);
      if (e == cudaSuccess) e = sgk::launch_update(x, w.y, bb, n, false, w.norms, s);
      c->kernels += 5;
      if (e != cudaSuccess || !sync_read()) break;
      inf.iterations = it + 1;
      inf.last_correction = hn[2] > 0 ? hn[1] / hn[2] : hn[1];
      if (herr) break;
      if (inf.last_correction <= o.refine_tol) {
        converged = true;
        break;
      }
      if (prev >= 0.0 && inf.last_correction > 0.5 * prev) {
        converged = true;   // stagnated: no further accuracy to gain
        break;
      }
      prev = inf.last_correction;
    }
    if (e != cudaSuccess) {
      status = err(c, SG_ERR_CUDA, cudaGetErrorString(e));
      cudaGetLastError();
    } else if (herr) {
      status = err(c, SG_ERR_TIMEOUT, "triangular solve wait gave up");
    }
  }

  // 4. final residual and the postcondition
  if (!status) {
    // the bound needs |A|_inf (norms[3]), max|x| (norms[2]) and max|b| (norms[4]),
    // read back with the last step
    e = cudaMemsetAsync(w.norms, 0, 8, s);
    if (e == cudaSuccess) {
      const double denom = hn[3] * hn[2] + hn[4];
      const bool check = c->mode >= SG_CONTRACTS_PRE_POST;
      e = cudaMemsetAsync(w.viol, 0, 8, s);
      if (e == cudaSuccess)
        e = sgk::launch_residual(a, n, bb, x, w.r, w.norms, o.residual_tol * denom,
                                 check ? w.viol : nullptr, s, prof);
      c->kernels += 1;
      if (e == cudaSuccess && sync_read()) {
        inf.residual = denom > 0 ? hn[0] / denom : hn[0];
        if (!converged) {
          status = err(c, SG_ERR_NOT_CONVERGED, "refinement did not converge");
        } else if (check && hviol) {
          c->has_violation = true;
          c->last_violation.contract_id = -1;
          c->last_violation.role = SG_POST;
          c->last_violation.kind = SG_C_RESIDUAL;
          c->last_violation.op_id = -1;
          c->last_violation.first_index = (int64_t)~hviol;
          c->last_violation.observed = inf.residual;
          xv->poisoned = true;
          status = err(c, SG_ERR_POSTCONDITION, "residual postcondition failed");
        }
      }
    }
    if (e != cudaSuccess && !status) {
      status = err(c, SG_ERR_CUDA, cudaGetErrorString(e));
      cudaGetLastError();
    }
  }
  if (c->prof.on) c->prof.collect();
  cudaFreeAsync(base, s);
  if (info) *info = inf;
  if (status == SG_OK || status == SG_ERR_NOT_CONVERGED || status == SG_ERR_POSTCONDITION) {
    auto* h = new sg_vector;
    h->ctx = c;
    h->v = xv;
    xv->handles = 1;
    *xout = h;
  }
  return status;
}

extern "C" sg_status sg_det(sg_ctx* c, sg_matrix* A, sg_precision prec, sg_det_result* out) {
  if (!c || !A || !A->v || !out) return err(c, SG_ERR_INVALID_ARG, "bad det arguments");
  if (c->planning_only) return err(c, SG_ERR_UNSUPPORTED, "planning-only context");
  if (prec < SG_PREC_F32_SIMT || prec > SG_PREC_F16_TC)
    return err(c, SG_ERR_INVALID_ARG, "bad precision");
  const int64_t n64 = A->v->rows;
  if (A->v->cols != n64) return err(c, SG_ERR_SHAPE, "det needs a square matrix");
  if (A->v->dt != SG_F32) return err(c, SG_ERR_DTYPE, "det needs SG_F32");
  if (n64 > sgk::kLuMaxN) return err(c, SG_ERR_SHAPE, "det supports n <= 9216");
  sg_status st = sg_flush(c);
  if (st && st != SG_ERR_PRECONDITION && st != SG_ERR_POSTCONDITION) return st;
  if (A->v->poisoned) return err(c, SG_ERR_POISONED, "input depends on a failed contract");
  const int n = (int)n64;
  if (n == 0) {   // the empty product
    *out = sg_det_result{1, 0, 0.0, 1.0};
    return SG_OK;
  }
  cudaStream_t s = c->stream;
  double* dout = nullptr;
  cudaError_t e = cudaMallocAsync((void**)&dout, 128, s);   // result, then launch_anorm's norms
  if (e != cudaSuccess) {
    cudaGetLastError();
    return err(c, SG_ERR_OOM, "det workspace allocation failed");
  }
  join_transfers(c, A->v->st.get());
  const float* a = static_cast<const float*>(A->v->st->ptr);
  e = cudaMemsetAsync(dout + 8, 0, 64, s);
  int hinfo = 0;
  sg_status st2 = e == cudaSuccess ? lu_factor(c, a, n, prec, dout + 8, &hinfo)
                                   : err(c, SG_ERR_CUDA, cudaGetErrorString(e));
  if (st2) {
    cudaFreeAsync(dout, s);
    return st2;
  }
  e = sgk::launch_lu_det(c->lu.lu, n, c->lu.piv, dout, s, &c->prof);
  c->kernels += 1;
  double h[2] = {0.0, 0.0};
  if (e == cudaSuccess) e = cudaMemcpyAsync(h, dout, sizeof h, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (c->prof.on) c->prof.collect();
  cudaFreeAsync(dout, s);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return err(c, SG_ERR_CUDA, cudaGetErrorString(e));
  }
  if (hinfo < 0) return err(c, SG_ERR_TIMEOUT, "panel exchange wait gave up");
  sg_det_result r;
  r.info = hinfo;
  if (hinfo) {   // the elimination stopped at an exactly zero pivot
    r.sign = 0;
    r.log_abs = -INFINITY;
    r.det = 0.0;
  } else {
    r.sign = (int32_t)h[0];
    r.log_abs = h[1];
    r.det = r.sign == 0 ? 0.0 : (double)r.sign * std::exp(h[1]);
  }
  *out = r;
  return SG_OK;
}

void LuCache::clear() {
  if (exec) cudaGraphExecDestroy(exec);
  if (exec_diag) cudaGraphExecDestroy(exec_diag);
  if (base) cudaFree(base);
  if (host) cudaFreeHost(host);
  if (cap) cudaStreamDestroy(cap);
  if (side) cudaStreamDestroy(side);
  if (fork) cudaEventDestroy(fork);
  if (join) cudaEventDestroy(join);
  exec = exec_diag = nullptr;
  base = host = nullptr;
  cap = side = nullptr;
  fork = join = nullptr;
  lu = nullptr;
  piv = nullptr;
  perm = nullptr;
  inv = nullptr;
  info = moves = gates = nullptr;
  operands = nullptr;
  n = 0;
  prec = -1;
  kernels = kernels_diag = 0;
}
