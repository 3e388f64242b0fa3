// Blocked fp64 lower Cholesky and triangular solves for the regularised weight recovery W = R (G + rho I)^-1 of the fp32
// mode and for the cached inverse of the input system.  The O(n^3) and O(m n^2) work is GEMMs on the diagonal-block
// inverses; only the 64 x 64 diagonal factorisation runs in a single thread block.  What bounds it: up to n of a few
// thousand the chain diagonal block -> panel -> next block column (about 33 us per 64 columns), above that the fp64 pipe.
// The inverse of a 4096-wide input system takes 4.7 ms (36 ms with scalar fp64 products and a solve for 4096 columns).
#include "sp_chol_block.cuh"
#include "sp_common.cuh"

namespace sp {
namespace {

constexpr int NB = kCholNB;
// Two-level updates on one stream: inverse of an input system, us: 768 wide 319 -> 332, 1024 549 -> 501, 2048 1481 -> 1339, 4096 5357 ->
// 4682.
constexpr int64_t kOuterMinF64 = 1024;
using Diag = DiagBlock<double, NB>;

__global__ void __launch_bounds__(Diag::THREADS) chol_diag64_kernel(const double* A, int64_t lda, int nb, double* dinv,
                                                                    int64_t block_row0, int32_t* status) {
  kernel_begin();
  Diag::run(A, lda, nb, dinv, nullptr, block_row0, status);
}

inline Operand op(const double* p, int64_t s0, int64_t s1) { return Operand{p, SP_F64, s0, s1}; }
inline OutOperand out(double* p, int64_t ld) { return OutOperand{p, SP_F64, ld}; }

#define SP_CU(x) do { cudaError_t e_ = (x); if (e_ != cudaSuccess) return e_; } while (0)

}  // namespace

// A step's chain is diagonal block -> panel -> update of the next block column ("near"); the rest of the trailing update
// ("far") runs on the assisting stream and is only waited for by the near update of the next step, which writes the
// first of its columns.  The rows below the matrix (right-hand sides, identity) are no part of the chain: they follow on a third
// stream, a panel and an update a step, behind the near update.  (Behind the panel, like the far update, their blocks and the near update's
// compete for the SMs, and which of the streams goes first differs from process to process: two fp32-mode iterations of 768 x 3072 14.42 ms
// in one half of the processes, 15.56 in the other, 50 instead of 39 us for each of the first blocks of the 3072-wide system; now 14.63 in all.)
cudaError_t potrf_lower_f64(double* A, int64_t n, int64_t lda, double* dinv, int32_t* status_dev, cudaStream_t stream,
                            const SolveAssist* assist, int64_t m_extra, bool identity) {
  static PerDeviceOnce attr_once;
  SP_CU(attr_once.run([] {
    return cudaFuncSetAttribute(chol_diag64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Diag::SMEM);
  }));
  const bool apart = assist && assist->far_stream && (m_extra > 0 || identity);
  constexpr int64_t OUTER = 4 * NB;
  const bool two_level = !assist && n >= kOuterMinF64;
  int last = -1;      // event of the far update still in flight
  for (int64_t k0 = 0, step = 0; k0 < n; k0 += NB, ++step) {
    const int nb = (int)((n - k0 < NB) ? (n - k0) : NB);
    double* Akk = A + k0 * lda + k0;
    double* dk = dinv + step * NB * NB;
    count_launch();
    launch(chol_diag64_kernel, 1, Diag::THREADS, Diag::SMEM, stream, Akk, lda, nb, dk, k0, status_dev);
    SP_CU(cudaGetLastError());
    const int64_t rem = n - k0 - nb;
    // row r of the identity's X is zero left of column r
    const int64_t extra = m_extra + (identity ? k0 + nb : 0), rows = rem + (apart ? 0 : extra);
    double* A21 = Akk + nb * lda;
    // L21 = A21 inv(L11)^T.  In place: one thread block of the GEMM covers all nb (<= tile width) columns of its
    // rows and finishes reading them before it writes.
    if (rows > 0)
      SP_CU(gemm_simt(rows, nb, nb, 1.0, op(A21, lda, 1), op(dk, 1, NB), 0.0, op(A21, lda, 1), out(A21, lda), false, true, stream));
    // one stream, wide matrix: the rest of an outer block's columns now, everything to its right once per outer block, with K four times as
    // long (a quarter of the passes over the matrix)
    if (two_level) {
      const int64_t o0 = k0 / OUTER * OUTER, end = o0 + OUTER < n ? o0 + OUTER : n;
      if (rem <= 0) break;
      double* A22 = A21 + nb;
      if (end > k0 + nb)
        SP_CU(gemm_simt(rows, end - k0 - nb, nb, -1.0, op(A21, lda, 1), op(A21, 1, lda), 1.0, op(A22, lda, 1), out(A22, lda), true,
                        true, stream));
      else
        SP_CU(gemm_simt(rows, rem, end - o0, -1.0, op(A + end * lda + o0, lda, 1), op(A + end * lda + o0, 1, lda), 1.0,
                        op(A22, lda, 1), out(A22, lda), true, true, stream));
      continue;
    }
    const auto rows_below = [&]() -> cudaError_t {
      cudaStream_t sx = assist->far_stream;
      double* E = A + n * lda + k0;
      SP_CU(cudaEventRecord(assist->near_done, stream));
      SP_CU(cudaStreamWaitEvent(sx, assist->near_done, 0));
      SP_CU(gemm_simt(extra, nb, nb, 1.0, op(E, lda, 1), op(dk, 1, NB), 0.0, op(E, lda, 1), out(E, lda), false, true, sx));
      if (rem > 0)
        SP_CU(gemm_simt(extra, rem, nb, -1.0, op(E, lda, 1), op(A21, 1, lda), 1.0, op(E + nb, lda, 1), out(E + nb, lda), false,
                        true, sx));
      return cudaSuccess;
    };
    if (rem <= 0) {
      if (apart) SP_CU(rows_below());
      break;
    }
    const int64_t wn = (assist && rem > NB) ? NB : rem;      // columns of the near update
    double* A22 = A21 + nb;
    if (wn < rem) {
      SP_CU(cudaEventRecord(assist->panel_done, stream));
      SP_CU(cudaStreamWaitEvent(assist->stream, assist->panel_done, 0));
    }
    if (last >= 0) SP_CU(cudaStreamWaitEvent(stream, assist->rest_done[last], 0));
    SP_CU(gemm_simt(rows, wn, nb, -1.0, op(A21, lda, 1), op(A21, 1, lda), 1.0, op(A22, lda, 1), out(A22, lda), true,
                    true, stream));
    if (apart) SP_CU(rows_below());
    last = -1;
    if (wn < rem) {
      double* L2 = A21 + wn * lda;
      double* Af = A22 + wn * lda + wn;
      SP_CU(gemm_simt(rows - wn, rem - wn, nb, -1.0, op(L2, lda, 1), op(L2, 1, lda), 1.0, op(Af, lda, 1), out(Af, lda),
                      true, true, assist->stream));
      last = (int)(step & 1);
      SP_CU(cudaEventRecord(assist->rest_done[last], assist->stream));
    }
  }
  // (the last step has no far update, and the one before it waited for its predecessor's)
  if (apart) {
    SP_CU(cudaEventRecord(assist->far_go, assist->far_stream));
    SP_CU(cudaStreamWaitEvent(stream, assist->far_go, 0));
  }
  return cudaSuccess;
}

// With the identity riding along the backward sweep, a chain of its own (20 us per 64 columns), becomes one product.
cudaError_t solve_inverse_f64(double* A, int64_t n, int64_t m, double* dinv, double* W, int32_t* status_dev, cudaStream_t stream,
                              const SolveAssist* assist) {
  double* Y = A + n * n;
  double* X = Y + m * n;
  SP_CU(set_identity(X, n, n, stream));
  SP_CU(potrf_lower_f64(A, n, n, dinv, status_dev, stream, assist, m, true));
  // W = Y X^T = Y L^-1; X[j, k] = 0 for k < j
  return gemm_simt(m, n, n, 1.0, op(Y, n, 1), op(X, 1, n), 0.0, op(W, n, 1), out(W, n), false, true, stream, kTriColumns);
}

cudaError_t potrs_backward_f64(double* X, int64_t m, int64_t n, int64_t ldx, const double* L, int64_t ldl,
                               const double* dinv, cudaStream_t stream, const SolveAssist* assist) {
  // W L = Y, block columns right to left; the far part of a step's update runs beside the next step's panel
  int last = -1;
  for (int64_t jb = ceil_div(n, (int64_t)NB) - 1; jb >= 0; --jb) {
    const int64_t j0 = jb * NB;
    const int nb = (int)((n - j0 < NB) ? (n - j0) : NB);
    double* Xj = X + j0;
    // W_j = Y_j inv(L_jj) : B(k, c) = dinv[k, c]
    SP_CU(gemm_simt(m, nb, nb, 1.0, op(Xj, ldx, 1), op(dinv + jb * NB * NB, NB, 1), 0.0, op(Xj, ldx, 1), out(Xj, ldx),
                    false, true, stream));
    if (j0 == 0) break;
    // Y[:, :j0] -= W_j L[j0:j0+nb, :j0] : B(k, c) = L[j0 + k, c]
    const double* Lb = L + j0 * ldl;
    const int64_t wn = (assist && j0 > NB) ? NB : j0, far = j0 - wn;
    if (far > 0) {
      SP_CU(cudaEventRecord(assist->panel_done, stream));
      SP_CU(cudaStreamWaitEvent(assist->stream, assist->panel_done, 0));
    }
    if (last >= 0) SP_CU(cudaStreamWaitEvent(stream, assist->rest_done[last], 0));
    SP_CU(gemm_simt(m, wn, nb, -1.0, op(Xj, ldx, 1), op(Lb + far, ldl, 1), 1.0, op(X + far, ldx, 1), out(X + far, ldx),
                    false, true, stream));
    last = -1;
    if (far > 0) {
      SP_CU(gemm_simt(m, far, nb, -1.0, op(Xj, ldx, 1), op(Lb, ldl, 1), 1.0, op(X, ldx, 1), out(X, ldx), false, true,
                      assist->stream));
      last = (int)(jb & 1);
      SP_CU(cudaEventRecord(assist->rest_done[last], assist->stream));
    }
  }
  return cudaSuccess;
}

}  // namespace sp
