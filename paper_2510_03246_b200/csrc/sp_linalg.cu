// Blocked fp64 lower Cholesky and triangular solves for the regularised weight recovery W = R (G + rho I)^-1 of the fp32
// mode and for the cached inverse of the input system.  The O(n^3) and O(m n^2) work is GEMMs on the diagonal-block
// inverses; only the 64 x 64 diagonal factorisation runs in a single thread block.  What bounds it: up to n of a few
// thousand the chain diagonal block -> panel -> next block column (about 40 us per 64 columns), above that the fp64 pipe.
// The inverse of a 4096-wide input system takes 8 ms (42 ms with scalar fp64 products and a solve for 4096 columns).
#include "sp_common.cuh"

namespace sp {
namespace {

constexpr int NB = kCholNB;
constexpr int DIAG64_BLOCKS = (NB / 4) * (NB / 4 + 1) / 2;   // 136 lower-triangular 4 x 4 blocks
constexpr int DIAG64_THREADS = 160;
constexpr int DIAG64_PITCH = NB + 1;

// Factor the nb x nb diagonal block at A (lower triangle, left as it is) and write inv(L) (lower, zero padded to
// NB x NB, unit diagonal on the padding) to dinv.  A non-positive pivot is reported once and replaced by 1.
//
// The kernel is a serial chain; what bounds it is the latency of one elimination step times the steps.  One thread owns
// one 4 x 4 block (bi, bj), bj <= bi, in registers and four columns are eliminated per step, so that 64 columns take
// 16 steps of two barriers: 20 us (a column at a time in shared memory, 64 steps of three barriers, took 111 us).  The row
// operations are applied to an identity block as well, which leaves inv(L): block m holds the trailing matrix on block
// columns > jb and the transformed identity on block columns <= jb.
__global__ void __launch_bounds__(DIAG64_THREADS) chol_diag64_kernel(const double* A, int64_t lda, int nb, double* dinv,
                                                                     int64_t block_row0, int32_t* status) {
  __shared__ double T[NB][DIAG64_PITCH];
  __shared__ __align__(16) double W[2][4][NB];   // W[k][i]: L[i, j0 + k] below the block, inv(L)[j0 + k, i] up to it
  __shared__ double Ci_s[2][16];                 // inverse of the 4 x 4 diagonal factor, row-major
  const int t = threadIdx.x;
  const bool active = t < DIAG64_BLOCKS;
  int bi = (int)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);   // t = bi (bi + 1) / 2 + bj
  while ((bi + 1) * (bi + 2) / 2 <= t) ++bi;
  while (bi * (bi + 1) / 2 > t) --bi;
  const int bj = t - bi * (bi + 1) / 2;
  for (int e = t; e < NB * NB; e += DIAG64_THREADS) {
    const int i = e / NB, j = e % NB;
    double v = 0.0;
    if (i < nb && j <= i) v = A[(int64_t)i * lda + j];
    if (i >= nb && i == j) v = 1.0;
    T[i][j] = v;
  }
  __syncthreads();
  double m[4][4];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int s = 0; s < 4; ++s) m[r][s] = active ? T[4 * bi + r][4 * bj + s] : 0.0;

  // the owner of diagonal block jb: C C^T = m, C^-1 -> m and the shared copies
  auto factor_diag = [&](int jb) {
    double c[4][4], ci[4][4], rd[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      double p = m[k][k];
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (q < k) p = fma(-c[k][q], c[k][q], p);
      if (!(p > 0.0)) {
        report_status(status, SP_ERR_NOT_SPD, (int32_t)(block_row0 + 4 * jb + k), 0);
        p = 1.0;
      }
      rd[k] = rsqrt(p);
#pragma unroll
      for (int r = 0; r < 4; ++r)
        if (r > k) {
          double v = m[r][k];
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (q < k) v = fma(-c[r][q], c[k][q], v);
          c[r][k] = v * rd[k];
        }
    }
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        if (r < s) { ci[r][s] = 0.0; continue; }
        if (r == s) { ci[r][s] = rd[s]; continue; }
        double v = 0.0;
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (q >= s && q < r) v = fma(c[r][q], ci[q][s], v);
        ci[r][s] = -v * rd[r];
      }
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        m[r][s] = ci[r][s];
        Ci_s[jb & 1][r * 4 + s] = ci[r][s];
        W[jb & 1][r][4 * jb + s] = ci[r][s];
      }
  };

  if (active && bi == 0) factor_diag(0);
  const int nsteps = (nb + 3) / 4;
  for (int jb = 0; jb < nsteps; ++jb) {
    double (*w)[NB] = W[jb & 1];
    const double* cs = Ci_s[jb & 1];
    __syncthreads();
    if (active && bj == jb && bi > jb) {          // L_i = A_i C^-T; the block starts its life as identity part from 0
      double l[4][4];
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          double v = 0.0;
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (q <= k) v = fma(m[r][q], cs[k * 4 + q], v);
          l[r][k] = v;
        }
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int r = 0; r < 4; ++r) { w[k][4 * bi + r] = l[r][k]; m[r][k] = 0.0; }
    }
    if (active && bi == jb && bj < jb) {          // final rows of inv(L): C^-1 B
      double bn[4][4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          double v = 0.0;
#pragma unroll
          for (int r = 0; r < 4; ++r)
            if (r <= k) v = fma(cs[k * 4 + r], m[r][s], v);
          bn[k][s] = v;
        }
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int s = 0; s < 4; ++s) { w[k][4 * bj + s] = bn[k][s]; m[k][s] = bn[k][s]; }
    }
    __syncthreads();
    if (active && bi > jb) {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        double wr[4], wc[4];
#pragma unroll
        for (int r = 0; r < 4; r += 2) {
          const double2 a = *reinterpret_cast<const double2*>(&w[k][4 * bi + r]);
          const double2 b = *reinterpret_cast<const double2*>(&w[k][4 * bj + r]);
          wr[r] = a.x; wr[r + 1] = a.y; wc[r] = b.x; wc[r + 1] = b.y;
        }
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int s = 0; s < 4; ++s) m[r][s] = fma(-wr[r], wc[s], m[r][s]);
      }
      if (bi == jb + 1 && bj == jb + 1 && jb + 1 < nsteps) factor_diag(jb + 1);
    }
  }

  __syncthreads();
  for (int e = t; e < NB * NB; e += DIAG64_THREADS) T[e / NB][e % NB] = 0.0;
  __syncthreads();
  if (active) {
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int s = 0; s < 4; ++s)
        if (4 * bj + s <= 4 * bi + r) T[4 * bi + r][4 * bj + s] = m[r][s];
  }
  __syncthreads();
  for (int e = t; e < NB * NB; e += DIAG64_THREADS) dinv[e] = T[e / NB][e % NB];
}

inline Operand op(const double* p, int64_t s0, int64_t s1) { return Operand{p, SP_F64, s0, s1}; }
inline OutOperand out(double* p, int64_t ld) { return OutOperand{p, SP_F64, ld}; }

#define SP_CU(x) do { cudaError_t e_ = (x); if (e_ != cudaSuccess) return e_; } while (0)

}  // namespace

// A step's chain is diagonal block -> panel -> update of the next block column ("near"); the rest of the trailing update
// ("far") runs on the assisting stream and is only waited for by the near update of the next step, which writes the
// first of its columns.
cudaError_t potrf_lower_f64(double* A, int64_t n, int64_t lda, double* dinv, int32_t* status_dev, cudaStream_t stream,
                            const SolveAssist* assist, int64_t m_extra, bool extra_is_identity) {
  int last = -1;      // event of the far update still in flight
  for (int64_t k0 = 0, step = 0; k0 < n; k0 += NB, ++step) {
    const int nb = (int)((n - k0 < NB) ? (n - k0) : NB);
    double* Akk = A + k0 * lda + k0;
    double* dk = dinv + step * NB * NB;
    count_launch();
    chol_diag64_kernel<<<1, DIAG64_THREADS, 0, stream>>>(Akk, lda, nb, dk, k0, status_dev);
    SP_CU(cudaGetLastError());
    const int64_t rem = n - k0 - nb;
    // row r of X (identity right-hand sides) is zero left of column r
    const int64_t rows = rem + ((extra_is_identity && k0 + nb < m_extra) ? k0 + nb : m_extra);
    if (rows <= 0) break;
    double* A21 = Akk + nb * lda;
    // L21 = A21 inv(L11)^T.  In place: one thread block of the GEMM covers all nb (<= tile width) columns of its
    // rows and finishes reading them before it writes.
    SP_CU(gemm_simt(rows, nb, nb, 1.0, op(A21, lda, 1), op(dk, 1, NB), 0.0, op(A21, lda, 1), out(A21, lda), false, true,
                    stream));
    if (rem <= 0) break;
    double* A22 = A21 + nb;
    const int64_t wn = (assist && rem > NB) ? NB : rem;      // columns of the near update
    if (wn < rem) {
      SP_CU(cudaEventRecord(assist->panel_done, stream));
      SP_CU(cudaStreamWaitEvent(assist->stream, assist->panel_done, 0));
    }
    if (last >= 0) SP_CU(cudaStreamWaitEvent(stream, assist->rest_done[last], 0));
    SP_CU(gemm_simt(rows, wn, nb, -1.0, op(A21, lda, 1), op(A21, 1, lda), 1.0, op(A22, lda, 1), out(A22, lda), true,
                    true, stream));
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
  return cudaSuccess;     // (the last step has no far update, and the one before it waited for its predecessor's)
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
