// Factorisation of one NB x NB diagonal block by one thread block, and the inverse of its factor: the serial link of the
// blocked Cholesky factorisations (fp32: NB = 128, fp64: NB = 64).
#pragma once
#include "sp_common.cuh"

namespace sp {

// 1 / sqrt(x), x > 0.
// fp32: the hardware approximation r (relative error d below 2^-22) and one step of Newton's method for f(r) = r^-2 - x,
// r - f(r) / f'(r) = r (3 - x r^2) / 2, which leaves 1.5 d^2 and the roundings of r^2 (counted half), of the bracket and of
// the product: 2.5 x 2^-24 together.  x is a normal number (the approximation takes subnormals for zero).
// fp64: CUDA's function, which takes subnormal and infinite pivots too (a column with an infinite pivot becomes zero).
__device__ __forceinline__ float recip_sqrt(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r * fmaf(-0.5f * x, r * r, 1.5f);
}
__device__ __forceinline__ double recip_sqrt(double x) { return rsqrt(x); }

// The block is eliminated in sub-blocks of 32 columns.  Rows to carry along are the rows of the matrix below the
// sub-block and the rows of an identity appended under the matrix (X L^T = I, so X = L^-T): together always NB rows.  Per sub-block
//   A  one warp factorises the 32 x 32 diagonal sub-block, one row per lane, columns handed round by shuffles;
//   B  one thread per row solves x L11^T = row for its 32 entries (L11 read as broadcasts);
//   C  the columns to the right receive the rank-32 update in 32 x 32 pieces, one warp each.  The next diagonal
//      sub-block comes first, by all warps; the other pieces run beside the next phase A.
// Every entry receives its updates column by column in ascending order, whatever the blocking.  What bounds the kernel is
// latency: A (about 120 cycles per column), B and the first piece of C; for 128 columns the other pieces take as long as
// A.  Measured inside a factorisation: 25 us for 128 columns in fp32, 14 us for 64 in fp64.  (One 4 x 4 block per thread,
// with two block barriers and all warps' shared update between one 4 x 4 pivot block and the next: 37 and 20 us.)
template <typename T, int NB>
struct DiagBlock {
  static constexpr int SB = 32, NS = NB / SB;
  static constexpr int V = 16 / (int)sizeof(T);              // elements per 16-byte access
  static constexpr int P = NB + V;                           // pitch: rows 16 bytes off a multiple of 128
  static constexpr int PL = SB + V;
  static constexpr int THREADS = 256;                        // seven warps for C, one for A
  static constexpr size_t SMEM = ((size_t)2 * NB * P + (size_t)SB * PL + 4 * SB) * sizeof(T);
  static_assert(NB % SB == 0 && NB <= 256, "rows map to threads");

  struct __align__(16) Vec { T v[V]; };

  // Four columns are eliminated at a time: C C^T = their 4 x 4 diagonal block, and a row's entries m in these columns become
  // l = m C^-T, with C^-1 (row-major, lower) in ci.
  static __device__ __forceinline__ void apply_ci(const T (&m)[4], const T* ci, T (&l)[4]) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      T v = (T)0;
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (q <= k) v = fma(m[q], ci[k * 4 + q], v);
      l[k] = v;
    }
  }

  // phase A on the sub-block at D (pitch P): LT[k][j] = L[j][k] below the 4 x 4 diagonal blocks, CI[k / 4] = their C^-1
  static __device__ __forceinline__ void factor(const T* D, T* LT, T* CI, int lane, int64_t row0, int32_t* status) {
    T a[SB];
#pragma unroll
    for (int c = 0; c < SB; c += V) {
      const Vec q = *reinterpret_cast<const Vec*>(D + lane * P + c);
#pragma unroll
      for (int v = 0; v < V; ++v) a[c + v] = q.v[v];
    }
    int bad = SB;
    T lp[4] = {(T)0, (T)0, (T)0, (T)0};            // this lane's L entries of the previous four columns
    // a[c .. c + 3] -= lp L[c .. c + 3]^T of the previous four columns (from k0 on)
    auto update = [&](int k0, int c) {
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int h = 0; h < 4; h += V) {
          const Vec q = *reinterpret_cast<const Vec*>(LT + (k0 + k) * PL + c + h);
#pragma unroll
          for (int v = 0; v < V; ++v) a[c + h + v] = fma(-lp[k], q.v[v], a[c + h + v]);
        }
    };
#pragma unroll
    for (int j = 0; j < SB; j += 4) {
      // critical chain: next four columns -> their diagonal block in every lane -> C, C^-1 -> l of these columns
      if (j > 0) update(j - 4, j);
      T m[4][4];
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (q <= r) m[r][q] = __shfl_sync(0xffffffffu, a[j + q], j + r);
      // the rest of the previous columns' update fills the chain's latencies
      if (j > 0) {
#pragma unroll
        for (int c = j + 4; c < SB; c += 4) update(j - 4, c);
      }
      T c[4][4], rd[4], ci[16];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        T p = m[k][k];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (q < k) p = fma(-c[k][q], c[k][q], p);
        bad = (p > (T)0 || bad < SB) ? bad : j + k;
        p = p > (T)0 ? p : (T)1;
        rd[k] = recip_sqrt(p);
#pragma unroll
        for (int r = 0; r < 4; ++r)
          if (r > k) {
            T v = m[r][k];
#pragma unroll
            for (int q = 0; q < 4; ++q)
              if (q < k) v = fma(-c[r][q], c[k][q], v);
            c[r][k] = v * rd[k];
          }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        ci[q * 4 + q] = rd[q];
#pragma unroll
        for (int r = 0; r < 4; ++r)
          if (r > q) {
            T v = (T)0;
#pragma unroll
            for (int z = 0; z < 4; ++z)
              if (z >= q && z < r) v = fma(c[r][z], ci[z * 4 + q], v);
            ci[r * 4 + q] = -v * rd[r];
          } else if (r < q) {
            ci[r * 4 + q] = (T)0;
          }
      }
      const T mine[4] = {a[j], a[j + 1], a[j + 2], a[j + 3]};
      apply_ci(mine, ci, lp);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (lane < j + 4) lp[k] = (T)0;
        LT[(j + k) * PL + lane] = lp[k];
      }
      if (lane == 0) {
#pragma unroll
        for (int q = 0; q < 16; q += V) {
          Vec u;
#pragma unroll
          for (int v = 0; v < V; ++v) u.v[v] = ci[q + v];
          *reinterpret_cast<Vec*>(CI + j * 4 + q) = u;
        }
      }
      __syncwarp();
    }
    if (bad < SB && lane == 0) report_status(status, SP_ERR_NOT_SPD, (int32_t)(row0 + bad), 0);
  }

  // phase B: x <- x L11^-T
  static __device__ __forceinline__ void solve_row(T* row, const T* LT, const T* CI) {
    T x[SB];
#pragma unroll
    for (int c = 0; c < SB; c += V) {
      const Vec q = *reinterpret_cast<const Vec*>(row + c);
#pragma unroll
      for (int v = 0; v < V; ++v) x[c + v] = q.v[v];
    }
#pragma unroll
    for (int j = 0; j < SB; j += 4) {
      T ci[16], l[4];
#pragma unroll
      for (int q = 0; q < 16; q += V) {
        const Vec u = *reinterpret_cast<const Vec*>(CI + j * 4 + q);
#pragma unroll
        for (int v = 0; v < V; ++v) ci[q + v] = u.v[v];
      }
      const T mine[4] = {x[j], x[j + 1], x[j + 2], x[j + 3]};
      apply_ci(mine, ci, l);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        x[j + k] = l[k];
#pragma unroll
        for (int c = j + 4; c < SB; c += V) {
          const Vec q = *reinterpret_cast<const Vec*>(LT + (j + k) * PL + c);
#pragma unroll
          for (int v = 0; v < V; ++v) x[c + v] = fma(-l[k], q.v[v], x[c + v]);
        }
      }
    }
#pragma unroll
    for (int c = 0; c < SB; c += V) {
      Vec q;
#pragma unroll
      for (int v = 0; v < V; ++v) q.v[v] = x[c + v];
      *reinterpret_cast<Vec*>(row + c) = q;
    }
  }

  // dst -= Y L^T over 32 values of K for one warp: 32 rows (from `row` on) x 4 C columns; dcol / ycol: first column of dst
  // and Y, L: offset of L's first element.  A lane has rows (lane >> 2) + 8 i and columns (lane & 3) + 4 j: no bank conflicts.
  template <int C>
  static __device__ __forceinline__ void rank32(T* sm, int row, int dcol, int ycol, int L, int lane) {
    T acc[4][C];
    const int lr = lane >> 2, lc = lane & 3;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < C; ++j) acc[i][j] = sm[(row + lr + i * 8) * P + dcol + lc + j * 4];
#pragma unroll 4
    for (int k = 0; k < SB; k += V) {
      Vec a[4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
        a[i] = *reinterpret_cast<const Vec*>(sm + (row + lr + i * 8) * P + ycol + k);
#pragma unroll
      for (int j = 0; j < C; ++j) {
        const Vec l = *reinterpret_cast<const Vec*>(sm + L + (lc + j * 4) * P + k);
#pragma unroll
        for (int v = 0; v < V; ++v)
#pragma unroll
          for (int i = 0; i < 4; ++i) acc[i][j] = fma(-a[i].v[v], l.v[v], acc[i][j]);
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < C; ++j) sm[(row + lr + i * 8) * P + dcol + lc + j * 4] = acc[i][j];
  }

  // A: the nb x nb block (lower triangle; rows and columns beyond nb are those of an identity).  inv [NB, NB] receives
  // inv(L), inv_t (nullptr: not wanted) its transpose; both dense, zero outside their triangle.
  static __device__ void run(const T* A, int64_t lda, int nb, T* inv, T* inv_t, int64_t row0, int32_t* status) {
    extern __shared__ __align__(16) unsigned char diag_smem[];
    T* M = reinterpret_cast<T*>(diag_smem);                  // matrix rows
    T* X = M + NB * P;                                       // identity rows
    T* LT = X + NB * P;
    T* CI = LT + SB * PL;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    constexpr int NW = THREADS / 32;
    // load: one warp per row and 32 V columns, 16 bytes per lane where the rows allow it
    const bool vec = lda % V == 0 && (reinterpret_cast<uintptr_t>(A) & 15u) == 0;
    constexpr int VPR = NB / V;
#pragma unroll
    for (int e = t; e < NB * VPR; e += THREADS) {
      const int i = e / VPR, c = (e % VPR) * V;
      Vec q;
      if (vec && i < nb && c + V <= nb) {
        q = *reinterpret_cast<const Vec*>(A + (int64_t)i * lda + c);
      } else {
#pragma unroll
        for (int v = 0; v < V; ++v) q.v[v] = (i < nb && c + v <= i) ? A[(int64_t)i * lda + c + v] : (T)0;
      }
#pragma unroll
      for (int v = 0; v < V; ++v) q.v[v] = c + v > i ? (T)0 : (i >= nb && c + v == i) ? (T)1 : q.v[v];
      *reinterpret_cast<Vec*>(M + i * P + c) = q;
#pragma unroll
      for (int v = 0; v < V; ++v) q.v[v] = c + v == i ? (T)1 : (T)0;
      *reinterpret_cast<Vec*>(X + i * P + c) = q;
    }
    __syncthreads();
    // columns cs .. cs + 31 of X: rows of inv(L) (lanes along a row) and columns of its transpose, by the NB threads from
    // STORE0 on
    constexpr int STORE0 = 96;
    auto store_inv = [&](int cs) {
      const int t = (int)threadIdx.x - STORE0;
      if (t >= NB) return;
#pragma unroll
      for (int c = 0; c < SB; c += V) {
        const Vec q = *reinterpret_cast<const Vec*>(X + t * P + cs + c);
        if (inv_t != nullptr) *reinterpret_cast<Vec*>(inv_t + t * NB + cs + c) = q;
#pragma unroll
        for (int v = 0; v < V; ++v) inv[(cs + c + v) * NB + t] = q.v[v];
      }
    };
    // sub-blocks beyond nb are those of an identity: nothing is eliminated there, their columns of X stay as they are (a
    // solve for 17 unknowns in fp32: 53 us, 65 through all four).  Two sub-blocks (fp64) are always run: a bound known at
    // compile time is worth more there (1 % of a fp32-mode layer).
    const int ns = NS > 2 ? (nb + SB - 1) / SB : NS;
    for (int s = 0; s < ns; ++s) {
      const int cs = s * SB, ce = cs + SB;
      if (warp == NW - 1) {
        factor(M + cs * P + cs, LT, CI, lane, row0 + cs, status);
      } else if (s > 0) {
        // rest of the update of sub-block s - 1: matrix rows, then identity rows (X follows M: its row r is row NB + r).
        // The factorising warp shares its scheduler with warp 3, which comes last; warps 3 to 6 also store.
        const int ps = cs - SB;
        int turn = 0;
        for (int cb = s; cb < ns; ++cb)
          for (int rb = cb == s ? s + 1 : cb; rb < NS + s; ++rb) {             // ((s, s) is done before)
            const int w = turn++ % (NW - 1);
            if (warp == (w < 3 ? w : w < 6 ? w + 1 : 3))
              rank32<8>(M, (rb < NS ? rb : NB / SB + rb - NS) * SB, cb * SB, ps, cb * SB * P + ps, lane);
          }
        if (t >= STORE0) store_inv(ps);
      }
      __syncthreads();
      if (t < NB) solve_row((t >= ce ? M : X) + t * P + cs, LT, CI);
      __syncthreads();
      if (s + 1 < ns) {
        // next diagonal sub-block, 32 x 4 entries per warp
        rank32<1>(M, ce, ce + warp * 4, cs, (ce + warp * 4) * P + cs, lane);
        __syncthreads();
      }
    }
    if (t >= STORE0)
      for (int cs = (ns - 1) * SB; cs < NB; cs += SB) store_inv(cs);
  }
};

}  // namespace sp
