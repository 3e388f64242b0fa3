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
// A.  Measured inside a factorisation: 14 us for 64 columns in fp64.  (One 4 x 4 block per thread, with two block barriers and
// all warps' shared update between one 4 x 4 pivot block and the next: 20 us.)  fp32 takes DiagTiles below.
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
    constexpr int VPR = NB / V, CNT = NB * VPR / THREADS;
    static_assert(NB * VPR % THREADS == 0, "block / thread mismatch");
    Vec in[CNT];
    if (vec && nb == NB) {                                   // (all loads in flight at once; behind a test each they take turns)
#pragma unroll
      for (int u = 0; u < CNT; ++u) {
        const int e = t + u * THREADS;
        in[u] = *reinterpret_cast<const Vec*>(A + (int64_t)(e / VPR) * lda + (e % VPR) * V);
      }
    } else {
#pragma unroll
      for (int u = 0; u < CNT; ++u) {
        const int e = t + u * THREADS, i = e / VPR, c = (e % VPR) * V;
#pragma unroll
        for (int v = 0; v < V; ++v) in[u].v[v] = (i < nb && c + v <= i) ? A[(int64_t)i * lda + c + v] : (T)0;
      }
    }
#pragma unroll
    for (int u = 0; u < CNT; ++u) {
      const int e = t + u * THREADS, i = e / VPR, c = (e % VPR) * V;
      Vec q = in[u];
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
    // (both sub-blocks are always run, also where the second is that of an identity: a bound known at compile time is worth
    // more, 1 % of a fp32-mode layer)
    constexpr int ns = NS;
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

// The 128 x 128 diagonal block in fp32, tile by tile: one warp per 32 x 32 tile of the factor's lower triangle (row block rb,
// column block s) and of X = inv(L)^T (an identity carried along: X L^T = I), 20 in all.  A tile takes its entries less the
// columns to its left (left-looking), then its own 32 columns four at a time: a tile on the diagonal eliminates them (the
// serial chain), the others of the column block apply the 4 x 4 inverse C^-1 and the columns it published.  Everything
// passes through shared memory by column (LT, XT: column k of L and X), groups of four columns signalled by one mbarrier per row
// block and group, so a tile starts on what is there and no block barrier stands between one column block and the next.
// Every entry receives its updates column by column in ascending order: the same bits as DiagBlock's.
// What bounds it: the chain (about 600 cycles per four columns) and, beside it, the registers that shared memory delivers (one
// per lane and cycle): the columns to the left are taken as 4 x 8 outer products per lane (12 loads for 32 multiply-adds; as
// broadcasts, 33 for 32, the other tiles' work is twice as long as the chain).  Measured against DiagBlock at 128 columns: 24.6 ->
// 18.8 us back to back, 30.5 -> 20.3 with cold caches, 27 -> 19 inside a factorisation.
struct DiagTiles {
  static constexpr int NB = 128, SB = 32, NS = NB / SB, GS = SB / 4, GROUPS = NB / 4;
  static constexpr int P = NB + 4;                            // pitch: 16-byte rows, 16 bytes off a multiple of 128
  static constexpr int TILES = NS * (NS + 1), THREADS = TILES * 32;
  static constexpr size_t SMEM = ((size_t)2 * NB * P + GROUPS * 16) * sizeof(float) + 2 * NS * GROUPS * 8;

  // Warp -> tile, as hex digits: X (1) or L (0), row block, column block.  Warps w, w + 4, ... share a scheduler: while a
  // column block is eliminated, its tile on the diagonal, the next one and the tile between them have different ones, and
  // the others' work is spread over what those leave.
  static __device__ __forceinline__ int tile_of(int warp) {
    constexpr int table[TILES] = {0x000, 0x011, 0x022, 0x033, 0x112, 0x032, 0x021, 0x010, 0x113, 0x100,
                                  0x020, 0x031, 0x103, 0x133, 0x030, 0x101, 0x122, 0x123, 0x102, 0x111};
    return table[warp];
  }
  // waits for a group's barrier, about a second at most
  static __device__ __forceinline__ bool wait(uint32_t bar, uint32_t parity) {
    const auto done = [&] {
      uint32_t ok;
      asm volatile(
          "{\n\t.reg .pred p;\n\t"
          "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
          "selp.u32 %0, 1, 0, p;\n\t}"
          : "=r"(ok)
          : "r"(bar), "r"(parity)
          : "memory");
      return ok != 0;
    };
    if (done()) return true;
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000000ll)
      if (done()) return true;
    return false;
  }
  static __device__ __forceinline__ void arrive(uint32_t bar, int lane) {      // by lane 0
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.eq.s32 p, %1, 0;\n\t"
        "@p mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];\n\t}" ::"r"(bar), "r"(lane)
        : "memory");
  }
  // {a0, a1} += f * {x, y} in one packed instruction
  static __device__ __forceinline__ void fma2(float& a0, float& a1, float f, float x, float y) {
    asm("{\n\t.reg .b64 a, b, c;\n\t"
        "mov.b64 a, {%2, %2};\n\tmov.b64 b, {%3, %4};\n\tmov.b64 c, {%0, %1};\n\t"
        "fma.rn.f32x2 c, a, b, c;\n\tmov.b64 {%0, %1}, c;\n\t}"
        : "+f"(a0), "+f"(a1)
        : "f"(f), "f"(x), "f"(y));
  }
  static __device__ __forceinline__ float4 ld(const float* p) { return *reinterpret_cast<const float4*>(p); }
  // a[c .. c + 3] += f * q
  static __device__ __forceinline__ void axpy(float (&a)[SB], int c, float f, const float4& q) {
    fma2(a[c], a[c + 1], f, q.x, q.y);
    fma2(a[c + 2], a[c + 3], f, q.z, q.w);
  }
  // l = m C^-T for a row's entries m of four columns
  static __device__ __forceinline__ void apply_ci(const float (&m)[4], const float* ci, float (&l)[4]) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      float v = 0.f;
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (q <= k) v = fmaf(m[q], ci[k * 4 + q], v);
      l[k] = v;
    }
  }

  static constexpr uint32_t BARS = 2 * NS * GROUPS;

  // Where the results go: inv(L) [NB, NB] and its transpose, fp32, dense.  (A tile of X: row rb * 32 + lane in registers, `own` the
  // same by columns.)
  struct Dense {
    float *inv, *inv_t;
    __device__ __forceinline__ void zeros(int rb, int s, int lane) const {   // the zeros on the other side of the diagonal
#pragma unroll 4
      for (int c = 0; c < SB; ++c) {
        inv[(rb * SB + c) * NB + s * SB + lane] = 0.f;
        inv_t[(s * SB + c) * NB + rb * SB + lane] = 0.f;
      }
    }
    __device__ __forceinline__ void tile(const float (&a)[SB], const float* own, bool live, int rb, int s, int lane) const {
#pragma unroll
      for (int c = 0; c < SB; ++c) inv[(s * SB + c) * NB + rb * SB + lane] = a[c];
      if (live) {
#pragma unroll
        for (int r = 0; r < SB; r += 4) {
          const float4 u = ld(own + lane * P + r);            // column s SB + lane, four rows
          inv_t[(rb * SB + r) * NB + s * SB + lane] = u.x;
          inv_t[(rb * SB + r + 1) * NB + s * SB + lane] = u.y;
          inv_t[(rb * SB + r + 2) * NB + s * SB + lane] = u.z;
          inv_t[(rb * SB + r + 3) * NB + s * SB + lane] = u.w;
        }
      } else {
#pragma unroll 8
        for (int r = 0; r < SB; ++r) inv_t[(rb * SB + r) * NB + s * SB + lane] = rb == s && r == lane ? 1.f : 0.f;
      }
    }
  };
  // A: the nb x nb block (lower triangle; rows and columns beyond nb are those of an identity).  inv [NB, NB] receives inv(L),
  // inv_t its transpose; both dense, zero outside their triangle.
  static __device__ void run(const float* A, int64_t lda, int nb, float* inv, float* inv_t, int64_t row0, int32_t* status) {
    extern __shared__ __align__(16) unsigned char diag_smem[];
    float* sm = reinterpret_cast<float*>(diag_smem);
    const uint32_t bars = (uint32_t)__cvta_generic_to_shared(sm + 2 * NB * P + GROUPS * 16);
    for (uint32_t b = threadIdx.x; b < BARS; b += THREADS)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bars + 8u * b) : "memory");
    __syncthreads();
    eliminate<false>(threadIdx.x, sm, bars, 0, A, lda, nb, Dense{inv, inv_t}, row0, status);
  }
  // place of entry (row, col) of a block that is staged in shared memory (STAGED): every tile by rows in its own place
  static __device__ __forceinline__ int staged_at(int row, int col) {
    return ((col / SB) * SB + row % SB) * P + (row / SB) * SB + col % SB;
  }

  // t: the thread.  The block comes from A, or (STAGED) sits in sm as staged_at() says: complete, that is zero above the diagonal
  // and an identity beyond nb.  bars: BARS barriers of one arrival, parity: their phase (a full block completes one of each that is
  // waited for).
  template <bool STAGED, typename Out>
  static __device__ __forceinline__ void eliminate(int t, float* sm, uint32_t bars, uint32_t parity, const float* A, int64_t lda, int nb,
                                                   const Out& out, int64_t row0, int32_t* status) {
    float* LT = sm;                                           // LT[k][row]
    float* XT = LT + NB * P;                                  // XT[k][row]
    float* CI = XT + NB * P;                                  // C^-1 of every group, row-major
    auto bar = [&](int row_block, int group) { return bars + 8u * (uint32_t)(row_block * GROUPS + group); };
    const int lane = t & 31;
    const int tl = tile_of(t >> 5);
    const bool mat = (tl >> 8) == 0;
    const int rb = (tl >> 4) & 15, s = tl & 15;
    // row blocks and column blocks beyond nb are those of an identity: nothing is eliminated there
    const int ns = (nb + SB - 1) / SB;
    const bool live = rb < ns && s < ns;
    float* own = (mat ? LT : XT) + s * SB * P + rb * SB;      // the tile, [column][row]
    const float* orow = (mat ? LT : XT) + rb * SB;            // its row block's columns
    const float* Ls = LT + s * SB;                            // rows of L that belong to its columns
    const int oid = mat ? rb : NS + rb;                       // row block of the barriers
    const int first = mat ? 0 : rb;                           // first column block with entries in this row block
    float a[SB];
    if (mat) {
      if constexpr (!STAGED) {
        // whole rows in, turned in the tile's own place
        const bool vec = lda % 4 == 0 && (reinterpret_cast<uintptr_t>(A) & 15u) == 0;
        const int c = (lane & 7) * 4, j = s * SB + c;
        float4 q[8];
        const float* p = A + (int64_t)(rb * SB + (lane >> 3)) * lda + j;
        if (vec && nb == NB) {                                  // (all loads in flight at once)
#pragma unroll
          for (int u = 0; u < 8; ++u) q[u] = ld(p + (int64_t)(4 * u) * lda);
        } else {
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const int gi = rb * SB + u * 4 + (lane >> 3);
            float v[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) v[e] = (gi < nb && j + e <= gi) ? p[(int64_t)(4 * u) * lda + e] : 0.f;
            q[u] = make_float4(v[0], v[1], v[2], v[3]);
          }
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int gi = rb * SB + u * 4 + (lane >> 3);
          float v[4] = {q[u].x, q[u].y, q[u].z, q[u].w};
#pragma unroll
          for (int e = 0; e < 4; ++e) v[e] = j + e > gi ? 0.f : (gi >= nb && j + e == gi) ? 1.f : v[e];
          q[u] = make_float4(v[0], v[1], v[2], v[3]);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) *reinterpret_cast<float4*>(own + (u * 4 + (lane >> 3)) * P + c) = q[u];
      }
      __syncwarp();
      if (s == 0) {
#pragma unroll
        for (int e = 0; e < SB; e += 4) {
          const float4 u = ld(own + lane * P + e);
          a[e] = u.x; a[e + 1] = u.y; a[e + 2] = u.z; a[e + 3] = u.w;
        }
        __syncwarp();
      }
    } else {
#pragma unroll
      for (int c = 0; c < SB; ++c) a[c] = rb == s && c == lane ? 1.f : 0.f;
      if (s > rb) out.zeros(rb, s, lane);
    }
    bool ok = true;
    if (live) {
      if (s > first) {
        // columns to the left; what the last column block waits for is not needed before the one in front of it is under
        // way, and the first one's elimination has the schedulers to itself
        if (s == NS - 1 || (!mat && s == NS - 2)) ok = ok && wait(bar(1, GS), parity);
        const int r0 = (lane >> 2) * 4, c0 = (lane & 3) * 8;  // four rows and eight columns per lane
        float acc[4][8];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int h = 0; h < 8; h += 4) {
            const float4 u = mat ? ld(own + (r0 + r) * P + c0 + h) : make_float4(0.f, 0.f, 0.f, 0.f);
            acc[r][h] = u.x; acc[r][h + 1] = u.y; acc[r][h + 2] = u.z; acc[r][h + 3] = u.w;
          }
        for (int g = first * GS; g < s * GS; ++g) {
          if (oid != s) ok = ok && wait(bar(oid, g), parity);
          ok = ok && wait(bar(s, g), parity);
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float4 l = ld(orow + (g * 4 + k) * P + r0);
            const float4 q0 = ld(Ls + (g * 4 + k) * P + c0), q1 = ld(Ls + (g * 4 + k) * P + c0 + 4);
            const float nl[4] = {-l.x, -l.y, -l.z, -l.w};
#pragma unroll
            for (int r = 0; r < 4; ++r) {
              fma2(acc[r][0], acc[r][1], nl[r], q0.x, q0.y);
              fma2(acc[r][2], acc[r][3], nl[r], q0.z, q0.w);
              fma2(acc[r][4], acc[r][5], nl[r], q1.x, q1.y);
              fma2(acc[r][6], acc[r][7], nl[r], q1.z, q1.w);
            }
          }
        }
        // one row per lane from here on
        __syncwarp();
#pragma unroll
        for (int c = 0; c < 8; ++c)
          *reinterpret_cast<float4*>(own + (c0 + c) * P + r0) = make_float4(acc[0][c], acc[1][c], acc[2][c], acc[3][c]);
        __syncwarp();
#pragma unroll
        for (int c = 0; c < SB; ++c) a[c] = own[c * P + lane];
        __syncwarp();
      }
      if (mat && rb == s) {
        factor(a, own, CI + s * GS * 16, lane, row0 + s * SB, status, bar(s, s * GS));
      } else {
#pragma unroll
        for (int g = 0; g < GS; ++g) {
          const int j = 4 * g, gg = s * GS + g;
          ok = ok && wait(bar(s, gg), parity);
          float ci[16], l[4];
#pragma unroll
          for (int q = 0; q < 16; q += 4) {
            const float4 u = ld(CI + gg * 16 + q);
            ci[q] = u.x; ci[q + 1] = u.y; ci[q + 2] = u.z; ci[q + 3] = u.w;
          }
          const float mine[4] = {a[j], a[j + 1], a[j + 2], a[j + 3]};
          apply_ci(mine, ci, l);
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            a[j + k] = l[k];
            own[(j + k) * P + lane] = l[k];
          }
          __syncwarp();
          arrive(bar(oid, gg), lane);
#pragma unroll
          for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int c = j + 4; c < SB; c += 4) axpy(a, c, -l[k], ld(Ls + (s * SB + j + k) * P + c));
        }
      }
    }
    if (!mat) out.tile(a, own, live, rb, s, lane);
    if (!ok && lane == 0) report_status(status, SP_ERR_TIMEOUT, (int32_t)row0, 12);
  }

  // Eliminates a 32 x 32 tile on the diagonal, one row per lane: own[k][row] = L below the 4 x 4 diagonal blocks, CI = their
  // C^-1, one arrival per group of four columns.  Every lane has the group's 4 x 4 block: its entries before the previous
  // group's update travel by shuffle while that group is worked on, and the update is repeated on them.
  static __device__ __forceinline__ void factor(float (&a)[SB], float* own, float* CI, int lane, int64_t row0, int32_t* status,
                                                uint32_t bar0) {
    int bad = SB;
    float m[4][4], nx[4][4], lp[4];
    auto fetch = [&](int j) {                                 // rows and columns j .. j + 3 as they are now
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (q <= r) nx[r][q] = __shfl_sync(0xffffffffu, a[j + q], j + r);
    };
    fetch(0);
#pragma unroll
    for (int g = 0; g < GS; ++g) {
      const int j = 4 * g;
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (q <= r) m[r][q] = nx[r][q];
      if (g > 0) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float4 u = ld(own + (j - 4 + k) * P + j);
          const float x[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
          for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int q = 0; q < 4; ++q)
              if (q <= r) m[r][q] = fmaf(-x[r], x[q], m[r][q]);
        }
        // off the chain: the previous group's update of this row
#pragma unroll
        for (int c = j; c < SB; c += 4)
#pragma unroll
          for (int k = 0; k < 4; ++k) axpy(a, c, -lp[k], ld(own + (j - 4 + k) * P + c));
      }
      if (g + 1 < GS) fetch(j + 4);
      float c[4][4], rd[4], ci[16];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        float p = m[k][k];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (q < k) p = fmaf(-c[k][q], c[k][q], p);
        bad = (p > 0.f || bad < SB) ? bad : j + k;
        const float r1 = recip_sqrt(p);
        rd[k] = p > 0.f ? r1 : 1.f;
#pragma unroll
        for (int r = 0; r < 4; ++r)
          if (r > k) {
            float v = m[r][k];
#pragma unroll
            for (int q = 0; q < 4; ++q)
              if (q < k) v = fmaf(-c[r][q], c[k][q], v);
            c[r][k] = v * rd[k];
          }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        ci[q * 4 + q] = rd[q];
#pragma unroll
        for (int r = 0; r < 4; ++r)
          if (r > q) {
            float v = 0.f;
#pragma unroll
            for (int z = 0; z < 4; ++z)
              if (z >= q && z < r) v = fmaf(c[r][z], ci[z * 4 + q], v);
            ci[r * 4 + q] = -v * rd[r];
          } else if (r < q) {
            ci[r * 4 + q] = 0.f;
          }
      }
      const float mine[4] = {a[j], a[j + 1], a[j + 2], a[j + 3]};
      apply_ci(mine, ci, lp);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (lane < j + 4) lp[k] = 0.f;
        own[(j + k) * P + lane] = lp[k];
      }
      if (lane == 0) {
#pragma unroll
        for (int q = 0; q < 16; q += 4)
          *reinterpret_cast<float4*>(CI + g * 16 + q) = make_float4(ci[q], ci[q + 1], ci[q + 2], ci[q + 3]);
      }
      __syncwarp();
      arrive(bar0 + 8u * g, lane);
    }
    if (bad < SB && lane == 0) report_status(status, SP_ERR_NOT_SPD, (int32_t)(row0 + bad), 0);
  }
};

}  // namespace sp
