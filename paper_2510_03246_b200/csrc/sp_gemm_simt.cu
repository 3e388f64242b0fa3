// GEMMs outside the bf16 tensor-core path.
//   gemm_dmma_kernel: fp64 accumulation of two fp32 or two fp64 operands on the fp64 matrix instruction; the fp32-mode
//                     contraction kernel and the workhorse of the blocked fp64 Cholesky / triangular solves.
//   gemm_simt_kernel: strided CUDA-core form for everything else (bf16 or mixed operands, two non-unit strides, fp32
//                     accumulation).  Operand element types are chosen at run time.
#include "sp_common.cuh"

namespace sp {
namespace {

template <typename Acc>
__device__ __forceinline__ Acc load_elem(const void* p, int32_t dt, int64_t idx) {
  switch (dt) {
    case SP_BF16: return (Acc)__bfloat162float(reinterpret_cast<const __nv_bfloat16*>(p)[idx]);
    case SP_F64: return (Acc) reinterpret_cast<const double*>(p)[idx];
    default: return (Acc) reinterpret_cast<const float*>(p)[idx];
  }
}

template <typename Acc>
__device__ __forceinline__ void store_elem(void* p, int32_t dt, int64_t idx, Acc v) {
  switch (dt) {
    case SP_BF16: reinterpret_cast<__nv_bfloat16*>(p)[idx] = __float2bfloat16_rn((float)v); break;
    case SP_F64: reinterpret_cast<double*>(p)[idx] = (double)v; break;
    default: reinterpret_cast<float*>(p)[idx] = (float)v; break;
  }
}

constexpr int BK = 16;

template <typename Acc, int BM, int BN, int TM, int TN>
__global__ void __launch_bounds__((BM / TM) * (BN / TN))
gemm_simt_kernel(int64_t M, int64_t N, int64_t K, Acc alpha, Operand A, Operand B, Acc beta, Operand Cin,
                 OutOperand C, int lower_only) {
  kernel_begin();
  constexpr int NT = (BM / TM) * (BN / TN);
  constexpr int EA = BM * BK / NT;
  constexpr int EB = BN * BK / NT;
  static_assert(BM * BK % NT == 0 && BN * BK % NT == 0, "tile / thread mismatch");

  const int64_t row0 = (int64_t)blockIdx.y * BM;
  const int64_t col0 = (int64_t)blockIdx.x * BN;
  if (lower_only && row0 + BM - 1 < col0) return;

  __shared__ Acc As[BK][BM + 4];
  __shared__ Acc Bs[BK][BN + 4];

  const int t = threadIdx.x;
  const int tx = t % (BN / TN);
  const int ty = t / (BN / TN);
  const bool a_kfast = (A.s1 == 1);
  const bool b_nfast = (B.s1 == 1);

  Acc acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = (Acc)0;

  Acc ra[EA], rb[EB];

  auto fetch = [&](int64_t k0) {
#pragma unroll
    for (int r = 0; r < EA; ++r) {
      const int e = t + r * NT;
      const int i = a_kfast ? e / BK : e % BM;
      const int k = a_kfast ? e % BK : e / BM;
      const int64_t gi = row0 + i, gk = k0 + k;
      ra[r] = (gi < M && gk < K) ? load_elem<Acc>(A.ptr, A.dtype, gi * A.s0 + gk * A.s1) : (Acc)0;
    }
#pragma unroll
    for (int r = 0; r < EB; ++r) {
      const int e = t + r * NT;
      const int j = b_nfast ? e % BN : e / BK;
      const int k = b_nfast ? e / BN : e % BK;
      const int64_t gj = col0 + j, gk = k0 + k;
      rb[r] = (gj < N && gk < K) ? load_elem<Acc>(B.ptr, B.dtype, gk * B.s0 + gj * B.s1) : (Acc)0;
    }
  };

  fetch(0);
  for (int64_t k0 = 0; k0 < K; k0 += BK) {
    __syncthreads();
#pragma unroll
    for (int r = 0; r < EA; ++r) {
      const int e = t + r * NT;
      const int i = a_kfast ? e / BK : e % BM;
      const int k = a_kfast ? e % BK : e / BM;
      As[k][i] = ra[r];
    }
#pragma unroll
    for (int r = 0; r < EB; ++r) {
      const int e = t + r * NT;
      const int j = b_nfast ? e % BN : e / BK;
      const int k = b_nfast ? e / BN : e % BK;
      Bs[k][j] = rb[r];
    }
    __syncthreads();
    if (k0 + BK < K) fetch(k0 + BK);
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      Acc av[TM], bv[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) av[i] = As[k][ty * TM + i];
#pragma unroll
      for (int j = 0; j < TN; ++j) bv[j] = Bs[k][tx * TN + j];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] += av[i] * bv[j];
    }
  }

#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int64_t gi = row0 + ty * TM + i;
    if (gi >= M) continue;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int64_t gj = col0 + tx * TN + j;
      if (gj >= N) continue;
      Acc v = alpha * acc[i][j];
      if (beta != (Acc)0) v += beta * load_elem<Acc>(Cin.ptr, Cin.dtype, gi * Cin.s0 + gj * Cin.s1);
      store_elem<Acc>(C.ptr, C.dtype, gi * C.ld + gj, v);
    }
  }
}


// ---- fp64 accumulation on the fp64 matrix instruction (tcgen05 has no fp64 kind, so this is mma.sync)
//
// A 64 x 64 (or 32 x 64) tile per block of four warps, each 32 x 32 (16 x 32): per 8 values of K a warp issues eight
// m16n8k8 instructions on fragments of 16 eight-byte shared-memory reads, so the fp64 pipe (64 fused multiply-adds per
// SM and cycle) is the bound and not shared memory, which bounds scalar products (16 fused multiply-adds per 8 reads and a
// conversion of every element on its way in).  Operands stay in their stored orientation in shared memory; a pitch of 4
// doubles beyond a multiple of 16 makes every fragment read conflict-free in both orientations.  The next K slab travels
// through registers (16-byte loads, fp32 widened there) while the current one is multiplied; small blocks let three
// of them share an SM, which hides the prologue and the read-modify-write of C in the K = 64 updates of the factorisation.
// Measured: token contractions of fp32 operands (3072 x 3072 lower, K = 2048) 29 TFLOP/s, scalar 12.
constexpr int DM_BN = 64, DM_BK = 16, DM_THREADS = 128, DM_PAD = 4;

__device__ __forceinline__ void dmma_16x8x8(double (&d)[4], const double (&a)[4], const double (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f64.f64.f64.f64 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+d"(d[0]), "+d"(d[1]), "+d"(d[2]), "+d"(d[3])
      : "d"(a[0]), "d"(a[1]), "d"(a[2]), "d"(a[3]), "d"(b[0]), "d"(b[1]));
}

// One DIM x DM_BK slab of an operand: rows of FAST contiguous elements (K when KFAST, else the M / N index).
template <typename T, bool KFAST, int DIM>
struct DmmaSlab {
  static constexpr int V = 16 / sizeof(T);
  static constexpr int FAST = KFAST ? DM_BK : DIM, OUTER = KFAST ? DIM : DM_BK;
  static constexpr int PITCH = FAST + DM_PAD, VPR = FAST / V, CNT = OUTER * VPR / DM_THREADS;
  static constexpr int ELEMS = OUTER * PITCH;
  static_assert(OUTER * VPR % DM_THREADS == 0, "slab / thread mismatch");
  alignas(16) T r[CNT][V];      // written 16 bytes at a time, wherever the compiler keeps it

  // d0: first index of the tile along M / N, k0: first K index, dim / kend: extents
  __device__ __forceinline__ void fetch(const T* p, int64_t ld, bool vec, int64_t d0, int64_t k0, int64_t dim,
                                        int64_t kend) {
    const int64_t o0 = KFAST ? d0 : k0, f0 = KFAST ? k0 : d0, olim = KFAST ? dim : kend, flim = KFAST ? kend : dim;
#pragma unroll
    for (int q = 0; q < CNT; ++q) {
      const int e = (int)threadIdx.x + q * DM_THREADS;
      const int64_t o = o0 + e / VPR, f = f0 + (e % VPR) * V;
      const T* src = p + o * ld + f;
      if (vec && o < olim && f + V <= flim) {
        *reinterpret_cast<int4*>(r[q]) = *reinterpret_cast<const int4*>(src);
      } else {
#pragma unroll
        for (int v = 0; v < V; ++v) r[q][v] = (o < olim && f + v < flim) ? src[v] : (T)0;
      }
    }
  }
  __device__ __forceinline__ void store(double* sm) const {
#pragma unroll
    for (int q = 0; q < CNT; ++q) {
      const int e = (int)threadIdx.x + q * DM_THREADS;
      double* dst = sm + (e / VPR) * PITCH + (e % VPR) * V;
#pragma unroll
      for (int v = 0; v < V; v += 2) *reinterpret_cast<double2*>(dst + v) = make_double2((double)r[q][v], (double)r[q][v + 1]);
    }
  }
  static __device__ __forceinline__ double at(const double* sm, int dim, int k) {
    return KFAST ? sm[dim * PITCH + k] : sm[k * PITCH + dim];
  }
};

template <typename T, bool A_KFAST, bool B_KFAST, int BM>
__global__ void __launch_bounds__(DM_THREADS, 3)
gemm_dmma_kernel(int64_t M, int64_t N, int64_t K, double alpha, const T* A, int64_t lda,
                 const T* B, int64_t ldb, double beta, Operand Cin, OutOperand C, int lower_only, int k_tri) {
  kernel_begin();
  using SlabA = DmmaSlab<T, A_KFAST, BM>;
  using SlabB = DmmaSlab<T, B_KFAST, DM_BN>;
  static_assert(alignof(SlabA) % 16 == 0 && alignof(SlabB) % 16 == 0, "16-byte pieces");
  constexpr int WM = BM / 2, MT = WM / 16;      // rows of a warp, its 16-row tiles
  const int64_t row0 = (int64_t)blockIdx.y * BM, col0 = (int64_t)blockIdx.x * DM_BN;
  if (lower_only && row0 + BM - 1 < col0) return;
  __shared__ __align__(16) double sa[2][SlabA::ELEMS];
  __shared__ __align__(16) double sb[2][SlabB::ELEMS];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, t = lane & 3;
  const int wm = (warp & 1) * WM, wn = (warp >> 1) * 32;
  constexpr int V = 16 / sizeof(T);
  const bool va = lda % V == 0 && (reinterpret_cast<uintptr_t>(A) & 15u) == 0;
  const bool vb = ldb % V == 0 && (reinterpret_cast<uintptr_t>(B) & 15u) == 0;

  double acc[MT][4][4];
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.0;

  // k_tri: both operands (kTriBoth) or B (kTriColumns) are zero for K indices below their own M / N index (upper-triangular rows)
  int64_t k0 = 0;
  if (k_tri) k0 = (k_tri == kTriBoth && row0 > col0 ? row0 : col0) / DM_BK * DM_BK;
  SlabA fa;
  SlabB fb;
  fa.fetch(A, lda, va, row0, k0, M, K);
  fb.fetch(B, ldb, vb, col0, k0, N, K);
  fa.store(sa[0]);
  fb.store(sb[0]);
  __syncthreads();
  for (int buf = 0; k0 < K; k0 += DM_BK, buf ^= 1) {
    const bool more = k0 + DM_BK < K;
    if (more) {
      fa.fetch(A, lda, va, row0, k0 + DM_BK, M, K);
      fb.fetch(B, ldb, vb, col0, k0 + DM_BK, N, K);
    }
#pragma unroll
    for (int kk = 0; kk < DM_BK; kk += 8) {
      double a[MT][4], b[4][2];
#pragma unroll
      for (int i = 0; i < MT; ++i) {
        const int m = wm + 16 * i + g;
        a[i][0] = SlabA::at(sa[buf], m, kk + t);
        a[i][1] = SlabA::at(sa[buf], m + 8, kk + t);
        a[i][2] = SlabA::at(sa[buf], m, kk + t + 4);
        a[i][3] = SlabA::at(sa[buf], m + 8, kk + t + 4);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        b[j][0] = SlabB::at(sb[buf], wn + 8 * j + g, kk + t);
        b[j][1] = SlabB::at(sb[buf], wn + 8 * j + g, kk + t + 4);
      }
#pragma unroll
      for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) dmma_16x8x8(acc[i][j], a[i], b[j]);
    }
    if (more) {      // the other buffer was last read before the previous barrier
      fa.store(sa[buf ^ 1]);
      fb.store(sb[buf ^ 1]);
      __syncthreads();
    }
  }

  // a thread holds columns 2t, 2t + 1 of rows g and g + 8 of every 16 x 8 tile
  const bool c64 = C.dtype == SP_F64;
  const bool vc = C.ld % 2 == 0 && (reinterpret_cast<uintptr_t>(C.ptr) & (c64 ? 15u : 7u)) == 0;
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int64_t gi = row0 + wm + 16 * i + 8 * h + g;
      if (gi >= M) continue;
      double v[4][2];
      if (beta != 0.0) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const int64_t gj = col0 + wn + 8 * j + 2 * t + q;
            v[j][q] = gj < N ? load_elem<double>(Cin.ptr, Cin.dtype, gi * Cin.s0 + gj * Cin.s1) : 0.0;
          }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int64_t gj = col0 + wn + 8 * j + 2 * t;
        double o[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          o[q] = alpha * acc[i][j][2 * h + q];
          if (beta != 0.0) o[q] += beta * v[j][q];
        }
        if (vc && gj + 2 <= N && C.dtype != SP_BF16) {
          if (c64) *reinterpret_cast<double2*>(reinterpret_cast<double*>(C.ptr) + gi * C.ld + gj) = make_double2(o[0], o[1]);
          else *reinterpret_cast<float2*>(reinterpret_cast<float*>(C.ptr) + gi * C.ld + gj) = make_float2((float)o[0], (float)o[1]);
        } else {
#pragma unroll
          for (int q = 0; q < 2; ++q)
            if (gj + q < N) store_elem<double>(C.ptr, C.dtype, gi * C.ld + gj + q, o[q]);
        }
      }
    }
}

// Products of at most 64 values of K with 16-byte aligned fp64 operands: the panels and the next block column's updates of the fp64
// factorisation and sweeps, links of its chain.  What bounds them is latency, so all of A, B (asynchronous copies) and C (registers)
// is on its way at once; the form above fetches 16 values of K at a time, each a round trip to memory.  Same instructions in
// the same order over K: the same bits.  A fp32-mode layer 768 wide: 16.18 -> 15.34 ms together with the diagonal blocks' loads.
template <bool A_KFAST, bool B_KFAST, int BM>
struct DmmaShort {
  static constexpr int KMAX = 64, FA = A_KFAST ? KMAX : BM, OA = A_KFAST ? BM : KMAX, FB = B_KFAST ? KMAX : DM_BN,
                       OB = B_KFAST ? DM_BN : KMAX;
  static constexpr int PA = FA + DM_PAD, PB = FB + DM_PAD;
  static constexpr size_t SMEM = ((size_t)OA * PA + (size_t)OB * PB) * sizeof(double);
  // rows [o0, o0 + OUTER) x [f0, f0 + FAST) of p, zero outside [0, olim) x [0, flim)
  template <int OUTER, int FAST, int PITCH>
  static __device__ __forceinline__ void fetch(double* sm, const double* p, int64_t ld, int64_t o0, int64_t f0, int64_t olim,
                                               int64_t flim) {
    constexpr int VPR = FAST / 2, CNT = OUTER * VPR / DM_THREADS;
    static_assert(OUTER * VPR % DM_THREADS == 0, "tile / thread mismatch");
#pragma unroll 8
    for (int q = 0; q < CNT; ++q) {
      const int e = (int)threadIdx.x + q * DM_THREADS;
      const int64_t o = o0 + e / VPR, f = f0 + (e % VPR) * 2;
      const int64_t left = o < olim ? flim - f : 0;
      const int bytes = left >= 2 ? 16 : left == 1 ? 8 : 0;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                       (uint32_t)__cvta_generic_to_shared(sm + (e / VPR) * PITCH + (e % VPR) * 2)),
                   "l"(bytes > 0 ? p + o * ld + f : p), "r"(bytes)
                   : "memory");
    }
  }
};
template <bool A_KFAST, bool B_KFAST, int BM>
__global__ void __launch_bounds__(DM_THREADS) gemm_dmma_short_kernel(int64_t M, int64_t N, int K, double alpha, const double* A,
                                                                     int64_t lda, const double* B, int64_t ldb, double beta,
                                                                     const double* Cin, double* C, int64_t ldc,
                                                                     int lower_only) {
  kernel_begin();
  using S = DmmaShort<A_KFAST, B_KFAST, BM>;
  constexpr int WM = BM / 2, MT = WM / 16;
  const int64_t row0 = (int64_t)blockIdx.y * BM, col0 = (int64_t)blockIdx.x * DM_BN;
  if (lower_only && row0 + BM - 1 < col0) return;
  extern __shared__ __align__(16) double short_smem[];
  double* sa = short_smem;
  double* sb = short_smem + S::OA * S::PA;
  S::template fetch<S::OA, S::FA, S::PA>(sa, A, lda, A_KFAST ? row0 : 0, A_KFAST ? 0 : row0, A_KFAST ? M : K, A_KFAST ? K : M);
  S::template fetch<S::OB, S::FB, S::PB>(sb, B, ldb, B_KFAST ? col0 : 0, B_KFAST ? 0 : col0, B_KFAST ? N : K, B_KFAST ? K : N);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, t = lane & 3;
  const int wm = (warp & 1) * WM, wn = (warp >> 1) * 32;
  // a thread holds columns 2t, 2t + 1 of rows g and g + 8 of every 16 x 8 tile
  double c[MT][2][4][2], acc[MT][4][4];
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int64_t gi = row0 + wm + 16 * i + 8 * h + g, gj = col0 + wn + 8 * j + 2 * t + q;
          c[i][h][j][q] = beta != 0.0 && gi < M && gj < N ? Cin[gi * ldc + gj] : 0.0;
          acc[i][j][2 * h + q] = 0.0;
        }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  const int kend = (K + 7) / 8 * 8;
#pragma unroll 2
  for (int kk = 0; kk < kend; kk += 8) {
    double a[MT][4], b[4][2];
    auto at_a = [&](int m, int k) { return A_KFAST ? sa[m * S::PA + k] : sa[k * S::PA + m]; };
    auto at_b = [&](int n, int k) { return B_KFAST ? sb[n * S::PB + k] : sb[k * S::PB + n]; };
#pragma unroll
    for (int i = 0; i < MT; ++i) {
      const int m = wm + 16 * i + g;
      a[i][0] = at_a(m, kk + t);
      a[i][1] = at_a(m + 8, kk + t);
      a[i][2] = at_a(m, kk + t + 4);
      a[i][3] = at_a(m + 8, kk + t + 4);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      b[j][0] = at_b(wn + 8 * j + g, kk + t);
      b[j][1] = at_b(wn + 8 * j + g, kk + t + 4);
    }
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) dmma_16x8x8(acc[i][j], a[i], b[j]);
  }
  const bool vc = ldc % 2 == 0 && (reinterpret_cast<uintptr_t>(C) & 15u) == 0;
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int64_t gi = row0 + wm + 16 * i + 8 * h + g;
      if (gi >= M) continue;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int64_t gj = col0 + wn + 8 * j + 2 * t;
        double o[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          o[q] = alpha * acc[i][j][2 * h + q];
          if (beta != 0.0) o[q] += beta * c[i][h][j][q];
        }
        if (vc && gj + 2 <= N) {
          *reinterpret_cast<double2*>(C + gi * ldc + gj) = make_double2(o[0], o[1]);
        } else {
#pragma unroll
          for (int q = 0; q < 2; ++q)
            if (gj + q < N) C[gi * ldc + gj + q] = o[q];
        }
      }
    }
}

template <bool A_KFAST, bool B_KFAST, int BM>
cudaError_t launch_dmma_short(int64_t M, int64_t N, int64_t K, double alpha, const Operand& A, const Operand& B, double beta,
                              const Operand& Cin, const OutOperand& C, bool lower_only, cudaStream_t stream) {
  using S = DmmaShort<A_KFAST, B_KFAST, BM>;
  static PerDeviceOnce attr_once;
  const auto kernel = gemm_dmma_short_kernel<A_KFAST, B_KFAST, BM>;
  const cudaError_t e = attr_once.run([&] {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::SMEM);
  });
  if (e != cudaSuccess) return e;
  return launch(kernel, dim3((unsigned)ceil_div(N, DM_BN), (unsigned)ceil_div(M, BM)), DM_THREADS, S::SMEM, stream, M, N, (int)K,
                alpha, reinterpret_cast<const double*>(A.ptr), A_KFAST ? A.s0 : A.s1, reinterpret_cast<const double*>(B.ptr),
                B_KFAST ? B.s1 : B.s0, beta, reinterpret_cast<const double*>(Cin.ptr), reinterpret_cast<double*>(C.ptr), C.ld,
                lower_only ? 1 : 0);
}
template <int BM>
cudaError_t launch_dmma_short(int64_t M, int64_t N, int64_t K, double alpha, const Operand& A, const Operand& B, double beta,
                              const Operand& Cin, const OutOperand& C, bool lower_only, cudaStream_t stream) {
  const bool ak = A.s1 == 1, bk = B.s0 == 1;
  if (ak && bk) return launch_dmma_short<true, true, BM>(M, N, K, alpha, A, B, beta, Cin, C, lower_only, stream);
  if (ak) return launch_dmma_short<true, false, BM>(M, N, K, alpha, A, B, beta, Cin, C, lower_only, stream);
  if (bk) return launch_dmma_short<false, true, BM>(M, N, K, alpha, A, B, beta, Cin, C, lower_only, stream);
  return launch_dmma_short<false, false, BM>(M, N, K, alpha, A, B, beta, Cin, C, lower_only, stream);
}

template <typename T, int BM>
void launch_dmma(int64_t M, int64_t N, int64_t K, double alpha, const Operand& A, const Operand& B, double beta,
                 const Operand& Cin, const OutOperand& C, bool lower_only, int tri, cudaStream_t stream) {
  const dim3 grid((unsigned)ceil_div(N, DM_BN), (unsigned)ceil_div(M, BM));
  const bool ak = A.s1 == 1, bk = B.s0 == 1;
  const int64_t lda = ak ? A.s0 : A.s1, ldb = bk ? B.s1 : B.s0;
  const T* a = reinterpret_cast<const T*>(A.ptr);
  const T* b = reinterpret_cast<const T*>(B.ptr);
  const int lo = lower_only ? 1 : 0;
  if (ak && bk) launch(gemm_dmma_kernel<T, true, true, BM>, grid, DM_THREADS, 0, stream, M, N, K, alpha, a, lda, b, ldb, beta, Cin, C, lo, tri);
  else if (ak) launch(gemm_dmma_kernel<T, true, false, BM>, grid, DM_THREADS, 0, stream, M, N, K, alpha, a, lda, b, ldb, beta, Cin, C, lo, tri);
  else if (bk) launch(gemm_dmma_kernel<T, false, true, BM>, grid, DM_THREADS, 0, stream, M, N, K, alpha, a, lda, b, ldb, beta, Cin, C, lo, tri);
  else launch(gemm_dmma_kernel<T, false, false, BM>, grid, DM_THREADS, 0, stream, M, N, K, alpha, a, lda, b, ldb, beta, Cin, C, lo, tri);
}

}  // namespace

cudaError_t gemm_simt(int64_t M, int64_t N, int64_t K, double alpha, Operand A, Operand B, double beta, Operand Cin,
                      OutOperand C, bool lower_only, bool acc64, cudaStream_t stream, int k_tri) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  count_launch();
  ProfScope prof(PK_GEMM_SIMT, (lower_only ? 1.0 : 2.0) * (double)M * (double)N * (double)K, 0.0, stream);
  const bool dmma = acc64 && A.dtype == B.dtype && (A.dtype == SP_F32 || A.dtype == SP_F64) &&
                    (A.s0 == 1 || A.s1 == 1) && (B.s0 == 1 || B.s1 == 1) && K > 0;
  if (dmma) {
    // 32-row tiles while 64-row ones would leave SMs idle (the block columns of a solve: one tile wide)
    const bool small = ceil_div(M, 64) * ceil_div(N, (int64_t)DM_BN) < sm_count();
    const auto al16 = [](const void* p, int64_t ld) { return ld % 2 == 0 && (reinterpret_cast<uintptr_t>(p) & 15u) == 0; };
    const bool is_short = A.dtype == SP_F64 && K <= 64 && !k_tri && small && al16(A.ptr, A.s1 == 1 ? A.s0 : A.s1) &&
                          al16(B.ptr, B.s0 == 1 ? B.s1 : B.s0) && C.dtype == SP_F64 &&
                          (beta == 0.0 || (Cin.dtype == SP_F64 && Cin.s1 == 1 && Cin.s0 == C.ld));
    if (is_short) {
      const cudaError_t e = launch_dmma_short<32>(M, N, K, alpha, A, B, beta, Cin, C, lower_only, stream);
      if (e != cudaSuccess) return e;
    } else if (A.dtype == SP_F64) {
      if (small) launch_dmma<double, 32>(M, N, K, alpha, A, B, beta, Cin, C, lower_only, k_tri, stream);
      else launch_dmma<double, 64>(M, N, K, alpha, A, B, beta, Cin, C, lower_only, k_tri, stream);
    } else {
      if (small) launch_dmma<float, 32>(M, N, K, alpha, A, B, beta, Cin, C, lower_only, k_tri, stream);
      else launch_dmma<float, 64>(M, N, K, alpha, A, B, beta, Cin, C, lower_only, k_tri, stream);
    }
  } else if (acc64) {
    constexpr int BM = 64, BN = 64;
    dim3 grid((unsigned)ceil_div(N, BN), (unsigned)ceil_div(M, BM));
    launch(gemm_simt_kernel<double, BM, BN, 4, 4>, grid, 256, 0, stream, M, N, K, alpha, A, B, beta, Cin, C,
                                                                      lower_only ? 1 : 0);
  } else {
    constexpr int BM = 128, BN = 128;
    dim3 grid((unsigned)ceil_div(N, BN), (unsigned)ceil_div(M, BM));
    launch(gemm_simt_kernel<float, BM, BN, 8, 8>, grid, 256, 0, stream, M, N, K, (float)alpha, A, B, (float)beta, Cin, C,
                                                                     lower_only ? 1 : 0);
  }
  return cudaGetLastError();
}

}  // namespace sp
