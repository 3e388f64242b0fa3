// fp32 Cholesky factorisation and triangular solves whose O(n^3) / O(m n^2) work runs on the tensor cores.
//
// The regularised weight recovery W = R (G + rho I)^-1 needs fp32-level accuracy (G is a Gram matrix of ReLU
// activations with a condition number of the order of its size), which a plain bf16 product cannot give.  Every fp32
// value is therefore held as an exact sum of three bf16 parts (hi + mid + lo, 3 x 8 mantissa bits), and a product
// of two such operands is taken as the six part products of weight >= 2^-16 (hi.hi, hi.mid, mid.hi, hi.lo, lo.hi,
// mid.mid), each a K segment of one tcgen05 GEMM with fp32 accumulation.  The dropped terms are below 2^-23.
//
// Systems that solve_in_one() names are solved in one launch instead (sp_solve_tc.cu); this form serves smaller and wider ones, the
// widest modules, and many systems at a time.
//
// Blocked right-looking algorithm with 128-wide panels:
//   diagonal block : one CTA factorises it and forms inv(L11) in the same sweep (sp_chol_block.cuh);
//   panel          : L21 = A21 inv(L11)^T on the CUDA cores (K = 128), written as fp32 and as the three bf16 parts;
//   trailing update: A22 -= L21 L21^T (lower triangle) as one six-segment tensor-core GEMM.
// The triangular solves X L^T = R, W L = X use the same two kernels block column by block column.
#include "sp_chol_block.cuh"
#include "sp_common.cuh"

namespace sp {
namespace {

constexpr int TB = kCholTcNB;          // 128

using Diag = DiagTiles;
static_assert(Diag::NB == TB, "one block");

// Diagonal block: inv(L) and its transpose to dinv[0 : TB*TB] and dinv[TB*TB : 2*TB*TB].  L itself is not written back:
// the solves use inv(L) of the diagonal blocks and the blocks of L below them only.
__global__ void __launch_bounds__(Diag::THREADS) chol_diag128_kernel(const float* A, int64_t lda, int nb, float* dinv,
                                                                     int64_t row0, int32_t* status,
                                                                     const int32_t* skip, int64_t a_bs, int64_t d_bs) {
  kernel_begin();
  if (skip != nullptr && *skip != 0) return;                  // conditional launch (see SkipScope)
  A += (int64_t)blockIdx.x * a_bs;                            // batched launch: one CTA per system
  dinv += (int64_t)blockIdx.x * d_bs;
  Diag::run(A, lda, nb, dinv, dinv + TB * TB, row0, status);
}

__device__ __forceinline__ void split3(float v, __nv_bfloat16& hi, __nv_bfloat16& mid, __nv_bfloat16& lo) {
  hi = __float2bfloat16_rn(v);
  const float r1 = v - __bfloat162float(hi);
  mid = __float2bfloat16_rn(r1);
  const float r2 = r1 - __bfloat162float(mid);
  lo = __float2bfloat16_rn(r2);
}

// ---- staging of one 128 x 128 fp32 block (64 KiB) into shared memory by bulk asynchronous copies
__device__ __forceinline__ uint32_t lin_smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// One thread: arm the barrier with the byte count and issue the copies (four of 16 KiB).
__device__ __forceinline__ void stage_block_issue(float* dst_smem, const float* src, uint64_t* bar) {
  const uint32_t b = lin_smem_u32(bar);
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b), "r"((uint32_t)(TB * TB * 4))
               : "memory");
#pragma unroll
  for (int q = 0; q < 4; ++q)
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(lin_smem_u32(dst_smem + q * (TB * TB / 4))), "l"(src + q * (TB * TB / 4)),
                   "r"((uint32_t)(TB * TB)), "r"(b)
                 : "memory");
}
__device__ __forceinline__ void stage_bar_init(uint64_t* bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(lin_smem_u32(bar)) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
// Every thread: wait for the block (phase `parity`), at most about a second.  Returns false when the wait ran out.
__device__ __forceinline__ bool stage_block_wait(uint64_t* bar, uint32_t parity) {
  const uint32_t b = lin_smem_u32(bar);
  const long long t0 = clock64();
  for (uint32_t it = 0;; ++it) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(b), "r"(parity)
        : "memory");
    if (ok) return true;
    if ((it & 0xffu) == 0xffu && clock64() - t0 > 2000000000ll) return false;
  }
}

// acc += {a, a} * {x, y} in one packed instruction
__device__ __forceinline__ void fma_dup(float2& acc, float a, float x, float y) {
  asm("{\n\t.reg .b64 a, b, c;\n\t"
      "mov.b64 a, {%2, %2};\n\tmov.b64 b, {%3, %4};\n\tmov.b64 c, {%0, %1};\n\t"
      "fma.rn.f32x2 c, a, b, c;\n\tmov.b64 {%0, %1}, c;\n\t}"
      : "+f"(acc.x), "+f"(acc.y)
      : "f"(a), "f"(x), "f"(y));
}

// Product of an R x 128 tile (At[k][row], pitch R + 4) with a 128 x 128 block (Lt[k][c]), summed over k in ascending order
// whatever R.  A warp takes RT rows, a lane four columns.  Shared memory delivers one register per lane and cycle and
// the multiply-adds wait for it, so few rows per block are what makes a block fast.
template <int R>
struct RowTile {
  static constexpr int THREADS = R == 32 ? 256 : 128;
  static constexpr int AP = R + 4, RT = R / (THREADS / 32);
  static_assert(R == 8 || R == 16 || R == 32, "tile shapes");
  struct __align__(RT == 2 ? 8 : 16) Rows { float v[RT]; };
  // thread t: rows row0(t) .. + RT - 1, columns col(t) .. + 3
  static __device__ __forceinline__ int row0(int t) { return (t >> 5) * RT; }
  static __device__ __forceinline__ int col(int t) { return (t & 31) * 4; }

  static __device__ __forceinline__ void product(const float* At, const float* Lt, float4 (&out)[RT]) {
    const float* ap = At + row0(threadIdx.x);
    const float* lp = Lt + col(threadIdx.x);
    float2 acc[RT][2];
#pragma unroll
    for (int r = 0; r < RT; ++r) acc[r][0] = acc[r][1] = make_float2(0.f, 0.f);
#pragma unroll 8
    for (int k = 0; k < TB; ++k) {
      const Rows a = *reinterpret_cast<const Rows*>(ap + k * AP);
      const float4 l = *reinterpret_cast<const float4*>(lp + k * TB);
#pragma unroll
      for (int r = 0; r < RT; ++r) {
        fma_dup(acc[r][0], a.v[r], l.x, l.y);
        fma_dup(acc[r][1], a.v[r], l.z, l.w);
      }
    }
#pragma unroll
    for (int r = 0; r < RT; ++r) out[r] = make_float4(acc[r][0].x, acc[r][0].y, acc[r][1].x, acc[r][1].y);
  }
  // this thread's entries into At
  static __device__ __forceinline__ void store(float* At, const float4 (&v)[RT]) { store_transposed(At, AP, v); }
  static __device__ __forceinline__ void store_transposed(float* base, int pitch, const float4 (&v)[RT]) {
    float* dst = base + col(threadIdx.x) * pitch + row0(threadIdx.x);
    Rows u[4];
#pragma unroll
    for (int r = 0; r < RT; ++r) { u[0].v[r] = v[r].x; u[1].v[r] = v[r].y; u[2].v[r] = v[r].z; u[3].v[r] = v[r].w; }
#pragma unroll
    for (int j = 0; j < 4; ++j) *reinterpret_cast<Rows*>(dst + j * pitch) = u[j];
  }
};
template <int R>
constexpr size_t pa_smem(bool with_near) {     // inv(L) block, row tile, (near) the block of L, barriers
  return ((size_t)TB * TB * (with_near ? 2 : 1) + (size_t)TB * RowTile<R>::AP) * sizeof(float) + 16;
}

// Optional first product of the same launch (backward triangular solve, TRANS form only): the block column W_p that the
// previous step left (nb_p columns, right of this one) is applied to this block column before it is multiplied by inv(L),
// X_j -= W_p L[p rows, j columns], so that the chain of a solve is one kernel per block column.  A CTA reads and writes
// its own rows only, and what the tensor-core updates on the other stream add into X_j is complete before the launch:
// every entry is summed in a fixed order.  L: fp32 factor, pointer to element (first row of block p, first column of block
// j), leading dimension ldl (a multiple of 4, 16-byte aligned rows); W: first column of W_p in X.
struct PanelNear {
  const float* L;    // nullptr: no such product
  int64_t ldl;
  const float* W;
  int nb_p;
};
constexpr PanelNear kNoNear{nullptr, 0, nullptr, 0};
// Batched launch of the panel kernel (grid.y = systems): element strides between the systems' arrays
struct PanelBatch {
  int64_t x = 0, dinv = 0, s = 0, near_l = 0;    // X (and near.W), dinv, S, near.L
};

// X[i, 0:nb] <- X[i, 0:nb] inv(L)^T (TRANS == false) or X[i, 0:nb] inv(L) (TRANS == true), for `rows` rows.
// dinv is the pair of TB x TB blocks written by chol_diag128_kernel.  The result is written back in fp32 (write_f32)
// and as three bf16 parts to S[i * lds + part * s_seg + c] for all TB columns (zero beyond nb).
// One CTA takes R rows.  The 64 KiB block of inv(L) comes in by bulk copies while the threads fetch and transpose the
// rows of X.  The kernel is a link of a serial chain: few rows per CTA shorten it as long as one wave covers all rows
// (see panel_rows): 768 rows, both products: 10.4 us with 48 CTAs of 16 rows, 15.4 us with 24 of 32.
template <bool TRANS, int R>
__global__ void __launch_bounds__(RowTile<R>::THREADS) panel_apply_kernel(float* X, int64_t ldx, int64_t rows, int nb,
                                                                 const float* dinv, __nv_bfloat16* S,
                                                                 int64_t lds, int64_t s_seg, int write_f32,
                                                                 int32_t* status, PanelNear near,
                                                                 const int32_t* skip, PanelBatch pb) {
  kernel_begin();
  if (skip != nullptr && *skip != 0) return;
  using Tile = RowTile<R>;
  constexpr int AP = Tile::AP;
  X += (int64_t)blockIdx.y * pb.x;
  dinv += (int64_t)blockIdx.y * pb.dinv;
  if (S) S += (int64_t)blockIdx.y * pb.s;
  if (near.L) { near.L += (int64_t)blockIdx.y * pb.near_l; near.W += (int64_t)blockIdx.y * pb.x; }
  extern __shared__ __align__(128) float pa_smem_raw[];
  const bool do_near = TRANS && near.L != nullptr;
  float* Lt = pa_smem_raw;                                                      // Lt[k][c]
  float* At = Lt + TB * TB;                                                     // At[k][row]
  float* Bn = At + TB * AP;                                                     // Bn[k][c] (near only)
  uint64_t* bar = reinterpret_cast<uint64_t*>(Bn + (do_near ? TB * TB : 0));    // Lt landed
  const int t = threadIdx.x;
  const int64_t r0 = (int64_t)blockIdx.x * R;
  const bool x_al = (ldx % 4 == 0) && ((reinterpret_cast<uintptr_t>(X) & 15u) == 0);
  if (t == 0) stage_bar_init(bar);
  __syncthreads();
  // Lt[k][c] = inv(L)[c][k] (the transposed copy) or inv(L)[k][c]: a straight copy either way
  if (t == 0) stage_block_issue(Lt, dinv + (TRANS ? 0 : TB * TB), bar);
  if (do_near) {
    // rows p .. p + nb_p - 1 of L, TB columns each; zeros below
    for (int e = t; e < TB * TB / 4; e += Tile::THREADS) {
      float* dst = Bn + e * 4;
      if (e / (TB / 4) < near.nb_p)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(lin_smem_u32(dst)),
                     "l"(near.L + (int64_t)(e / (TB / 4)) * near.ldl + (e % (TB / 4)) * 4)
                     : "memory");
      else
        *reinterpret_cast<float4*>(dst) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  const int c0 = Tile::col(t), i0 = Tile::row0(t);      // the thread loads and stores columns c0 .. c0 + 3 of RT rows
  auto load_rows = [&](const float* M, int width, float4 (&v)[Tile::RT]) {
#pragma unroll
    for (int q = 0; q < Tile::RT; ++q) {
      const int64_t gi = r0 + i0 + q;
      v[q] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (gi < rows) {
        const float* src = M + gi * ldx + c0;
        if (x_al && c0 + 4 <= width) {
          v[q] = *reinterpret_cast<const float4*>(src);
        } else {
          if (c0 < width) v[q].x = src[0];
          if (c0 + 1 < width) v[q].y = src[1];
          if (c0 + 2 < width) v[q].z = src[2];
          if (c0 + 3 < width) v[q].w = src[3];
        }
      }
    }
  };
  float4 xv[Tile::RT], out[Tile::RT];
  load_rows(X, nb, xv);
  if (do_near) {
    load_rows(near.W, near.nb_p, out);
    Tile::store(At, out);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    Tile::product(At, Bn, out);
#pragma unroll
    for (int q = 0; q < Tile::RT; ++q) {
      xv[q].x -= out[q].x; xv[q].y -= out[q].y; xv[q].z -= out[q].z; xv[q].w -= out[q].w;
    }
    __syncthreads();     // everyone is done reading At
  }
  Tile::store(At, xv);
  // (the outcome is made uniform over the block: a thread whose wait ran out must not leave while others go on)
  const bool staged = __syncthreads_and(stage_block_wait(bar, 0) ? 1 : 0) != 0;
  if (!staged) {   // the copies did not land in time: report and leave X untouched
    if (t == 0) report_status(status, SP_ERR_TIMEOUT, (int32_t)blockIdx.x, 10);
    return;
  }
  Tile::product(At, Lt, out);
  const bool x_vec = write_f32 && x_al;
#pragma unroll
  for (int q = 0; q < Tile::RT; ++q) {
    const int64_t gi = r0 + i0 + q;
    float v[4] = {out[q].x, out[q].y, out[q].z, out[q].w};
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (c0 + j >= nb) v[j] = 0.f;
    out[q] = make_float4(v[0], v[1], v[2], v[3]);
    if (gi >= rows) continue;
    if (write_f32) {
      float* dst = X + gi * ldx + c0;
      if (x_vec && c0 + 4 <= nb) {
        *reinterpret_cast<float4*>(dst) = out[q];
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (c0 + j < nb) dst[j] = v[j];
      }
    }
    if (S) {   // S + gi * lds + part * s_seg + c0 is 8-byte aligned by construction (lds, s_seg multiples of 8)
      __align__(8) __nv_bfloat16 part[3][4];
#pragma unroll
      for (int j = 0; j < 4; ++j) split3(v[j], part[0][j], part[1][j], part[2][j]);
#pragma unroll
      for (int z = 0; z < 3; ++z)
        *reinterpret_cast<uint2*>(S + gi * lds + z * s_seg + c0) = *reinterpret_cast<const uint2*>(part[z]);
    }
  }
}

template <bool TRANS, int R>
cudaError_t launch_panel_rows(float* X, int64_t ldx, int64_t rows, int nb, const float* dinv, __nv_bfloat16* S, int64_t lds,
                              int64_t s_seg, bool write_f32, int32_t* status, cudaStream_t stream, PanelNear near,
                              int batch, PanelBatch pb) {
  static PerDeviceOnce attr_once;      // one per instantiation; the attribute belongs to the device's context
  cudaError_t e = attr_once.run([] {
    return cudaFuncSetAttribute(panel_apply_kernel<TRANS, R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)pa_smem<R>(true));
  });
  if (e != cudaSuccess) return e;
  const bool with_near = TRANS && near.L != nullptr;
  launch(panel_apply_kernel<TRANS, R>, dim3((unsigned)ceil_div(rows, R), (unsigned)batch), RowTile<R>::THREADS,
                                 pa_smem<R>(with_near), stream, X, ldx, rows, nb, dinv, S, lds, s_seg, write_f32 ? 1 : 0, status, near,
                                           skip_flag(), pb);
  return cudaGetLastError();
}

// Rows per CTA: the fewest (8, 16, 32) for which `ctas` CTAs cover all rows, since every CTA stages the whole block of
// inv(L) whatever its rows; 32 beyond.
inline int panel_rows(int64_t rows, int batch, int64_t ctas) {
  return ceil_div(rows, (int64_t)8) * batch <= ctas ? 8 : ceil_div(rows, (int64_t)16) * batch <= ctas ? 16 : 32;
}

template <bool TRANS>
cudaError_t launch_panel_apply(float* X, int64_t ldx, int64_t rows, int nb, const float* dinv, __nv_bfloat16* S,
                               int64_t lds, int64_t s_seg, bool write_f32, int32_t* status, cudaStream_t stream,
                               PanelNear near = kNoNear, int batch = 1, PanelBatch pb = PanelBatch{}, int per_cta = 0) {
  if (rows <= 0) return cudaSuccess;
  count_launch();
  const bool with_near = TRANS && near.L != nullptr;
  ProfScope prof(PK_PANEL_APPLY, (with_near ? 4.0 : 2.0) * (double)rows * TB * TB, 0.0, stream);
  if (per_cta == 0) per_cta = panel_rows(rows, batch, sm_count());
  if (per_cta == 8)
    return launch_panel_rows<TRANS, 8>(X, ldx, rows, nb, dinv, S, lds, s_seg, write_f32, status, stream, near, batch, pb);
  if (per_cta == 16)
    return launch_panel_rows<TRANS, 16>(X, ldx, rows, nb, dinv, S, lds, s_seg, write_f32, status, stream, near, batch, pb);
  return launch_panel_rows<TRANS, 32>(X, ldx, rows, nb, dinv, S, lds, s_seg, write_f32, status, stream, near, batch, pb);
}

// ---------------------------------------------------------------------------------------------------------------
// Lookahead of the factorisation: the NEXT diagonal block, updated with the block column just factored, in one small
// launch, so that its factorisation does not wait for the full panel and the trailing update:
//   Lm = A21 inv(L_kk)^T  (nb2 x 128),   S = A22 - Lm Lm^T  (nb2 x nb2, fp32, into a scratch block with ld 128)
// with A21 = A[next block rows, block k columns] and A22 = A[next block, next block] as the trailing updates up to
// step k - 1 left them.  One cluster of 8 CTAs, 16 rows each: every CTA forms its rows of Lm, publishes them
// (transposed, in global scratch LmT[c][row]), the cluster meets, and every CTA forms its rows of S from all of Lm.
constexpr int NM_ROWS = 16, NM_THREADS = RowTile<NM_ROWS>::THREADS, NM_CTAS = TB / NM_ROWS;
constexpr size_t NM_SMEM = ((size_t)TB * TB + (size_t)TB * RowTile<NM_ROWS>::AP) * sizeof(float) + 16;
static_assert(NM_CTAS == 8, "one portable cluster covers the block");

// (no time limit: the CTAs of a cluster start together and each reaches the barrier, also after a wait that ran out)
__device__ __forceinline__ void cluster_meet() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Where the rows of Lm go: they are the first rows of the panel of this block column, whose own kernel therefore starts below
// them.  (A21 has all 128 columns: only the last block of a matrix is narrower.)
struct NextRows {
  __nv_bfloat16* P;      // parts at P[i * ldp + part * seg + c]
  int64_t ldp, seg;
  int vec;               // 16-byte aligned rows of A21
};

// MODE 0: both stages in one launch, the CTAs being one cluster (they meet between the stages);
// MODE 1 / MODE 2: the stages as two launches of 8 independent CTAs (for use beside persistent GEMM CTAs that hold
// most SMs, where a cluster of 8 waits for a free group of SMs).
template <int MODE>
__device__ __forceinline__ void next_diag_body(float* A21, const float* A22, int64_t lda, int nb2,
                                               const float* dinv, float* LmT, float* S, NextRows out_rows,
                                               int32_t* status) {
  extern __shared__ __align__(128) float nm_smem[];
  using Tile = RowTile<NM_ROWS>;
  constexpr int AP = Tile::AP;
  float* Lt = nm_smem;                   // Lt[k][c]
  float* At = nm_smem + TB * TB;         // At[k][row]
  uint64_t* bar = reinterpret_cast<uint64_t*>(At + TB * AP);
  const int t = threadIdx.x;
  const int i0 = (int)blockIdx.x * NM_ROWS;
  const int c0 = Tile::col(t), ir = Tile::row0(t);      // columns c0 .. c0 + 3 of rows i0 + ir .. + RT - 1
  float4 out[Tile::RT];
  if (MODE != 2) {
    // ---- stage 1: rows i0 .. i0 + 15 of Lm; Lt[k][c] = inv(L)[c][k] comes in by bulk copies
    if (t == 0) stage_bar_init(bar);
    __syncthreads();
    if (t == 0) stage_block_issue(Lt, dinv + TB * TB, bar);
#pragma unroll
    for (int q = 0; q < Tile::RT; ++q) {
      const int i = i0 + ir + q;
      float v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = i < nb2 ? A21[(int64_t)i * lda + c0 + j] : 0.f;
      out[q] = make_float4(v[0], v[1], v[2], v[3]);
    }
    Tile::store(At, out);
  }
  // this thread's entries of A22
  float4 base[Tile::RT];
  if (MODE != 1) {
#pragma unroll
    for (int q = 0; q < Tile::RT; ++q) {
      const int i = i0 + ir + q;
      float v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = (i < nb2 && c0 + j <= i) ? A22[(int64_t)i * lda + c0 + j] : 0.f;
      base[q] = make_float4(v[0], v[1], v[2], v[3]);
    }
  }
  if (MODE != 2) {
    const bool staged = __syncthreads_and(stage_block_wait(bar, 0) ? 1 : 0) != 0;
    if (!staged && t == 0) report_status(status, SP_ERR_TIMEOUT, (int32_t)blockIdx.x, 11);
    // (a CTA whose copies did not land still goes on to the barrier below; its rows are then wrong and the status
    //  says so)
    Tile::product(At, Lt, out);
    __syncthreads();   // everyone is done with At and Lt
    Tile::store(At, out);                          // own rows, left operand of stage 2
    Tile::store_transposed(LmT + i0, TB, out);     // for the other CTAs
    // the panel's result for these rows: fp32 in place, bf16 parts
#pragma unroll
    for (int q = 0; q < Tile::RT; ++q) {
      const int i = i0 + ir + q;
      if (i >= nb2) continue;
      const float v[4] = {out[q].x, out[q].y, out[q].z, out[q].w};
      float* dst = A21 + (int64_t)i * lda + c0;
      if (out_rows.vec) {
        *reinterpret_cast<float4*>(dst) = out[q];
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) dst[j] = v[j];
      }
      __align__(8) __nv_bfloat16 part[3][4];
#pragma unroll
      for (int j = 0; j < 4; ++j) split3(v[j], part[0][j], part[1][j], part[2][j]);
#pragma unroll
      for (int z = 0; z < 3; ++z)
        *reinterpret_cast<uint2*>(out_rows.P + i * out_rows.ldp + z * out_rows.seg + c0) = *reinterpret_cast<const uint2*>(part[z]);
    }
    if (MODE == 1) return;
    cluster_meet();
  }
  // ---- stage 2: rows i0 .. i0 + 15 of S; Lt[c][j] = Lm[j][c]
  {
    const float4* src = reinterpret_cast<const float4*>(LmT);
    float4* dst = reinterpret_cast<float4*>(Lt);
#pragma unroll 16
    for (int q = 0; q < TB * TB / 4 / NM_THREADS; ++q) dst[t + q * NM_THREADS] = __ldcg(src + t + q * NM_THREADS);
    if (MODE == 2)     // own rows of Lm come from the first launch
      for (int e = t; e < NM_ROWS * TB; e += NM_THREADS) {
        const int c = e / NM_ROWS, i = e % NM_ROWS;
        At[c * AP + i] = __ldcg(&LmT[(int64_t)c * TB + i0 + i]);
      }
  }
  __syncthreads();
  Tile::product(At, Lt, out);
#pragma unroll
  for (int q = 0; q < Tile::RT; ++q) {
    const int i = i0 + ir + q;
    const float d[4] = {base[q].x - out[q].x, base[q].y - out[q].y, base[q].z - out[q].z, base[q].w - out[q].w};
    float v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = (i < nb2 && c0 + j <= i) ? d[j] : 0.f;
    *reinterpret_cast<float4*>(&S[i * TB + c0]) = make_float4(v[0], v[1], v[2], v[3]);
  }
}

__global__ void __cluster_dims__(NM_CTAS, 1, 1) __launch_bounds__(NM_THREADS)
    chol_next_diag_kernel(float* A21, const float* A22, int64_t lda, int nb2,
                          const float* dinv, float* LmT, float* S, NextRows out_rows, int32_t* status,
                          const int32_t* skip) {
  kernel_begin();
  if (skip != nullptr && *skip != 0) return;
  next_diag_body<0>(A21, A22, lda, nb2, dinv, LmT, S, out_rows, status);
}
__global__ void __launch_bounds__(NM_THREADS)
    chol_next_diag_stage1_kernel(float* A21, int64_t lda, int nb2, const float* dinv, float* LmT,
                                 NextRows out_rows, int32_t* status, const int32_t* skip) {
  kernel_begin();
  if (skip != nullptr && *skip != 0) return;
  next_diag_body<1>(A21, nullptr, lda, nb2, dinv, LmT, nullptr, out_rows, status);
}
__global__ void __launch_bounds__(NM_THREADS)
    chol_next_diag_stage2_kernel(const float* A22, int64_t lda, int nb2, float* LmT, float* S,
                                 const int32_t* skip) {
  kernel_begin();
  if (skip != nullptr && *skip != 0) return;
  next_diag_body<2>(nullptr, A22, lda, nb2, nullptr, LmT, S, NextRows{}, nullptr);
}

// The six kept part products of two three-part operands: A parts (hi, hi, mid, hi, lo, mid) against B parts
// (hi, mid, hi, lo, hi, mid).
constexpr int kPartA[6] = {0, 0, 1, 0, 2, 1};
constexpr int kPartB[6] = {0, 1, 0, 2, 0, 1};

}  // namespace

int64_t chol_tc_pad(int64_t n) { return (n + TB - 1) / TB * TB; }

sp_status potrf_lower_tc(float* A, int64_t n, int64_t lda, float* dinv, void* Pv, int32_t* status_dev,
                         cudaStream_t stream, const SolveAssist* assist, int64_t m_extra, bool split_lookahead) {
  __nv_bfloat16* P = reinterpret_cast<__nv_bfloat16*>(Pv);
  const int64_t np = chol_tc_pad(n), ldp = 3 * np;
  const int64_t nblk = ceil_div(n, (int64_t)TB);
  const int32_t* skip = skip_flag();
  static PerDeviceOnce attr_once;
  if (attr_once.run([] {
        cudaError_t e = cudaFuncSetAttribute(chol_diag128_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)Diag::SMEM);
        if (e == cudaSuccess)
          e = cudaFuncSetAttribute(chol_next_diag_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)NM_SMEM);
        if (e == cudaSuccess)
          e = cudaFuncSetAttribute(chol_next_diag_stage1_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)NM_SMEM);
        if (e == cudaSuccess)
          e = cudaFuncSetAttribute(chol_next_diag_stage2_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)NM_SMEM);
        return e;
      }) != cudaSuccess)
    return SP_ERR_CUDA;
#define SP_CUDA_OK(x) do { if ((x) != cudaSuccess) return SP_ERR_CUDA; } while (0)
  // With an assisting stream the chain of diagonal blocks runs ahead: after block k is factored, a small kernel
  // forms the next diagonal block (into scratch behind the inverses), and the next factorisation starts from it while
  // the full panel and the trailing update of step k run on the assisting stream.
  float* S = dinv + nblk * 2 * TB * TB;      // [128, 128] next diagonal block
  float* LmT = S + TB * TB;                  // [128, 128] scratch of the lookahead kernel
  bool rec[2] = {false, false};
  // Far part of a step's trailing update on a stream of its own: it adds into the matrix through the GEMM's atomic TMA
  // reduction (which needs 16-byte aligned rows and a width that is a multiple of 4).  What must see it complete waits for its
  // events: the lookahead kernel of step kb reads block (kb+1, kb+1), last touched by the far update of step kb - 2, and
  // the near update of step kb adds to the first block column of the far update of step kb - 1.
  // The far GEMM leaves a few SM pairs to the kernels of the chain, which would otherwise wait for its tiles to end.
  const bool far_apart = assist && assist->far_stream && n % 4 == 0 && lda % 4 == 0 &&
                         (reinterpret_cast<uintptr_t>(A) & 15u) == 0 && !reproducible_mode();
  bool far_rec[2] = {false, false};
  constexpr int kFarPairs = 64;
  // Two-level blocking for large systems: the trailing update of a step is bound by the read-modify-write of the fp32
  // matrix when K is only 128 (n = 28672: 430 GB per factorisation).  With OB > 1 the steps of an outer block of OB
  // diagonal blocks update only the rest of that outer block's columns at once; everything to the right of it gets
  // ONE update per outer block with K = OB * 128, which divides that traffic by OB.
  const int64_t OB = (assist && n >= kOuterMinN) ? kOuterBlocks : 1;
  for (int64_t kb = 0; kb < nblk; ++kb) {
    const int64_t k0 = kb * TB;
    const int nb = (int)((n - k0 < TB) ? (n - k0) : TB);
    float* dk = dinv + kb * 2 * TB * TB;
    const int64_t ob_start = kb / OB * OB;
    const int64_t ob_end_blk = (ob_start + OB < nblk) ? ob_start + OB : nblk;
    const int64_t ob_end_col = (ob_end_blk * TB < n) ? ob_end_blk * TB : n;
    const bool outer = OB > 1;
    const bool inner_last = outer && kb == ob_end_blk - 1;
    const bool inner_first = outer && kb == ob_start;
    {
      // the first block of an outer block is read from the matrix itself, once the first columns of the previous
      // outer block's update have landed; every other block comes from the lookahead kernel's scratch
      const bool from_scratch = assist && kb > 0 && !inner_first;
      if (assist && inner_first && kb > 0) SP_CUDA_OK(cudaStreamWaitEvent(stream, assist->near_done, 0));
      count_launch();
      ProfScope prof(PK_CHOL_DIAG, (double)nb * nb * nb * (2.0 / 3.0), 0.0, stream);
      launch(chol_diag128_kernel, 1, Diag::THREADS, Diag::SMEM, stream, from_scratch ? S : A + k0 * lda + k0,
                                                                  from_scratch ? (int64_t)TB : lda, nb, dk, k0,
                                                                  status_dev, skip, 0, 0);
      if (cudaGetLastError() != cudaSuccess) return SP_ERR_CUDA;
    }
    const int64_t rem = n - k0 - nb;
    // rows below the block that the panel covers: the rest of the matrix and the m_extra appended rows (right-hand
    // sides of a system X L^T = B stored below A: the panel and the trailing update are exactly their forward
    // substitution, so it costs no steps of its own)
    const int64_t prow = rem + m_extra;
    if (prow <= 0) break;
    cudaStream_t sb = stream;
    // last block with appended rows: their panel runs on `stream`, behind the assisting stream's last update
    if (assist && rem <= 0 && kb >= 1) {
      SP_CUDA_OK(cudaStreamWaitEvent(stream, assist->rest_done[(kb - 1) & 1], 0));
      for (int q = 0; q < 2; ++q)
        if (far_rec[q]) SP_CUDA_OK(cudaStreamWaitEvent(stream, assist->far_done[q], 0));
    }
    // rows of the panel that the lookahead kernel takes: the next diagonal block's
    const int64_t ahead = assist && rem > 0 && !inner_last ? (rem < TB ? rem : TB) : 0;
    if (assist && rem > 0) {
      if (ahead > 0) {
        // next diagonal block: it reads blocks (kb+1, kb) and (kb+1, kb+1), i.e. the first two block columns of the
        // trailing update of step kb - 1, which that step issues first and signals on their own
        if (kb >= 1) SP_CUDA_OK(cudaStreamWaitEvent(stream, assist->near_done, 0));
        if (far_rec[kb & 1]) SP_CUDA_OK(cudaStreamWaitEvent(stream, assist->far_done[kb & 1], 0));   // far update of step kb - 2
        const int nb2 = (int)ahead;
        float* A21 = A + (k0 + nb) * lda + k0;
        const NextRows rows{P + (k0 + nb) * ldp + k0, ldp, np, lda % 4 == 0 && (reinterpret_cast<uintptr_t>(A) & 15u) == 0};
        count_launch();
        ProfScope prof(PK_PANEL_APPLY, 4.0 * TB * TB * TB, 0.0, stream);
        if (!split_lookahead) {
          launch(chol_next_diag_kernel, NM_CTAS, NM_THREADS, NM_SMEM, stream, A21, A21 + nb, lda, nb2, dk, LmT, S, rows,
                 status_dev, skip);
        } else {
          launch(chol_next_diag_stage1_kernel, NM_CTAS, NM_THREADS, NM_SMEM, stream, A21, lda, nb2, dk, LmT, rows,
                 status_dev, skip);
          count_launch();
          launch(chol_next_diag_stage2_kernel, NM_CTAS, NM_THREADS, NM_SMEM, stream, A21 + nb, lda, nb2, LmT, S, skip);
        }
        if (cudaGetLastError() != cudaSuccess) return SP_ERR_CUDA;
      }
      // The panel needs the diagonal block alone, but it starts behind the lookahead kernel: the next diagonal block waits for
      // that one, and beside it the panel's CTAs would be in its way (its cluster needs eight SMs that have room at once).
      // Panel behind / beside it: a solve of 4096 unknowns and 1024 right-hand sides 1.71 / 1.86 ms, of 2048 and 4096 1.04 /
      // 1.17, an ADMM step 2048 x 8192 14.10 / 14.27, 1096 x 4376 and 768 x 3072 equal within 1 %.
      SP_CUDA_OK(cudaEventRecord(assist->panel_done, stream));
      sb = assist->stream;
      SP_CUDA_OK(cudaStreamWaitEvent(sb, assist->panel_done, 0));
    }
    // L21 = A21 inv(L11)^T, fp32 in place and as bf16 parts in P[k0+nb.., part * np + k0 ..]
    const int64_t p0 = k0 + nb + ahead;
    if (launch_panel_apply<false>(A + p0 * lda + k0, lda, prow - ahead, nb, dk, P + p0 * ldp + k0, ldp, np, true,
                                  status_dev, sb) != cudaSuccess)
      return SP_ERR_CUDA;
    if (rem <= 0) break;     // last block: the appended rows are done, nothing is left to update
    if (far_apart && !outer && rem > 2 * TB) SP_CUDA_OK(cudaEventRecord(assist->far_go, sb));   // the panel's parts exist
    // the far update of the step before has added to the columns that this step's near update adds to: every entry receives
    // its updates in step order, whatever the streams' timing
    if (kb >= 1 && far_rec[(kb - 1) & 1]) SP_CUDA_OK(cudaStreamWaitEvent(sb, assist->far_done[(kb - 1) & 1], 0));
    // A22 -= L21 L21^T on the lower triangle
    TcOperand ta{P + (k0 + nb) * ldp, ldp, true}, tb{P + (k0 + nb) * ldp, ldp, true};
    ta.kext = tb.kext = ldp;
    ta.mnext = prow;
    tb.mnext = rem;
    TcSegments sg;
    sg.nseg = 6;
    for (int q = 0; q < 6; ++q) {
      sg.a_k[q] = (int32_t)(kPartA[q] * np + k0);
      sg.b_k[q] = (int32_t)(kPartB[q] * np + k0);
    }
    float* A22 = A + (k0 + nb) * lda + (k0 + nb);
    constexpr int64_t kNear = 2 * TB;     // block columns of the update that the next step's chain kernels read
    if (outer) {
      // (a) the rest of this outer block's columns, all rows below: K = 128
      const int64_t cols_in = ob_end_col - (k0 + nb);
      if (cols_in > 0) {
        tb.mnext = cols_in;
        sp_status st = gemm_tc(prow, cols_in, TB, -1.f, ta, tb, 1.f, Operand{A22, SP_F32, lda, 1},
                               OutOperand{A22, SP_F32, lda}, true, status_dev, sb, &sg,
                               (2.0 * (double)prow * (double)cols_in - (double)cols_in * (double)cols_in) * (double)nb);
        if (st != SP_OK) return st;
        SP_CUDA_OK(cudaEventRecord(assist->near_done, sb));
      }
      // (b) after the outer block's last step: everything to its right, K = the outer block's width
      const int64_t cols_out = n - ob_end_col;
      if (inner_last && cols_out > 0) {
        const int64_t o0 = ob_start * TB, kw = ob_end_col - o0, prow_out = cols_out + m_extra;
        TcSegments so;
        so.nseg = 6;
        for (int q = 0; q < 6; ++q) {
          so.a_k[q] = (int32_t)(kPartA[q] * np + o0);
          so.b_k[q] = (int32_t)(kPartB[q] * np + o0);
        }
        float* Aout = A + ob_end_col * lda + ob_end_col;
        const int64_t wn = cols_out < kNear ? cols_out : kNear;
        TcOperand na{P + ob_end_col * ldp, ldp, true}, nbo{P + ob_end_col * ldp, ldp, true};
        na.kext = nbo.kext = ldp;
        na.mnext = prow_out;
        nbo.mnext = wn;
        sp_status st = gemm_tc(prow_out, wn, kw, -1.f, na, nbo, 1.f, Operand{Aout, SP_F32, lda, 1},
                               OutOperand{Aout, SP_F32, lda}, true, status_dev, sb, &so,
                               (2.0 * (double)prow_out * (double)wn - (double)wn * (double)wn) * (double)kw);
        if (st != SP_OK) return st;
        SP_CUDA_OK(cudaEventRecord(assist->near_done, sb));
        if (cols_out > wn) {
          TcOperand fa{P + (ob_end_col + wn) * ldp, ldp, true}, fb{P + (ob_end_col + wn) * ldp, ldp, true};
          fa.kext = fb.kext = ldp;
          fa.mnext = prow_out - wn;
          fb.mnext = cols_out - wn;
          float* Afar = Aout + wn * lda + wn;
          const double fr = (double)(cols_out - wn);
          st = gemm_tc(prow_out - wn, cols_out - wn, kw, -1.f, fa, fb, 1.f, Operand{Afar, SP_F32, lda, 1},
                       OutOperand{Afar, SP_F32, lda}, true, status_dev, sb, &so,
                       (fr * fr + 2.0 * (double)m_extra * fr) * (double)kw);
          if (st != SP_OK) return st;
        }
      }
    } else if (assist && rem > kNear) {
      // two launches: the first two block columns (all rows below), signalled at once, then the rest
      tb.mnext = kNear;
      sp_status st = gemm_tc(prow, kNear, TB, -1.f, ta, tb, 1.f, Operand{A22, SP_F32, lda, 1},
                             OutOperand{A22, SP_F32, lda}, true, status_dev, sb, &sg,
                             (2.0 * (double)prow * (double)kNear - (double)kNear * (double)kNear) * (double)nb);
      if (st != SP_OK) return st;
      SP_CUDA_OK(cudaEventRecord(assist->near_done, sb));
      cudaStream_t sf = sb;
      if (far_apart) {
        sf = assist->far_stream;
        SP_CUDA_OK(cudaStreamWaitEvent(sf, assist->far_go, 0));
      }
      // (one launch: as two, the block columns that the next near update waits for first, it fills the SMs worse, and a solve of
      // 8192 unknowns takes 6.35 instead of 6.04 ms)
      const int64_t fw = rem - kNear, r0 = k0 + nb + kNear, rows_f = prow - kNear;
      TcOperand fa{P + r0 * ldp, ldp, true}, fb{P + r0 * ldp, ldp, true};
      fa.kext = fb.kext = ldp;
      fa.mnext = rows_f;
      fb.mnext = fw;
      float* Afar = A + r0 * lda + r0;
      st = gemm_tc(rows_f, fw, TB, -1.f, fa, fb, 1.f, Operand{Afar, SP_F32, lda, 1}, OutOperand{Afar, SP_F32, lda}, true,
                   status_dev, sf, &sg, (double)fw * (2.0 * (double)rows_f - (double)fw) * (double)nb, far_apart ? kFarPairs : 0);
      if (st != SP_OK) return st;
      if (far_apart) {
        SP_CUDA_OK(cudaEventRecord(assist->far_done[kb & 1], sf));
        far_rec[kb & 1] = true;
      }
    } else {
      sp_status st = gemm_tc(prow, rem, TB, -1.f, ta, tb, 1.f, Operand{A22, SP_F32, lda, 1},
                             OutOperand{A22, SP_F32, lda}, true, status_dev, sb, &sg,
                             ((double)rem * (double)rem + 2.0 * (double)m_extra * (double)rem) * (double)nb);
      if (st != SP_OK) return st;
      if (assist) SP_CUDA_OK(cudaEventRecord(assist->near_done, sb));
    }
    if (assist) {
      SP_CUDA_OK(cudaEventRecord(assist->rest_done[kb & 1], sb));
      rec[kb & 1] = true;
    }
  }
  // the factor is complete on `stream` once the assisting stream has drained
  for (int q = 0; q < 2; ++q) {
    if (assist && rec[q]) SP_CUDA_OK(cudaStreamWaitEvent(stream, assist->rest_done[q], 0));
    if (far_rec[q]) SP_CUDA_OK(cudaStreamWaitEvent(stream, assist->far_done[q], 0));
  }
#undef SP_CUDA_OK
  return SP_OK;
}

sp_status potrs_right_tc(float* X, int64_t m, int64_t n, int64_t ldx, const void* Pv, const float* dinv, void* Xsv,
                         int32_t* status_dev, cudaStream_t stream, const SolveAssist* assist, bool forward_done,
                         const float* Lf, int64_t ldl, int64_t n_factor) {
  const __nv_bfloat16* P = reinterpret_cast<const __nv_bfloat16*>(Pv);
  __nv_bfloat16* Xs = reinterpret_cast<__nv_bfloat16*>(Xsv);
  if (n_factor > n && n % TB != 0) return SP_ERR_SHAPE;
  const int64_t np = chol_tc_pad(n_factor > n ? n_factor : n), ldp = 3 * np;
  const int64_t lds = 3 * TB;
  const int64_t nblk = ceil_div(n, (int64_t)TB);
  // Every step applies the inverse diagonal block to one block column (panel) and then updates the columns still to
  // come.  With an assisting stream the update is cut in two: the next block column, which the next panel needs, stays
  // on `stream`; the rest runs on the assisting stream and overlaps the next panel.  Panel jj then needs the "rest"
  // update of step jj - 2 (and reuses its buffer of bf16 parts), which is what the two alternating events order.
#define SP_CUDA_OK(x) do { if ((x) != cudaSuccess) return SP_ERR_CUDA; } while (0)
  // The tensor-core update adds atomically only through its TMA reduction, which needs 16-byte aligned rows of X;
  // without it everything stays on one stream.
  const bool x_al16 = (ldx % 4 == 0) && ((reinterpret_cast<uintptr_t>(X) & 15u) == 0);
  if (!x_al16) assist = nullptr;
  // Reproducible mode stays on one stream, where every column receives its updates in step order.  With an assisting stream
  // a far update and the next step's near update add into the same columns in an order that depends on timing, unless the
  // panel pulls the near update (fuse_near: added last, in either mode).
  if (reproducible_mode()) assist = nullptr;
  // Backward sweep: the update by the previous block column can ride in the panel kernel (fp32, from the fp32 factor)
  // when the factor's rows are 16-byte aligned too.
  // (its 144 KB of shared memory allow one CTA per SM: only while all row blocks fit in one wave)
  const bool fuse_near = Lf != nullptr && x_al16 && (ldl % 4 == 0) && ((reinterpret_cast<uintptr_t>(Lf) & 15u) == 0) &&
                         ceil_div(m, (int64_t)32) <= sm_count();
  // Backward sweep: a panel runs beside the far update of the step before, whose CTAs take a whole SM each; one that has to
  // wait for SMs lengthens the chain by the update's time.  So the panel gets half of the SMs and the update the rest,
  // unless the update has so many tiles that the two one after the other, each with all SMs, are shorter.  Measured on the
  // step's kernels: 8 us and 6.2 us for every round of tiles for the update, 12 us for the panel.
  const int64_t sms = sm_count();
  const int rows_beside = panel_rows(m, 1, sms / 2);
  const int64_t beside_pairs = (sms - ceil_div(m, (int64_t)rows_beside)) / 2;
  auto tiles_of = [&](int64_t w) { return ceil_div(m, (int64_t)256) * ceil_div(w, (int64_t)256); };
  auto runs_beside = [&](int64_t w) {
    if (beside_pairs < 1) return false;
    return 6.2 * (double)ceil_div(tiles_of(w), beside_pairs) < 12.0 + 6.2 * (double)ceil_div(tiles_of(w), sms / 2);
  };
  bool rec[2] = {false, false};
  auto run_sweep = [&](bool forward) -> sp_status {
    for (int64_t step = 0; step < nblk; ++step) {
      const int64_t jb = forward ? step : nblk - 1 - step;
      const int64_t j0 = jb * TB;
      const int nb = (int)((n - j0 < TB) ? (n - j0) : TB);
      const float* dj = dinv + jb * 2 * TB * TB;
      __nv_bfloat16* Xcur = Xs + (step & 1) * m * lds;
      if (assist && rec[step & 1]) SP_CUDA_OK(cudaStreamWaitEvent(stream, assist->rest_done[step & 1], 0));
      // columns still to be updated: [lo, hi)
      const int64_t lo = forward ? j0 + nb : 0, hi = forward ? n : j0;
      // backward: the near columns are the whole block before j (TB wide), which the next panel updates itself
      const bool near_in_panel = !forward && fuse_near;
      PanelNear pn = kNoNear;
      if (near_in_panel && j0 + nb < n) {
        const int64_t p0 = j0 + nb;
        pn = PanelNear{Lf + p0 * ldl + j0, ldl, X + p0, (int)((n - p0 < TB) ? n - p0 : TB)};
      }
      cudaError_t e = forward ? launch_panel_apply<false>(X + j0, ldx, m, nb, dj, Xcur, lds, TB, true, status_dev, stream)
                              : launch_panel_apply<true>(X + j0, ldx, m, nb, dj, Xcur, lds, TB, true, status_dev, stream,
                                                         pn, 1, PanelBatch{},
                                                         near_in_panel && assist && runs_beside(j0) ? rows_beside : 0);
      if (e != cudaSuccess) return SP_ERR_CUDA;
      if (hi <= lo) break;
      if (assist) SP_CUDA_OK(cudaEventRecord(assist->panel_done, stream));
      TcOperand ta{Xcur, lds, true};
      ta.kext = lds;
      ta.mnext = m;
      // near part (next block column) and far part of the update
      const int64_t wn = (hi - lo < TB) ? hi - lo : TB;
      const int64_t near_lo = forward ? lo : hi - wn, far_lo = forward ? lo + wn : lo, far_w = hi - lo - wn;
      for (int part = 0; part < 2; ++part) {
        const int64_t c0 = part == 0 ? near_lo : far_lo, w = part == 0 ? wn : far_w;
        if (w <= 0 || (part == 0 && near_in_panel)) continue;
        const bool on_assist = assist && part == 1;
        cudaStream_t st_run = on_assist ? assist->stream : stream;
        if (on_assist) SP_CUDA_OK(cudaStreamWaitEvent(st_run, assist->panel_done, 0));
        TcSegments sg;
        sg.nseg = 6;
        TcOperand tb{nullptr, ldp, forward};
        if (forward) {
          // X[:, c0:c0+w] -= Y_j L[c0:c0+w, j0:j0+nb]^T : B(k, c) = L[c0 + c, j0 + k], K-major rows of P
          tb.ptr = P + c0 * ldp;
          tb.kext = ldp;
          tb.mnext = w;
          for (int q = 0; q < 6; ++q) {
            sg.a_k[q] = kPartA[q] * TB;
            sg.b_k[q] = (int32_t)(kPartB[q] * np + j0);
          }
        } else {
          // X[:, c0:c0+w] -= W_j L[j0:j0+nb, c0:c0+w] : B(k, c) = L[j0 + k, c0 + c], rows of P, columns (N) contiguous
          tb.ptr = P + j0 * ldp;
          tb.kext = n - j0;      // rows of L that exist; beyond them the tensor map returns zero
          tb.mnext = ldp;
          for (int q = 0; q < 6; ++q) {
            sg.a_k[q] = kPartA[q] * TB;
            sg.b_mn[q] = (int32_t)(kPartB[q] * np + c0);
          }
        }
        float* Xc = X + c0;
        sp_status stt = gemm_tc(m, w, TB, -1.f, ta, tb, 1.f, Operand{Xc, SP_F32, ldx, 1}, OutOperand{Xc, SP_F32, ldx},
                                false, status_dev, st_run, &sg, 2.0 * (double)m * (double)w * (double)nb,
                                on_assist && near_in_panel && runs_beside(w) ? (int)beside_pairs : 0);
        if (stt != SP_OK) return stt;
        if (on_assist) {
          SP_CUDA_OK(cudaEventRecord(assist->rest_done[step & 1], st_run));
          rec[step & 1] = true;
        }
      }
    }
    // the sweep is complete on `stream` once the far updates still in flight have landed
    for (int q = 0; q < 2; ++q)
      if (assist && rec[q]) {
        SP_CUDA_OK(cudaStreamWaitEvent(stream, assist->rest_done[q], 0));
        rec[q] = false;
      }
    return SP_OK;
  };
  // Two-level backward sweep of large systems: with K = 128 a far update is bound by the read-modify-write of X (n = 28672, 7168
  // right-hand sides: 0.45 ms for 0.3 TFLOP, 224 times).  The panels of an outer block update the rest of that block
  // only, and everything to its left receives one update per outer block with K = 512.
  auto backward_outer = [&]() -> sp_status {
    constexpr int64_t OBW = kOuterBlocks * TB, ldo = 3 * OBW;
    // X[:, c0:c0+w] -= W[:, a0:a0+K of the outer block] L[r0:r0+K, c0:c0+w]
    auto update = [&](int64_t a0, int64_t r0, int64_t K, int64_t c0, int64_t w) -> sp_status {
      if (w <= 0) return SP_OK;
      TcOperand ta{Xs, ldo, true}, tb{P + r0 * ldp, ldp, false};
      ta.kext = ldo;
      ta.mnext = m;
      tb.kext = n - r0;
      tb.mnext = ldp;
      TcSegments sg;
      sg.nseg = 6;
      for (int q = 0; q < 6; ++q) {
        sg.a_k[q] = (int32_t)(kPartA[q] * OBW + a0);
        sg.b_mn[q] = (int32_t)(kPartB[q] * np + c0);
      }
      return gemm_tc(m, w, K, -1.f, ta, tb, 1.f, Operand{X + c0, SP_F32, ldx, 1}, OutOperand{X + c0, SP_F32, ldx}, false,
                     status_dev, stream, &sg, 2.0 * (double)m * (double)w * (double)K);
    };
    for (int64_t b1 = nblk; b1 > 0;) {
      const int64_t b0 = (b1 - 1) / kOuterBlocks * kOuterBlocks, o0 = b0 * TB;
      for (int64_t jb = b1 - 1; jb >= b0; --jb) {
        const int64_t j0 = jb * TB, p0 = j0 + TB;
        const int nb = (int)((n - j0 < TB) ? (n - j0) : TB);
        PanelNear pn = kNoNear;
        if (fuse_near && jb + 1 < b1) pn = PanelNear{Lf + p0 * ldl + j0, ldl, X + p0, (int)((n - p0 < TB) ? n - p0 : TB)};
        if (launch_panel_apply<true>(X + j0, ldx, m, nb, dinv + jb * 2 * TB * TB, Xs + (j0 - o0), ldo, OBW, true,
                                     status_dev, stream, pn) != cudaSuccess)
          return SP_ERR_CUDA;
        sp_status r = update(j0 - o0, j0, TB, o0, j0 - o0 - (fuse_near ? TB : 0));
        if (r != SP_OK) return r;
      }
      sp_status r = update(0, o0, (b1 - b0) * TB, 0, o0);
      if (r != SP_OK) return r;
      b1 = b0;
    }
    return SP_OK;
  };
  if (!forward_done) {               // (done already when X rode along with the factorisation as appended rows)
    sp_status r = run_sweep(true);    // Y L^T = X, block columns left to right
    if (r != SP_OK) return r;
  }
  return n >= kOuterMinN ? backward_outer() : run_sweep(false);     // W L = Y, block columns right to left
#undef SP_CUDA_OK
}


// ---------------------------------------------------------------------------------------------------------------
// B independent systems of one size, solved together: every step of the factorisation and of the backward sweep is
// one launch over all systems (diagonal blocks: one CTA per system; panels: grid.y = systems; updates: one batched
// tensor-core launch), so the parallelism comes from the batch and no lookahead or second stream is used.
// Layout: system b at A + b * a_bs ([n + m, n] fp32, the m right-hand sides below the matrix, lda = n), its bf16 parts
// at P + b * (np + m) * 3 np, its inverse diagonal blocks at dinv + b * d_bs, its sweep buffers at Xs + b * 2 m 3 TB.
// n must be a multiple of 128 here (the callers' systems are d x d with d % 128 == 0; others take the plain path).
sp_status potrf_potrs_tc_batched(float* A, int64_t n, int64_t m, int batch, int64_t a_bs, float* dinv, int64_t d_bs,
                                 void* Pv, void* Xsv, int32_t* status_dev, cudaStream_t stream) {
  if (n % TB != 0 || batch < 1 || m < 1) return SP_ERR_SHAPE;
  __nv_bfloat16* P = reinterpret_cast<__nv_bfloat16*>(Pv);
  __nv_bfloat16* Xs = reinterpret_cast<__nv_bfloat16*>(Xsv);
  const int64_t np = n, ldp = 3 * np, lda = n;
  const int64_t p_bs = (np + m) * ldp;
  const int64_t nblk = n / TB;
  const int32_t* skip = skip_flag();
  static PerDeviceOnce attr_once;
  if (attr_once.run([] {
        return cudaFuncSetAttribute(chol_diag128_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Diag::SMEM);
      }) != cudaSuccess)
    return SP_ERR_CUDA;
  TcBatch bt;
  bt.nb0 = batch; bt.nb1 = 1;
  bt.a_s0 = bt.b_s0 = p_bs; bt.a_s1 = bt.b_s1 = p_bs;
  bt.c_s0 = bt.cin_s0 = a_bs; bt.c_s1 = bt.cin_s1 = a_bs;
  bt.a_planes = bt.b_planes = 1; bt.a_plane = bt.b_plane = 0;
  // ---- factorisation; the appended rows receive their forward substitution on the way
  for (int64_t kb = 0; kb < nblk; ++kb) {
    const int64_t k0 = kb * TB;
    float* dk = dinv + kb * 2 * TB * TB;
    count_launch();
    launch(chol_diag128_kernel, batch, Diag::THREADS, Diag::SMEM, stream, A + k0 * lda + k0, lda, TB, dk, k0, status_dev, skip,
                                                                  a_bs, d_bs);
    if (cudaGetLastError() != cudaSuccess) return SP_ERR_CUDA;
    const int64_t rem = n - k0 - TB, prow = rem + m;
    PanelBatch pb;
    pb.x = a_bs; pb.dinv = d_bs; pb.s = p_bs;
    if (launch_panel_apply<false>(A + (k0 + TB) * lda + k0, lda, prow, TB, dk, P + (k0 + TB) * ldp + k0, ldp, np, true,
                                  status_dev, stream, kNoNear, batch, pb) != cudaSuccess)
      return SP_ERR_CUDA;
    if (rem <= 0) break;
    TcOperand ta{P + (k0 + TB) * ldp, ldp, true}, tb{P + (k0 + TB) * ldp, ldp, true};
    ta.kext = tb.kext = ldp;
    ta.mnext = prow;
    tb.mnext = rem;
    TcSegments sg;
    sg.nseg = 6;
    for (int q = 0; q < 6; ++q) {
      sg.a_k[q] = (int32_t)(kPartA[q] * np + k0);
      sg.b_k[q] = (int32_t)(kPartB[q] * np + k0);
    }
    float* A22 = A + (k0 + TB) * lda + (k0 + TB);
    sp_status st = gemm_tc(prow, rem, TB, -1.f, ta, tb, 1.f, Operand{A22, SP_F32, lda, 1}, OutOperand{A22, SP_F32, lda},
                           true, status_dev, stream, &sg,
                           ((double)rem * rem + 2.0 * (double)m * rem) * TB * batch, 0, &bt);
    if (st != SP_OK) return st;
  }
  // ---- backward sweep W L = Y on the appended rows, block columns right to left
  float* X = A + n * lda;                       // [m, n] per system
  const int64_t lds = 3 * TB, xs_bs = 2 * m * lds;
  const bool fuse_near = ceil_div(m, (int64_t)32) * batch <= sm_count();
  TcBatch bs = bt;
  bs.a_s0 = bs.a_s1 = xs_bs;
  for (int64_t step = 0; step < nblk; ++step) {
    const int64_t jb = nblk - 1 - step, j0 = jb * TB;
    const float* dj = dinv + jb * 2 * TB * TB;
    __nv_bfloat16* Xcur = Xs + (step & 1) * m * lds;
    PanelNear pn = kNoNear;
    if (fuse_near && step > 0) pn = PanelNear{A + (j0 + TB) * lda + j0, lda, X + j0 + TB, TB};
    PanelBatch pb;
    pb.x = a_bs; pb.dinv = d_bs; pb.s = xs_bs; pb.near_l = a_bs;
    if (launch_panel_apply<true>(X + j0, lda, m, TB, dj, Xcur, lds, TB, true, status_dev, stream, pn, batch, pb) !=
        cudaSuccess)
      return SP_ERR_CUDA;
    const int64_t w = fuse_near ? j0 - TB : j0;     // columns still to be updated by a product: [0, w)
    if (w <= 0) continue;
    TcOperand ta{Xcur, lds, true}, tb{P + j0 * ldp, ldp, false};
    ta.kext = lds;
    ta.mnext = m;
    tb.kext = n - j0;
    tb.mnext = ldp;
    TcSegments sg;
    sg.nseg = 6;
    for (int q = 0; q < 6; ++q) {
      sg.a_k[q] = kPartA[q] * TB;
      sg.b_mn[q] = (int32_t)(kPartB[q] * np);
    }
    sp_status st = gemm_tc(m, w, TB, -1.f, ta, tb, 1.f, Operand{X, SP_F32, lda, 1}, OutOperand{X, SP_F32, lda}, false,
                           status_dev, stream, &sg, 2.0 * (double)m * w * TB * batch, 0, &bs);
    if (st != SP_OK) return st;
  }
  return SP_OK;
}

}  // namespace sp
