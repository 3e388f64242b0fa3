// Shared declarations of the libsp translation units (host-side launchers and small device helpers).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>
#include <utility>
#include <type_traits>

#include "../../include/sp.h"

namespace sp {

// Device status word layout: status_dev[0] = code, [1] = failing index, [2] = aux, [3] = reserved.
__device__ __forceinline__ void report_status(int32_t* status, int32_t code, int32_t index, int32_t aux) {
  if (status == nullptr) return;
  if (atomicCAS(status, 0, code) == 0) {
    status[1] = index;
    status[2] = aux;
  }
}

// ---- launch accounting and CUDA-event profiling (sp_profile.cu) ---------------------------------------------------
enum ProfKind : int {
  PK_GEMM_TC = 0, PK_GEMM_SIMT = 1, PK_SOLVE = 2, PK_FUSED_UPDATE = 3, PK_PREP_H = 4, PK_SCORES = 5, PK_TOPK = 6,
  PK_ELEMENTWISE = 7, PK_ALLOCATE = 8, PK_CHOL_DIAG = 9, PK_PANEL_APPLY = 10,
  PK_GEMM_TC_SHARED = 11,   // tensor-core GEMMs launched on a subset of the SM pairs, beside other work
  PK_CONDITIONAL = 12,      // tensor-core GEMMs queued under a SkipScope: whether they run is decided on the device, so
                            // neither their flops nor their time is attributed to the GEMM kinds
  PK_COUNT = 13
};
void count_launch(int n = 1);
// sp_set_reproducible: when on, every floating-point sum of the library is taken in an order fixed by the call's
// arguments (no product is cut along K, the triangular solves run on one stream), so equal inputs give equal bits.
bool reproducible_mode();
// sp_set_wait_budget: clock cycles a barrier wait of the tensor-core GEMM may take (0: the built-in default)
long long wait_budget_cycles();
// Device-side conditional work without a host round trip: while a SkipScope is alive on the calling host thread, the
// launchers that honour it (the kernels of the regularised solves, the tensor-core GEMM, the column gathers and
// scatters) pass its flag to their kernels, and every such kernel returns at once when the flag is non-zero at the
// time it starts.  The flag is written by an earlier kernel of the same stream order.  Scopes do not nest.
const int32_t* skip_flag();
struct SkipScope {
  explicit SkipScope(const int32_t* flag);
  ~SkipScope();
};
// Brackets the kernels launched during its lifetime with a CUDA event pair on `stream` when profiling is enabled.
// Scopes nest: only the outermost one records, so a phase scope absorbs the kernels launched inside it.
struct ProfScope {
  ProfScope(int kind, double flops, double bytes, cudaStream_t stream);
  ~ProfScope();
  int slot;
  cudaStream_t stream;
};

// One-time set-up per device (function attributes, device properties): run(fn) calls fn the first time it is reached
// with a given device current, under a lock, and remembers success per device; a process may drive several GPUs.
class PerDeviceOnce {
 public:
  template <typename F>
  cudaError_t run(F&& fn) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> guard(mu_);
    if (done_[dev]) return cudaSuccess;
    e = fn();
    if (e == cudaSuccess) done_[dev] = true;
    return e;
  }
  static constexpr int kMaxDevices = 64;

 private:
  std::mutex mu_;
  bool done_[kMaxDevices] = {};
};
// Multiprocessor count of the current device (cached per device).
int sm_count();

__host__ __device__ __forceinline__ int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }
__host__ __device__ __forceinline__ size_t align_up(size_t a, size_t b) { return (a + b - 1) / b * b; }

// Programmatic dependent launch.  Every kernel of the library starts with kernel_begin() (the GEMM after setting up its
// barriers and tensor memory): the next kernel of the stream may be brought onto the SMs from here on, and nothing of the
// kernels before is touched until they have completed.  Each kernel waits, so the completion of one implies that of all
// before it, as without the attribute; only launch latency, block start and the set-up ahead of the wait overlap.  Both
// instructions do nothing in a kernel that was launched plainly.
// A kernel's life begins while what it reads is still being written, by the library's or by the caller's kernels.  So no kernel
// has __restrict__ pointers: const and __restrict__ together allow loads on the read-only path, whose contract is that the data
// does not change during the kernel's whole life, and which the wait need not precede.  Loads through plain pointers stay
// behind the wait (it clobbers memory) and are coherent, but they stay behind the stores before them too: loads that are to be
// in flight together stand before the first store of a round (for_strip_move; split_planes 90 -> 140 us where they do not).
// The attribute is given inside an OverlapScope only, which the entry points open for calls whose kernels are short: their
// time is launches and gaps (attention step 768 wide, 284 kernels: 2.68 -> 2.42 ms; ADMM step 768 x 3072 2.27 -> 2.11).  Long
// kernels lose: waiting blocks hold SMs that another stream's kernels could use.
__device__ __forceinline__ void dependents_may_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_predecessors() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void kernel_begin() {
  dependents_may_launch();
  wait_for_predecessors();
}
bool& overlap_flag();                   // of this host thread (sp_profile.cu)
struct OverlapScope {
  bool saved;
  explicit OverlapScope(bool on) : saved(overlap_flag()) { overlap_flag() = on; }
  ~OverlapScope() { overlap_flag() = saved; }
  OverlapScope(const OverlapScope&) = delete;
};
// Weight phase of an ADMM step (and the cached input inverse): modules up to this width.  Attribute off / on, ms a step: 768 x 3072 on 2048
// tokens 1.320 / 1.265, on 32768 tokens 2.014 / 1.999, 1096 x 4376 on 9973 tokens 2.535 / 2.508, on 65536 tokens equal.  Wider
// modules keep plain launches: with recoveries by launches per block column 2048 x 8192 on 32768 tokens gained 1.7 % and 3072 x 9216 less
// than its runs differ; most recoveries are one launch now, and the line was not measured again.
constexpr int64_t kOverlapMaxN = 4608;
// Token pass of such a step: chunks of up to this many entries of Z.  Attribute off / on: 6.3 M entries 2.14 / 2.11 ms a step, 12.6 M
// 2.20 / 2.17, 25 and 33 M equal, 38 M 2.38 / 2.40, 50 M 2.48 / 2.52, 101 M in eight chunks 9.4 / 10.7.
constexpr int64_t kOverlapMaxChunk = int64_t(1) << 25;
// Recoveries by themselves (sp_ridge_solve, sp_linear_refit): matrices up to this width, of which a refit solves a part.  Attribute
// off / on, us: 128 unknowns, 128 right-hand sides 49 / 36, 256 / 256 92 / 77, 128 of 256 62 / 42, 384 of 768 132 / 119, 768 / 768 196 / 192,
// 1024 / 2048 254 / 248.  Wider ones keep plain launches; that is not a measured line: they ran with the attribute in the passes among
// which one stood still.
constexpr int64_t kOverlapMaxSolve = 1024;
inline bool may_overlap_launches(cudaStream_t stream) {
  if (!overlap_flag()) return false;
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(stream, &capture) == cudaSuccess) return capture == cudaStreamCaptureStatusNone;
  cudaGetLastError();
  return false;
}
template <typename... P, typename... A>
inline cudaError_t launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, A&&... args) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = &attr;
  // a grid of more than two waves of threads hides its own launch, and its successor's waiting blocks would only hold SMs
  // that other streams' kernels could use
  const int64_t threads = (int64_t)grid.x * grid.y * grid.z * block.x * block.y * block.z;
  cfg.numAttrs = threads <= (int64_t)sm_count() * 4096 && may_overlap_launches(stream) ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

// Shape of the kernels that move whole matrices: blocks of 256 threads, gridDim.x strips of columns (a thread has four of a
// strip's, blockDim.x apart, so that every access of a warp is one line), blockDim.y and gridDim.y walk the rows.  No
// index is divided, and what depends on the column alone is read once per block.  A block covers 256 columns of one row, and
// the kernels know that width at compile time (W = 256; 65536 rows of 768 columns lose 3 % without); a matrix of at most
// 128 columns puts as many rows into a block as fill its threads (W = 0: blockDim.x columns).  A solve for 262144 rows of 16
// columns, most of it gather, panel and scatter: 0.86 ms with one row per block, 0.57 with 16.
constexpr int kStripThreads = 256, kStripPer = 4;
// 256 threads, as many of them along a row as it has columns (a power of two)
inline dim3 strip_block(int64_t cols) {
  unsigned bx = 1;
  while (bx < (unsigned)kStripThreads && (int64_t)bx < cols) bx *= 2;
  return dim3(bx, kStripThreads / bx);
}
// launch(W, grid, block) with W as an integral constant
template <typename F>
inline void strip_launch(int64_t rows, int64_t cols, F&& launch) {
  const dim3 block = strip_block(cols);
  const int64_t gx = ceil_div(cols, (int64_t)block.x * kStripPer), row_blocks = ceil_div(rows, (int64_t)block.y);
  int64_t gy = ceil_div((int64_t)sm_count() * 8, gx);
  if (gy > row_blocks) gy = row_blocks;
  const dim3 grid((unsigned)(gx > 0 ? gx : 1), (unsigned)(gy > 0 ? (gy < 65535 ? gy : 65535) : 1));
  if (block.y == 1) launch(std::integral_constant<int, kStripThreads>{}, grid, block);
  else launch(std::integral_constant<int, 0>{}, grid, block);
}
inline unsigned lower_tiles(int64_t n, int64_t tile) {
  const int64_t nt = ceil_div(n, tile);
  return (unsigned)(nt * (nt + 1) / 2);
}
#ifdef __CUDACC__
// columns of a block, this thread's first column and row, and the distance of its rows
template <int W> __device__ __forceinline__ int strip_width() { return W > 0 ? W : (int)blockDim.x; }
template <int W> __device__ __forceinline__ int64_t strip_col() {
  return (int64_t)blockIdx.x * (strip_width<W>() * kStripPer) + threadIdx.x;
}
template <int W = 0> __device__ __forceinline__ int64_t strip_row() {
  return W > 0 ? (int64_t)blockIdx.y : (int64_t)blockIdx.y * blockDim.y + threadIdx.y;
}
template <int W = 0> __device__ __forceinline__ int64_t strip_rows() {
  return W > 0 ? (int64_t)gridDim.y : (int64_t)gridDim.y * blockDim.y;
}
// f(i, j, q) for this thread's rows i and columns j, q = 0 .. 3 their number
template <int W, typename F>
__device__ __forceinline__ void for_strip(int64_t rows, int64_t cols, F&& f) {
  const int64_t c0 = strip_col<W>();
#pragma unroll 2
  for (int64_t i = strip_row<W>(); i < rows; i += strip_rows<W>())
#pragma unroll
    for (int q = 0; q < kStripPer; ++q) {
      const int64_t j = c0 + q * strip_width<W>();
      if (j < cols) f(i, j, q);
    }
}
// store(i, j, q, load(i, j, q)) for this thread's rows and columns, the loads of two rows in flight before a store
template <int W, typename L, typename S>
__device__ __forceinline__ void for_strip_move(int64_t rows, int64_t cols, L&& load, S&& store) {
  const int64_t c0 = strip_col<W>(), step = strip_rows<W>();
  for (int64_t i = strip_row<W>(); i < rows; i += 2 * step) {
    decltype(load(i, c0, 0)) v[2][kStripPer] = {};
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int q = 0; q < kStripPer; ++q) {
        const int64_t r = i + h * step, j = c0 + q * strip_width<W>();
        if (r < rows && j < cols) v[h][q] = load(r, j, q);
      }
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int q = 0; q < kStripPer; ++q) {
        const int64_t r = i + h * step, j = c0 + q * strip_width<W>();
        if (r < rows && j < cols) store(r, j, q, v[h][q]);
      }
  }
}
// tile (row block y, column block x <= y) of a lower triangle of tiles counted row by row
__device__ __forceinline__ void lower_tile(unsigned t, unsigned& y, unsigned& x) {
  y = (unsigned)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
  while ((unsigned long long)(y + 1) * (y + 2) / 2 <= t) ++y;
  while ((unsigned long long)y * (y + 1) / 2 > t) --y;
  x = t - (unsigned)((unsigned long long)y * (y + 1) / 2);
}
// idx[j] (idx == nullptr: j) of this thread's columns
template <int W>
__device__ __forceinline__ void strip_index(const int32_t* idx, int64_t cols, int64_t (&at)[kStripPer]) {
  const int64_t c0 = strip_col<W>();
#pragma unroll
  for (int q = 0; q < kStripPer; ++q) {
    const int64_t j = c0 + q * strip_width<W>();
    at[q] = j < cols ? (idx ? (int64_t)idx[j] : j) : 0;
  }
}
#endif

inline size_t dtype_size(int32_t dt) { return dt == SP_BF16 ? 2 : (dt == SP_F64 ? 8 : 4); }

// A strided operand of the SIMT GEMM: element (i, k) lives at ptr[i * s0 + k * s1].
struct Operand {
  const void* ptr;
  int32_t dtype;
  int64_t s0, s1;
};

struct OutOperand {
  void* ptr;
  int32_t dtype;
  int64_t ld;
  // bf16 output of the tensor-core GEMM only: lo_off > 0 writes the result as two bf16 parts, bf16(v) at column j and
  // bf16(v - bf16(v)) at column lo_off + j of the same row, so that it can serve as a split operand of the next product
  int64_t lo_off = 0;
};

// C[M,N] (row-major) = alpha * sum_k A(i,k) B(k,j) + beta * Cin[i,j].  Cin may alias C or be another matrix of
// another dtype; beta == 0 never reads Cin.  lower_only skips tiles that lie strictly above the diagonal.
// acc64: accumulate in fp64 (else fp32).  k_tri: B(k, j) = 0 for k < j and (kTriBoth) A(i, k) = 0 for k < i, so that a tile may
// start its sum there (honoured where it pays; the stored zeros are read otherwise).
constexpr int kTriBoth = 1, kTriColumns = 2;
cudaError_t gemm_simt(int64_t M, int64_t N, int64_t K, double alpha, Operand A, Operand B, double beta,
                      Operand Cin, OutOperand C, bool lower_only, bool acc64, cudaStream_t stream, int k_tri = 0);

// tcgen05 path: bf16 operands, fp32 accumulation in tensor memory.
//   a_kmajor: A is stored [M, K] row-major (K contiguous) ; else [K, M] row-major (M contiguous).
//   b_kmajor: B is stored [N, K] row-major (K contiguous) ; else [K, N] row-major (N contiguous).
// Returns SP_ERR_UNSUPPORTED when alignment rules of the tensor maps are not met (the caller may then use gemm_simt).
struct TcOperand {
  const void* ptr;  // bf16
  int64_t ld;       // elements between consecutive rows of the stored matrix
  bool kmajor;
  int64_t kext = 0;   // extent of the stored matrix along K (0: the K of the call); reads beyond it return zero
  int64_t mnext = 0;  // extent along M (for A) or N (for B) (0: the M / N of the call)
};
// K segments: the contraction runs over nseg segments of K indices each; segment s reads A at K offset a_k[s] and
// M offset a_mn[s], B at K offset b_k[s] and N offset b_mn[s] (elements).  This is how split operands (an fp32 value
// held as a sum of bf16 parts stored side by side) are multiplied: one segment per kept product of parts.
constexpr int kTcMaxSegments = 6;
struct TcSegments {
  int32_t nseg = 1;
  int32_t a_k[kTcMaxSegments] = {0, 0, 0, 0, 0, 0}, a_mn[kTcMaxSegments] = {0, 0, 0, 0, 0, 0};
  int32_t b_k[kTcMaxSegments] = {0, 0, 0, 0, 0, 0}, b_mn[kTcMaxSegments] = {0, 0, 0, 0, 0, 0};
  // batched launches only: the plane of A / B the segment reads (see TcBatch)
  int32_t a_p[kTcMaxSegments] = {0, 0, 0, 0, 0, 0}, b_p[kTcMaxSegments] = {0, 0, 0, 0, 0, 0};
};
// Batched form: nb0 * nb1 independent products C_b = alpha A_b B_b (+ beta Cin_b) of the same shape in ONE launch.
// Operand X of product (b0, b1) starts at ptr + b0 * x_s0 + b1 * x_s1 (elements); this is how the per-head,
// per-sequence products of an attention module (head = a column slice of a token-major tensor, sequence = a row range)
// are issued together.  A and B may also consist of several planes (e.g. the hi and lo parts of a split operand, each
// a whole tensor, x_plane elements apart); a K segment then names the plane it reads.  Every stride times the element
// size must be a multiple of 16 bytes.  Not available together with a cut along K.
struct TcBatch {
  int32_t nb0 = 1, nb1 = 1;
  int64_t a_s0 = 0, a_s1 = 0, b_s0 = 0, b_s1 = 0, c_s0 = 0, c_s1 = 0, cin_s0 = 0, cin_s1 = 0;
  int32_t a_planes = 1, b_planes = 1;
  int64_t a_plane = 0, b_plane = 0;
  bool b_shared0 = false;       // B is the same for all nb0 products (b_s0 unused)
  // one segment: A(i, k) is zero for k in later (kTriALower) or earlier (kTriAUpper) blocks of kTcTileRows than i's, and not read there
  int32_t k_tri = 0;
};
constexpr int32_t kTriALower = 1, kTriAUpper = 2;
constexpr int64_t kTcTileRows = 256;
// K is the extent of ONE segment.  alg_flops >= 0 overrides the flop count recorded for profiling.  max_pairs > 0
// limits the launch to that many CTA pairs (SM pairs), leaving the other SMs to kernels of another stream.
sp_status gemm_tc(int64_t M, int64_t N, int64_t K, float alpha, TcOperand A, TcOperand B, float beta, Operand Cin,
                  OutOperand C, bool lower_only, int32_t* status_dev, cudaStream_t stream,
                  const TcSegments* segs = nullptr, double alg_flops = -1.0, int max_pairs = 0,
                  const TcBatch* batch = nullptr);
bool gemm_tc_supported(int64_t M, int64_t N, int64_t K, TcOperand A, TcOperand B);

struct SolveAssist;
// fp64 factorisation and solves (sp_linalg.cu), block columns of kCholNB.
constexpr int kCholNB = 64;
//   potrf_lower_f64: in-place lower Cholesky of the n x n matrix A (ld lda); the strict upper triangle and the diagonal
//   blocks of the factor are not written; dinv: ceil(n / kCholNB) inverse diagonal blocks [kCholNB, kCholNB].
//   m_extra > 0: A has m_extra more rows below row n, right-hand sides B of X L^T = B that ride along and hold X on
//   return.  identity: n more rows below those hold an identity, whose X = L^-T is upper triangular; a step touches only its
//   rows that are no longer zero.
cudaError_t potrf_lower_f64(double* A, int64_t n, int64_t lda, double* dinv, int32_t* status_dev, cudaStream_t stream,
                            const SolveAssist* assist, int64_t m_extra, bool identity = false);
// W[m, n] = B L^-T L^-1 with the factor of the n x n matrix A, the right-hand sides B below it and, below those, room for n more
// rows (all dense, leading dimension n).
cudaError_t solve_inverse_f64(double* A, int64_t n, int64_t m, double* dinv, double* W, int32_t* status_dev, cudaStream_t stream,
                              const SolveAssist* assist);
// Which systems (n unknowns, m right-hand sides) are solved that way: more than one diagonal block (one has no chain: 64 / 256 33 us by the
// sweep, 45 with the identity; 65 / 65 72 -> 60), up to 4096 unknowns (the identity costs n^3 / 3 operations, which pay while the chain
// leaves the fp64 pipe idle).  Inside a step it runs beside the chain (assisted; fp32 mode, a step of 128 x 512 0.64 -> 0.56 ms, 768 x 3072
// 5.8 -> 4.9, 1024 x 4096 10.0 -> 9.0).  On one stream its rows are the chain's own: for wide systems only with right-hand sides enough
// that the sweep would cost more.  Sweep / identity, us: 1024 / 256 536 / 482, 2560 / 16 1780 / 1712, 3072 / 16 2264 / 2326, 3072 / 768 3024 /
// 2830, 3584 / 448 3406 / 3503, 3584 / 896 4011 / 3849, 4096 / 1024 5136 / 5290, 4096 / 2048 6742 / 6440, 4096 / 16384 29889 / 22979.
constexpr int64_t kInverseMaxN = 4096, kInverseAloneN = 3072;
inline bool inverse_f64(int64_t n, int64_t m, bool assisted) {
  return n > kCholNB && n <= kInverseMaxN && (assisted || 2 * m >= 3 * (n - kInverseAloneN));
}
// fp64 elements of a solve's system, right-hand sides, identity and result, for up to n unknowns and m right-hand sides
inline size_t solve_f64_elems(int64_t n, int64_t m, bool assisted) {
  const int64_t most = assisted ? kInverseMaxN : kInverseAloneN + 2 * m / 3;
  const int64_t inv = n < most ? n : most < kInverseMaxN ? most : kInverseMaxN;
  const size_t sweep = (size_t)(n + m) * n, inverse = inv > kCholNB ? 2 * (size_t)(inv + m) * inv : 0;
  return sweep > inverse ? sweep : inverse;
}
// X[m,n] <- X L^-1 (backward sweep with the factor of potrf_lower_f64).
cudaError_t potrs_backward_f64(double* X, int64_t m, int64_t n, int64_t ldx, const double* L, int64_t ldl,
                               const double* dinv, cudaStream_t stream, const SolveAssist* assist);

// fp32 factorisation / solves with tensor-core trailing updates (sp_linalg_tc.cu).  Panels are kCholTcNB wide.
//   dinv: ceil(n / kCholTcNB) blocks of 2 * kCholTcNB^2 floats (inverse diagonal blocks and their transposes)
//   P   : bf16 [chol_tc_pad(n), 3 * chol_tc_pad(n)] — the factor below its diagonal blocks as three bf16 parts
//   Xs  : chol_tc_xs_elems(n, m) bf16 — the current block columns of the right-hand sides as three bf16 parts
constexpr int kCholTcNB = 128;
// Two-level blocking of the factorisation and of the backward sweep: systems of at least kOuterMinN unknowns, outer blocks
// of kOuterBlocks diagonal blocks.
constexpr int64_t kOuterMinN = 12288;
constexpr int64_t kOuterBlocks = 4;
int64_t chol_tc_pad(int64_t n);
// two buffers of one block column, or one of an outer block
inline int64_t chol_tc_xs_elems(int64_t n, int64_t m) {
  return m * 3 * kCholTcNB * (n >= kOuterMinN ? kOuterBlocks : 2);
}
// Optional second stream (with three events) that carries the part of each step that the next step's first kernel
// does not wait for: the far part of a solve step's update; the panel and trailing update of a factorisation step.
struct SolveAssist {
  cudaStream_t stream;
  cudaEvent_t panel_done, rest_done[2];
  cudaEvent_t near_done;   // factorisation: the first two block columns of a step's trailing update have landed
  // Optional third stream of a factorisation: the far part of a step's trailing update (everything right of the first
  // two block columns), so that the next step's panel and near update do not queue behind it.
  cudaStream_t far_stream = nullptr;
  cudaEvent_t far_go = nullptr, far_done[2] = {nullptr, nullptr};
};
// dinv must have room for ceil(n / 128) + 1 pairs of 128 x 128 blocks (the last pair is scratch).
// m_extra > 0: A has m_extra more rows below row n (same lda), the right-hand sides B of a system X L^T = B; they
// are carried through the panels and trailing updates and hold X on return (P then needs n + m_extra rows).
sp_status potrf_lower_tc(float* A, int64_t n, int64_t lda, float* dinv, void* P, int32_t* status_dev,
                         cudaStream_t stream, const SolveAssist* assist = nullptr, int64_t m_extra = 0,
                         bool split_lookahead = false);   // lookahead kernel as two launches without a cluster
// forward_done: X already holds the solution of the forward system (it rode along with the factorisation).
// Lf / ldl (optional): the fp32 factor potrf_lower_tc left in A; with it the backward sweep updates a block column by
// the one before it inside the panel kernel instead of by a GEMM of its own.
sp_status potrs_right_tc(float* X, int64_t m, int64_t n, int64_t ldx, const void* P, const float* dinv, void* Xs,
                         int32_t* status_dev, cudaStream_t stream, const SolveAssist* assist = nullptr,
                         bool forward_done = false, const float* Lf = nullptr, int64_t ldl = 0,
                         int64_t n_factor = 0);
// n_factor > n: the factor in P / dinv / Lf is that of a larger system of n_factor rows and the solve uses its leading
// n x n block, which is the factor of the system's leading block (n a multiple of kCholTcNB).

// The whole solve W = R G^-1 in one launch (sp_solve_tc.cu), systems that solve_in_one() names.
//   A: [nn + m, nn] fp32, lower triangle of G and the right-hand sides below it; W [m, nn] may be the latter's place.
//   lead != nullptr: also the solution [m, lead_k] of the leading lead_k x lead_k system with the leading right-hand sides.
//   P: bf16 [pad(nn) + pad(m), 3 pad(nn)], Y: bf16 [pad(m), 3 kCholTcNB], flags: solve_tc_flag_words(nn, m) words; pad = chol_tc_pad.
//   batch > 1: that many systems, A and W a_bs elements apart, the other arrays one system's behind the other's (no lead).
struct SolveOneBufs {
  void *P, *Y;
  float* pre;         // 2 ceil(nn / kCholTcNB) blocks of kCholTcNB^2, and behind those of all systems ceil(nn / kCholTcNB) times kCholTcNB
  uint32_t* flags;
};
// Launches per block column (sp_linalg_tc.cu) against one launch, unknowns / right-hand sides, us: 128 / 128 41 -> 59, 256 / 256 78 -> 86,
// 257 / 100 154 -> 104, 384 / 768 129 -> 116, 768 / 768 265 -> 194, 1024 / 2048 374 -> 250, 2048 / 4096 1036 -> 587, 3072 / 768 1183 -> 728,
// 4096 / 3302 2312 -> 1270, 5734 / 7168 13410 -> 3920, 8192 / 2048 6055 -> 3990, 9216 / 3072 8970 -> 6230; with two levels of blocks
// 12288 / 4096 14740 -> 14510.
constexpr int64_t kSolveOneMinN = 256, kSolveOneMaxN = kOuterMinN - 1;
// A step's recoveries: modules up to this width.  Not for speed and not for accuracy: the sign select of the z-update turns differences of
// rounding into differences of the recovered weights, and beyond it a step by this form differs from one by the other form's roundings by
// about a percent of W1, the size of its distance from 64 bits, which is the same for both.  n x n / 4 on 8192 tokens, 20 % kept, five
// iterations: W1 moves by 0.83 / 0.88 / 0.96 / 1.03 % for n = 18432 / 20480 / 24576 / 28672 (16384 on 4096 tokens: 0.8), is
// 1.25 / 1.30 / 1.39 / 1.45 % from 64 bits either way (W2: 0.48 .. 0.58 and 0.95 .. 1.03 %), and a step takes 46.2 / 59.2 / 97.6 / 149.0 against 43.4 / 57.1 / 95.4 / 143.1 ms.
constexpr int64_t kSolveOneModule = 16384;
inline bool solve_in_one(int64_t n) { return n > kSolveOneMinN && n <= kSolveOneMaxN; }
size_t solve_tc_flag_words(int64_t n, int64_t m);
sp_status solve_tc(const float* A, int64_t nn, int64_t m, int64_t lda, float* W, int64_t ldw, const SolveOneBufs& b,
                   float* lead, int64_t ld_lead, int64_t lead_k, int32_t* status_dev, cudaStream_t stream, int batch = 1,
                   int64_t a_bs = 0);

// `batch` independent systems of one size n (a multiple of kCholTcNB) with m right-hand sides each, every step one launch
// over all of them.  System b: A + b * a_bs = [n + m, n] fp32 (lower triangle of the matrix, then the right-hand sides
// B of X (L L^T) = B; on return they hold X), dinv + b * d_bs (room as for potrf_lower_tc), P = batch x
// [n + m, 3 n] bf16, Xs = batch x 2 x [m, 3 * kCholTcNB] bf16.
sp_status potrf_potrs_tc_batched(float* A, int64_t n, int64_t m, int batch, int64_t a_bs, float* dinv, int64_t d_bs,
                                 void* P, void* Xs, int32_t* status_dev, cudaStream_t stream);

// ---- elementwise / reduction launchers (sp_elementwise.cu) ------------------------------------------------------
cudaError_t convert_matrix(const void* src, int32_t sdt, int64_t lds, void* dst, int32_t ddt, int64_t ldd,
                           int64_t rows, int64_t cols, cudaStream_t stream);
cudaError_t symmetrize_lower(float* G, int64_t n, int64_t ld, cudaStream_t stream);
// dst[i, 0:cols] = bf16(src[i,:]) and dst[i, kpad:kpad+cols] = bf16(src - hi); padding columns are zero.
// dst is [rows, 2*kpad] bf16.
// row_idx != nullptr: row i of dst comes from row row_idx[i] of src.
cudaError_t split_bf16(const float* src, int64_t lds, const int32_t* row_idx, int64_t rows, int64_t cols, int64_t kpad,
                       void* dst, cudaStream_t stream);
// dst [rows, 3 * kpad] bf16: the hi, mid and lo parts of src side by side (an fp32 value as an exact sum of three bf16)
// row_idx as above
cudaError_t split3_bf16(const float* src, int64_t lds, const int32_t* row_idx, int64_t rows, int64_t cols, int64_t kpad,
                        void* dst, cudaStream_t stream);
// dst[j, i] = (TD) src[i, j]
template <typename TD>
cudaError_t transpose_convert(const float* src, int64_t lds, int64_t rows, int64_t cols, TD* dst, int64_t ldd,
                              cudaStream_t stream);
int column_stats_row_blocks(int64_t T, int64_t C);
int score_row_blocks(int64_t rows, int64_t cols);
size_t wanda_scratch_doubles(int64_t rows, int64_t cols);
// weight statistics of the "-distribute" importances (sp_mask.cu); scratch: (148 * 8 + n_blocks) * 3 doubles
int weight_stats_parts(int64_t n_blocks, int64_t block_rows);
cudaError_t weight_stats(const void* W, int32_t dt, int64_t ld, int64_t rows, int64_t cols, int axis, int64_t group,
                         bool accumulate, double* stats, double* scratch, cudaStream_t stream);
cudaError_t distribute_importance(const double* head_stats, int n_heads, const double* fc_stats, int n_fc, int L,
                                  double rho, double gamma, double* I_attn, double* I_mlp, cudaStream_t stream);
// dst[i,j] = (T) G[i*ld + j] (+ rho on the diagonal) for the lower triangle; rho read from device (rho_dev[0]).
template <typename T>
cudaError_t load_spd(const float* G, int64_t ldg, int64_t n, const double* rho_dev, T* dst, int64_t ldd,
                     cudaStream_t stream);
// gathered version: dst[a,b] = G[idx[a], idx[b]] (+rho on diagonal), count read from host k.
template <typename T>
cudaError_t load_spd_gather(const float* G, int64_t ldg, const int32_t* idx, int64_t k, const double* rho_dev, T* dst,
                            int64_t ldd, cudaStream_t stream);
// dst [rows, kpad] (dense) = the first k columns of src followed by zero columns
cudaError_t copy_cols_padded(const float* src, int64_t lds, int64_t rows, int64_t k, int64_t kpad, float* dst,
                             cudaStream_t stream);
// dst[i, a] = (T) src[i, idx[a]]  (idx == nullptr: identity)
template <typename T>
cudaError_t gather_cols(const float* src, int64_t lds, const int32_t* idx, int64_t rows, int64_t k, T* dst,
                        int64_t ldd, cudaStream_t stream);
// dst[i, :] = src[idx[i], :]
cudaError_t gather_rows(const float* src, int64_t lds, const int32_t* idx, int64_t rows, int64_t cols, float* dst,
                        int64_t ldd, cudaStream_t stream);
// dst (fp32, [rows, n]) = 0 ; dst[i, idx[a]] = src[i, a]
template <typename T>
cudaError_t scatter_cols(const T* src, int64_t lds, const int32_t* idx, int64_t rows, int64_t k, int64_t n,
                         float* dst, int64_t ldd, cudaStream_t stream);
// rho_out[0] = rho * trace(G)/n (relative) or rho
cudaError_t effective_ridge(const float* G, int64_t ldg, int64_t n, double rho, int rel, double* rho_out,
                            cudaStream_t stream);

struct UpdateArgs {
  float* Z;          // [T, n] in/out
  float* U;          // [T, n] in/out or null
  const float* z1;   // [T, ldk] compact on the kept channels
  const float* D;    // [T, ldk] compact: correction term of the a-update
  const float* gate; // [T, n] gate factor of a gated module (phi(z) = gate * z), or null: phi = ReLU
  int64_t ldk, k;    // leading dimension of the compact tensors, number of kept channels
  const int32_t* grp_base;   // per group of 8 channels: kept channels before the group
  const uint8_t* grp_mask;   // per group of 8 channels: bit q = channel 8 g + q is kept
  void* A_out;       // [T, n] storage dtype
  void* At_out = nullptr;  // bf16 [n, ldt]: A transposed (then A_out is not written)
  int64_t ldt = 0;
  void* Zb_out;      // [T, n] storage dtype copy of Z_new
  int32_t out_dtype;
  int64_t T, n;
  float alpha, beta;
  int32_t z_rule;
  double* partial;   // [blocks * 4] block partial sums: res_act, z_sq, a_sq, |z_new - z1|^2
  double* absA_part; // [row_blocks, n] partial column sums of |A|
  int32_t row_blocks;
  // At_out with its rows in "kept channels first" order: kept channel c goes to row (number of kept channels before
  // c), pruned channel c to row k + (number of pruned channels before c).
  int32_t at_kept_first = 0;
  // Both set (bf16 storage, ReLU, no dual variable, n % 4 == 0, At_out with at_kept_first; grid from
  // fused_update_next_grid): the update also writes what the next step reads, rows in the order of At_out, pitch ldt:
  // Zt_out [n, ldt] = bf16(Z_new)^T (the pruned channels' rows only when *zt_pruned_flag != 0 or the flag is null) and
  // Ht_out [k, ldt] = bf16(max(Z_new, 0))^T on the kept channels.  Zb_out is then not written.
  void* Zt_out = nullptr;
  void* Ht_out = nullptr;
  const int32_t* zt_pruned_flag = nullptr;
};
// grp_base / grp_mask of a u8 mask over n channels, the first k that it keeps (see sp_elementwise.cu)
cudaError_t build_group_map(const uint8_t* mask, int64_t n, int64_t k, int32_t* grp_base, uint8_t* grp_mask, cudaStream_t stream);
// H[T, ldh] (compact on the k kept channels idx[0..k), ldh a multiple of 8) = storage(phi(Z) - U);
// phi(z) = gate * z when gate != nullptr, else ReLU.
// lo_off > 0 (bf16 storage, a multiple of 8, 2 * lo_off <= ldh): H is split into bf16 hi and lo parts, the hi part in
// columns [0, lo_off), the lo part in columns [lo_off, 2 * lo_off); columns k..lo_off-1 of both are zero.
cudaError_t launch_prep_h(const float* Z, const float* U, const float* gate, void* H, int32_t hdt, int64_t T,
                          int64_t n, int64_t ldh, int64_t k, const int32_t* idx, cudaStream_t stream,
                          int64_t lo_off = 0);
cudaError_t launch_fused_update(const UpdateArgs& a, cudaStream_t stream);
// Ht [k, ldt] bf16 = max(Z, 0)^T on the kept channels, rows in compact order (n % 4 == 0; ReLU, no dual variable): h of
// a step in the transposed layout in which the fused update leaves it for the next one.  Honours SkipScope.
cudaError_t launch_gather_ht(const float* Z, int64_t T, int64_t n, int64_t k, const int32_t* grp_base,
                             const uint8_t* grp_mask, void* Ht, int64_t ldt, cudaStream_t stream);
int fused_update_next_grid(int64_t T, int64_t n, int* row_blocks);
int fused_update_next_partial_rows(int row_blocks);   // rows of absA_part that this form of the update writes
int fused_update_next_row_cap(int64_t n);              // upper bound of the row blocks fused_update_next_grid returns
int64_t fused_update_next_max_blocks(int64_t n);       // ... and of its blocks
int fused_update_grid(int64_t T, int64_t n, int* row_blocks);
// out[j] (+)= sum_r part[r, j]
cudaError_t reduce_col_partials(const double* part, int32_t row_blocks, int64_t n, double* out, bool accumulate,
                                cudaStream_t stream);
// rep[field] (+)= sum of partial triples
cudaError_t reduce_report(const double* partial, int nblocks, sp_step_report* rep, bool accumulate, double alpha,
                          cudaStream_t stream);
// out[0] (+)= scale * sum of squares of a fp32 matrix; scratch: kSumsqBlocks doubles
constexpr int kSumsqBlocks = 592;
cudaError_t sumsq_accumulate(const float* x, int64_t ld, int64_t rows, int64_t cols, double scale, double* out,
                             bool accumulate, double* scratch, cudaStream_t stream);
// reused (device, may be null): non-zero when the recovery on the kept support reused the unrestricted factor
// scaled (device, may be null): non-zero when the pruned parts of G_A and R2 were obtained by scaling
cudaError_t init_report(sp_step_report* rep, const double* rho1, const double* rho2, double kept,
                        const int32_t* reused, const int32_t* scaled, cudaStream_t stream);
// relu + storage conversion for the init pass: A = phi(Z) -> storage dtype, and |A| column partials
// gate_io (gated modules): holds the gate pre-activation on entry and SiLU of it on return; A = gate * Z then
cudaError_t launch_init_act(const float* Z, float* gate_io, void* A_out, void* Zb_out, int32_t out_dtype, int64_t T,
                            int64_t n, double* absA_part, int32_t row_blocks, cudaStream_t stream);
cudaError_t column_stats(const void* X, int32_t dt, int64_t ld, int64_t T, int64_t C, double* rowstats,
                         double* scratch, cudaStream_t stream);

// ---- multi-head-attention auxiliary updates (sp_mha.cu); [pairs, T, T] tensors, pair = sequence * heads + head --------
// S <- softmax over each row (in place); causal: key u > query t gets 0; Sb: optional bf16 copy (plane > 0: hi and,
// `plane` elements further, lo parts)
cudaError_t mha_softmax_rows(float* S, int64_t pairs, int T, bool causal, void* Sb, int64_t plane, cudaStream_t stream);
// P <- P - eta_pair (-2 alpha G1 + 2 beta (P - Phi)); Pb: optional bf16 copy of the new P (hi / lo planes as above)
cudaError_t mha_p_update(float* P, const float* Phi, const float* G1, const float* eta, int64_t pairs, int T,
                         double alpha, double beta, void* Pb, int64_t plane, cudaStream_t stream);
// dS = 2 beta Phi (E - rowsum(E Phi)), Phi = softmax(S), E = Phi - P, as bf16 to dSb or (dSb == nullptr) in place of S;
// causal: zero for keys u > query t, written up to the end of the query's block of `tail` keys
cudaError_t mha_softmax_backward_rows(float* S, const float* P, int64_t pairs, int T, bool causal, int tail, double beta,
                                      void* dSb, cudaStream_t stream);
// per-pair step sizes from the squared norms of the [T, d_h] slices of x (and y): mode 0: 1 / (2 (alpha s + beta)),
// mode 1: eta_z / (2 alpha + beta s / d_h); sums: n_seq * H doubles of scratch
cudaError_t mha_step_sizes(const float* x, const float* y, int64_t ld, int64_t n_seq, int T, int d_h, int H, int mode,
                           double alpha, double beta, double eta_z, double* sums, float* eta, cudaStream_t stream);
// Z <- Z - eta_pair (G + 2 alpha (Z - T)) for Zq and Zk ([tokens, d] dense); Zqs / Zks: optional bf16 hi / lo planes
cudaError_t mha_z_update(float* Zq, float* Zk, const float* Gq, const float* Gk, const float* Tq, const float* Tk,
                         const float* eta, int64_t tokens, int d, int T, int d_h, double alpha, void* Zqs, void* Zks,
                         int64_t plane, cudaStream_t stream);
// Selected heads of a chunk, for the recovery of W_V: dst[plane][seq][slot][per_pair] = bf16 hi / lo parts of
// P[seq][heads.h[slot]][per_pair] (per_pair a multiple of 4)
constexpr int kMaxHeadGroup = 256;
struct HeadList {
  int32_t n = 0;
  uint16_t h[kMaxHeadGroup];
};
cudaError_t mha_split_heads(const float* P, int64_t n_seq, int64_t H, int64_t per_pair, const HeadList& heads, void* dst,
                            int64_t plane, cudaStream_t stream);
// dst[(slot * tokens + t) * ld + c] = bf16 hi part of A[t, heads.h[slot] * d_h + c], lo part lo_off columns to the right
cudaError_t mha_split_head_cols(const float* A, int64_t tokens, int64_t d, int64_t d_h, const HeadList& heads, void* dst,
                                int64_t ld, int64_t lo_off, cudaStream_t stream);
// per system b: G_b[i, i] += rel ? rho tr(G_b) / n : rho (G_b [n, n], dense rows, bs elements apart)
cudaError_t add_ridge_batched(float* G, int64_t bs, int64_t n, int batch, double rho, bool rel, cudaStream_t stream);
// W[(heads.h[slot] * d_h + r) * ldw + c] = src[slot * bs + r * d + c]
cudaError_t mha_place_heads(const float* src, int64_t bs, int64_t d_h, int64_t d, const HeadList& heads, float* W,
                            int64_t ldw, cudaStream_t stream);
// A[n, n] (ld) = identity
template <typename T>
cudaError_t set_identity(T* A, int64_t n, int64_t ld, cudaStream_t stream);
// dst[e] = bf16(x[e]), dst[plane + e] = bf16(x[e] - hi) (plane == 0: hi only)
cudaError_t split_planes(const float* x, int64_t total, void* dst, int64_t plane, cudaStream_t stream);

// ---- scores / allocation / selection (sp_mask.cu) -----------------------------------------------------------------
cudaError_t wanda_scores(int kind, int group, const float* W, int64_t rows, int64_t ldw, const float* colsq,
                         int64_t colsq_stride, const double* colabs, double inv_tokens, int64_t n_units,
                         float* scores, double* importance, double* scratch, cudaStream_t stream);
cudaError_t lemma1_scores_stream(const sp_mat& b, const sp_mat& c, const sp_mat& dd, const sp_mat& t, int group,
                                 int64_t n_units, float* scores, double* importance, double* relaxed, double r_layer,
                                 double* scratch, cudaStream_t stream);
// s_j = (cb_j + cc_j) / (2 cc_j) with cb_j = <T0[j,:], W1t[j,:]>, cc_j = <T0[j,:], W10[j,:]>, T0 = W10 G_X
cudaError_t lemma1_scores_gram(const float* T0, const float* W1t, const float* W10, int64_t n, int64_t d,
                               float* scores, double* importance, double* scratch, cudaStream_t stream);
cudaError_t allocate_sparsity(const double* I, const int64_t* n_units, int L, double rbar, double T, int mode,
                              double clip_hi, double* r_out, int64_t* k_out, cudaStream_t stream);
cudaError_t topk_select(const float* scores, int64_t n, int64_t k, uint8_t* mask, float* tau, int32_t* kept_idx,
                        cudaStream_t stream);
// kept_idx from an existing mask (ascending), count must equal k
// `batch` independent problems in one launch (one block each); k_list (device, may be nullptr) overrides k_all.
cudaError_t topk_select_batched(const float* scores, int64_t ld_scores, int64_t n, int64_t batch, int64_t k_all,
                                const int64_t* k_list, uint8_t* mask, int64_t ld_mask, float* tau, int32_t* kept_idx,
                                int64_t ld_idx, cudaStream_t stream, bool skip_negative = false);
// allocation for a grid of n_T temperatures in one launch: T_list (device), relative to mean |I| when T_relative;
// r_out / k_out are [n_T, L]
cudaError_t allocate_sparsity_grid(const double* I, const int64_t* n_units, int L, double rbar, const double* T_list,
                                   int n_T, bool T_relative, int mode, double clip_hi, double* r_out, int64_t* k_out,
                                   cudaStream_t stream);
// one threshold over the L x n scores (rows ld_scores apart): the K largest kept (ties: earlier layer, lower index),
// a layer left with fewer than min_keep units keeps its own min_keep best; counts_out[l] = kept units of layer l
size_t global_select_scratch_bytes(int64_t total, int L);
cudaError_t global_select(const float* scores, int64_t ld_scores, int64_t n, int L, int64_t K, int64_t min_keep,
                          uint8_t* mask, int64_t ld_mask, float* tau, int64_t* counts_out, void* scratch,
                          cudaStream_t stream);
cudaError_t mask_to_index(const uint8_t* mask, int64_t n, int32_t* kept_idx, cudaStream_t stream);
// reports SP_ERR_SHAPE (index = the number of kept units found) through the device status word when `mask` does not
// keep exactly k units; no-op without a status word
cudaError_t mask_count_check(const uint8_t* mask, int64_t n, int64_t k, int32_t* status, cudaStream_t stream);
// C[i, j] *= f^power for the rows x cols block at C (ld); f is read from the device (a float stored in an int32 slot)
cudaError_t scale_block(float* C, int64_t ld, int64_t rows, int64_t cols, const int32_t* f_bits, int power,
                        cudaStream_t stream);
// G[perm[i], perm[j]] = G[perm[j], perm[i]] = Gp[i, j] for i >= j (Gp: lower triangle in permuted order)
cudaError_t unpermute_gram(const float* Gp, const int32_t* perm, int64_t n, float* G, int32_t* inv,
                           cudaStream_t stream);
// R[r, perm[j]] = Rp[r, j]
cudaError_t unpermute_cols(const float* Rp, const int32_t* perm, int64_t rows, int64_t n, float* R,
                           cudaStream_t stream);
// tag[1] = k when `valid`, else -1; tag[2] = bits of the float c; tag[4], tag[5] = size of the h buffer per token and
// token chunk with which h was written for the next step (0: none was written; its layout depends on both)
cudaError_t decay_tag_set(int32_t* tag, int64_t k, float c, bool valid, int64_t h_ld, int64_t h_chunk,
                          cudaStream_t stream);
// ready[0] = 1 when same[0] != 0 and the tag says that h was written for h_ld and h_chunk, else 0; ready[1] = 1 - ready[0]
cudaError_t h_next_ready(const int32_t* same, const int32_t* tag, int64_t h_ld, int64_t h_chunk, int32_t* ready,
                         cudaStream_t stream);
// R[perm[i], :] = Rp[i, :]
cudaError_t unpermute_rows(const float* Rp, const int32_t* perm, int64_t n, int64_t cols, float* R,
                           cudaStream_t stream);
// perm[0..n) = the kept channels of `mask` in ascending order followed by the pruned ones; count[0] = kept channels
cudaError_t mask_to_perm(const uint8_t* mask, int64_t n, int32_t* perm, int32_t* count, cudaStream_t stream);
// flags[0] = 1 when the kept channels of `mask` are not exactly perm[0..k) with count_old[0] == k; flags[1] = 1 - flags[0]
cudaError_t mask_changed(const uint8_t* mask, const int32_t* perm, const int32_t* count_old, int64_t k, int32_t* flags,
                         cudaStream_t stream);
cudaError_t zero_pruned(const uint8_t* mask, int group, float* W_rows, int64_t r_rows, int64_t r_cols, int64_t r_ld,
                        float* W_cols, int64_t c_rows, int64_t c_cols, int64_t c_ld, cudaStream_t stream);
// dst[idx[p], :] = src[p, :] for the k >= 1 listed rows (ascending), zero rows where the mask is zero; rows that it keeps beyond the list:
// R[i, :] M (R [rows, cols], M [cols, cols])
cudaError_t place_rows(const uint8_t* mask, const int32_t* idx, int64_t k, const float* src, int64_t lds, const float* R, const float* M,
                       float* dst, int64_t ldd, int64_t rows, int64_t cols, cudaStream_t stream);
// dst[i,:] = mask[i] ? src[i,:] : 0
cudaError_t mask_rows_copy(const uint8_t* mask, const float* src, int64_t lds, float* dst, int64_t ldd, int64_t rows,
                           int64_t cols, cudaStream_t stream);

}  // namespace sp
