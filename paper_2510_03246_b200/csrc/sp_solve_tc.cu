// A regularised solve W = R G^-1 in ONE launch: fp32 Cholesky factorisation of G, forward substitution of the right-hand sides
// R, the inverse of the factor, and the product of both, as a graph of 128 x 128 tiles on the tensor cores.
//
// Tiles (row block r, column block j), all held as three bf16 parts (see sp_linalg_tc.cu) in one array P of np + m rows:
//   r > j  : L(r, j) of the factor;
//   r <= j : X(r, j) of X = inv(L)^T, whose rows are those of an identity carried along (X L^T = I);
//   r >= nblk: the forward-substituted right-hand sides Y.
// A tile is one task of one thread block.  It takes its entry of [G; I; R] less sum_k tile(r, k) L(j, k)^T over the k that exist to
// its left (left-looking: the running value stays in registers, nothing is read back and rewritten), and
//   the chain: factorises the blocks on the diagonal and inverts the factor (DiagTiles): X(j, j), then the tile below it and its
//             part of the next diagonal block's sum, all in one thread block (their sums over k < j come from other blocks, PRE);
//   T(r, j) : multiplies by X(j, j) = inv(L_jj)^T;
//   W(r, j) : sum_k Y(r, k) X(j, k)^T over k >= j, the result (last, when all columns are there).
// So there is no backward sweep, a serial chain of its own, and what follows a diagonal block waits for flags of its own tiles, not for
// launches.
//
// What bounds it: up to about 6000 unknowns the chain, 28 us per 128 unknowns (elimination 16, X and the tile below it into operand
// form 2, their product 2.2, its result into operand form 1, the diagonal block's update 2.2; as one task per diagonal block, handed on
// through memory, 36); above, the loads of the products (192 KB per two tiles' product; 3.8 us at 8192 unknowns, where the tensor core
// takes 1.6.  Four slots of half the depth, with rows of 64 bytes, are slower: 3.96 -> 4.44 ms).  3072 unknowns and 768 right-hand
// sides: 1183 us as launches per block column, 1015 with a task per diagonal block, 728.
//
// Tasks are taken by a counter in an order in which every task comes after those it reads (the chain, first, runs beside them).  A block
// that waits therefore waits for a task that a running block has: two resident blocks make progress, beside whatever else runs on
// the GPU, and a wait that runs out ends the launch with a status.
//
// Every product of two tiles is the six part products of weight >= 2^-16, hi.hi in one accumulator of 128 columns of tensor memory
// and the five small ones in a second: the tensor core truncates its sums, so what is added one after the other to a sum of full
// size is kept short.  The two are added in fp32, then to the register value, in ascending order of k: a fixed order, whatever
// the timing.  With everything in one accumulator the error against 64 bits is four times as large (1024 unknowns, 2048 right-hand
// sides: 1.4e-5 against 3.3e-6; the launches per block column: 1.1e-5).
#include <string.h>

#include "sp_chol_block.cuh"
#include "sp_tc.cuh"

namespace sp {
namespace {

constexpr int TB = kCholTcNB;
using Diag = DiagTiles;
constexpr int THREADS = Diag::THREADS;                    // 20 warps: producer, MMA issuer, two idle, 16 of the epilogue
constexpr int EPI0 = 4, EPI_WARPS = 16;
constexpr uint32_t BOX = 64 * TB * 2;                     // 64 columns of 128 rows, bf16: 16 KB
constexpr uint32_t OPER = 3 * BOX;                        // the three parts of 64 columns: 48 KB
constexpr uint32_t SLOT = 2 * OPER;                       // both operands of a half chunk (64 of K)
constexpr uint32_t DATA = 2 * SLOT;
constexpr uint32_t PRE_BYTES = TB * TB * 4;
constexpr uint32_t PRE_AT = (uint32_t)(Diag::SMEM - Diag::BARS * 8);   // chain block: a tile's sum, behind DiagTiles' arrays
constexpr uint32_t AREA = PRE_AT + PRE_BYTES > DATA ? PRE_AT + PRE_BYTES : DATA;
constexpr uint32_t NBARS = 11;
// [4][128] floats: maxima of a tile's rows; chain block: the rows' factors of the tile that PRE_AT holds
constexpr uint32_t ROW_MAX_AT = (AREA + (NBARS + Diag::BARS) * 8 + 15) / 16 * 16;
constexpr size_t SMEM = ROW_MAX_AT + 4 * TB * sizeof(float) + 1024 /*alignment*/;
static_assert(Diag::SMEM - Diag::BARS * 8 <= DATA, "the diagonal block's arrays lie over the operand slots");
constexpr uint32_t TMEM_COLS = 4 * TB;                    // two pairs of accumulators in turn
// about 16 seconds: a block may wait for others of its launch that have no room yet beside another stream's long kernels
constexpr long long WAIT_BUDGET = 32000000000LL;
constexpr long long DRAIN = 200000000LL;
constexpr int kFlags0 = 32;                               // flags[0]: the task counter; [1] of the first system: blocks that have come

struct SolveParams {
  const float* A;              // [nn + m, nn] fp32: lower triangle of the system, right-hand sides below
  int64_t lda;
  int nn, m, nblk, mb, group;
  __nv_bfloat16* P;            // pitch 3 np
  float* W;                    // [m, nn], may be the right-hand sides' own place
  int64_t ldw;
  float* lead;                 // optional [m, .]: the solution of the leading lead_k x lead_k system
  int64_t ld_lead;
  int lead_k;
  float* pre;                  // [2 nblk][128][128]: what the chain block takes over of a column (see TASK_PRE)
  float* pre_back;             // [nblk][128]: factors of the rows of the tile below a diagonal block (see scale_tiny_row)
  uint32_t* flags;
  int32_t* status;
  const int32_t* skip;
  long long budget;
  int64_t a_bs;                // distance of the systems' A (and W), systems = gridDim.y; the rest lies one system behind the other
  int rows, flag_words;        // rows of P and words of flags of a system
};

__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
// the tile is in memory: for loads by TMA of other blocks
__device__ __forceinline__ void publish(uint32_t* p) {
  asm volatile("fence.proxy.async;" ::: "memory");
  asm volatile("fence.acq_rel.gpu;" ::: "memory");
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(1u) : "memory");
}
// whether the predicate holds in any thread of the epilogue
__device__ __forceinline__ bool epi_any(bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "barrier.cta.red.or.pred q, 1, 512, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)v)
      : "memory");
  return r != 0;
}
// Block barrier: whether any wait of the block has run out, one answer for all threads.  (Read by each for itself behind a plain
// barrier, the flag may be set by a warp that is ahead, and the block's warps would end up at different barriers.)
__device__ __forceinline__ bool given_up(volatile int* abort_flag) { return __syncthreads_or(*abort_flag) != 0; }
__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, 512;" ::: "memory"); }
// Rows of tiny values are brought to the order of one by a power of two before they are split: below 2^-110 the low parts would be cut
// off.  row_part_max: of a thread's 32 columns of a row; where that is tiny() in any thread of the epilogue, all of them call
// scale_tiny_row (thread of row i, columns 32 g .. + 31): the factor that takes the row's product back.
__device__ __forceinline__ bool tiny(float top) { return top > 0.f && top < 0x1p-80f; }
__device__ __forceinline__ float row_part_max(const float (&v)[32]) {
  float top = 0.f;
#pragma unroll
  for (int c = 0; c < 32; ++c) top = fmaxf(top, fabsf(v[c]));
  return top;
}
__device__ __forceinline__ float scale_tiny_row(float (&v)[32], float top, float* row_max, int g, int i) {
  row_max[g * kCholTcNB + i] = top;
  epi_sync();
#pragma unroll
  for (int q = 0; q < 4; ++q) top = fmaxf(top, row_max[q * kCholTcNB + i]);
  if (!tiny(top)) return 1.f;
  const float up = top < 0x1p-104f ? 0x1p104f : 0x1p80f;
#pragma unroll
  for (int c = 0; c < 32; ++c) v[c] *= up;
  return 1.f / up;
}
__device__ __forceinline__ void arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}
// 128 x 128 x 16, bf16 operands, fp32 accumulator
__device__ __forceinline__ uint32_t instr_desc(bool b_kmajor) {
  return 1u << 4 | 1u << 7 | 1u << 10 | (b_kmajor ? 0u : 1u) << 16 | (uint32_t)(TB >> 3) << 17 | (uint32_t)(TB >> 4) << 24;
}
// parts of the six products kept, in the order of sp_linalg_tc.cu
__device__ __forceinline__ constexpr int part_a(int q) { return q == 2 || q == 5 ? 1 : q == 4 ? 2 : 0; }
__device__ __forceinline__ constexpr int part_b(int q) { return q == 1 || q == 5 ? 1 : q == 3 ? 2 : 0; }

// two values -> their three parts, packed
__device__ __forceinline__ void split3x2(float x, float y, uint32_t (&o)[3]) {
  __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
  float rx = x - __low2float(h), ry = y - __high2float(h);
  __nv_bfloat162 m = __floats2bfloat162_rn(rx, ry);
  rx -= __low2float(m);
  ry -= __high2float(m);
  __nv_bfloat162 l = __floats2bfloat162_rn(rx, ry);
  o[0] = *reinterpret_cast<uint32_t*>(&h);
  o[1] = *reinterpret_cast<uint32_t*>(&m);
  o[2] = *reinterpret_cast<uint32_t*>(&l);
}

// X(j, j) of DiagTiles is read where it lies in shared memory
struct NoOut {
  __device__ __forceinline__ void zeros(int, int, int) const {}
  __device__ __forceinline__ void tile(const float (&)[32], const float*, bool, int, int, int) const {}
};
// 32 values of a row, from chunk u0 (8 columns) of its box on, as three parts in the layout of the operands: rows of 64 columns,
// 128-byte swizzle, the parts a box apart
__device__ __forceinline__ void put_parts(uint8_t* box, int row, int u0, const float (&v)[32]) {
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    uint32_t o[4][3];
#pragma unroll
    for (int w = 0; w < 4; ++w) split3x2(v[8 * u + 2 * w], v[8 * u + 2 * w + 1], o[w]);
    uint8_t* at = box + row * 128 + (((u0 + u) ^ (row & 7)) << 4);
#pragma unroll
    for (int z = 0; z < 3; ++z) *reinterpret_cast<uint4*>(at + z * BOX) = make_uint4(o[0][z], o[1][z], o[2][z], o[3][z]);
  }
}
// place of chunk q (4 columns) of row i in a tile's sum handed to the chain block: no bank conflicts for a row per lane
__device__ __forceinline__ int pre_at(int i, int q) { return i * TB + ((q ^ (i & 31)) << 2); }
// all of an operand area (two halves of 64 columns, three parts) to memory; one thread, up to the point where the area may be written again
__device__ __forceinline__ void store_tile(const CUtensorMap* map, int part_cols, int col, int row, uint32_t src) {
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int z = 0; z < 3; ++z) tma_store_2d(map, z * part_cols + col + h * 64, row, src + h * OPER + z * BOX);
  bulk_commit();
  asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
// The six products of one pair of 16-wide slices, at the descriptors of their hi parts (a box apart: the other parts): hi.hi into d, the small
// ones into d + TB; later = 0 for the first slice of a sum.
__device__ __forceinline__ void mma_slice(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t later) {
  mma(d, a, b, idesc, later);
#pragma unroll
  for (int s = 1; s < 6; ++s)
    mma(d + TB, a + part_a(s) * (BOX >> 4), b + part_b(s) * (BOX >> 4), idesc, s > 1 ? 1u : later);
}
// the tile whose last product is multiplied by X(j, j): A (K-major) at a, X at b (rows of K, columns contiguous)
__device__ __forceinline__ void mma_by_x(uint32_t d, uint32_t a, uint32_t b) {
  const uint64_t bd = make_smem_desc(b, false, OPER);
#pragma unroll 1
  for (int k = 0; k < 8; ++k)
    mma_slice(d, make_smem_desc(a + (k >> 2) * OPER + (k & 3) * 32, true, 0), bd + k * (16 * 128 >> 4), instr_desc(false),
              k > 0 ? 1u : 0u);
}
// half h (64 of K) of the product of two tiles
__device__ __forceinline__ void mma_half(uint32_t d, uint32_t a, uint32_t b, int h) {
  const uint64_t ad = make_smem_desc(a, true, 0), bd = make_smem_desc(b, true, 0);
#pragma unroll 1
  for (int k = 0; k < 4; ++k) mma_slice(d, ad + k * 2, bd + k * 2, instr_desc(true), h > 0 || k > 0 ? 1u : 0u);
}

enum TaskKind : int { TASK_T = 0, TASK_W = 1, TASK_PRE = 2 };
struct Task {
  int kind, R, j;       // row block (in rows of P), column block
  int k0, k1;           // tiles to the left (W: of the sum)
  int lead;             // W: k of the leading system's last block (-1: none)
  int pre;              // PRE: its place
};
// The chain; then groups of p.group columns.  A group begins with the tiles that its own columns need: what the chain takes over of the
// tile below a diagonal block and of the next diagonal block (their sums over k < j), and the factor's tiles down to the first row
// behind the group; then row by row the group's tiles of the rows below, of the right-hand sides and of X.  nblk + mb tasks a
// column (one less in the last), then the W, longest sums first.
__device__ __forceinline__ Task task_of(const SolveParams& p, int t) {
  Task q;
  q.lead = q.pre = -1;
  const int C = p.nblk + p.mb, cols = p.nblk * C;
  if (t >= cols) {
    const int u = t - cols;
    q.kind = TASK_W;
    q.j = u / p.mb;
    q.R = p.nblk + u % p.mb;
    q.k0 = q.j;
    q.k1 = p.nblk;
    if (p.lead != nullptr && q.j * TB < p.lead_k) q.lead = (p.lead_k - 1) / TB;
    return q;
  }
  // (t > 0: the chain is not a task of this kind)
  const int j0 = (t - 1) / (p.group * C) * p.group, n_col = p.nblk - j0 < p.group ? p.nblk - j0 : p.group;
  const int last = j0 + p.group < p.nblk - 1 ? j0 + p.group : p.nblk - 1;     // last row of the first part
  int idx = t - 1 - j0 * C;
  q.kind = TASK_T;
  q.R = -1;
  for (int j = j0; j < j0 + n_col && q.R < 0; ++j) {
    const int pre = j + 1 < p.nblk ? 2 : 0, count = pre + (last - j - 1 > 0 ? last - j - 1 : 0);
    if (idx < count) {
      q.j = j;
      q.R = idx < pre ? j + 1 : j + 2 + idx - pre;
      if (idx < pre) {
        q.kind = TASK_PRE;
        q.pre = 2 * j + idx;
      }
    } else {
      idx -= count;
    }
  }
  if (q.R < 0) {
    const int below = p.nblk - 1 - last, rows = below + p.mb + j0;
    if (idx < rows * n_col) {
      const int r = idx / n_col;
      q.j = j0 + idx % n_col;
      q.R = r < below ? last + 1 + r : r < below + p.mb ? p.nblk + r - below : r - below - p.mb;
    } else {                                             // X within the group
      idx -= rows * n_col;
      for (q.j = j0 + 1; idx >= q.j - j0; ++q.j) idx -= q.j - j0;
      q.R = j0 + idx;
    }
  }
  q.k0 = q.R < q.j ? q.R : 0;
  q.k1 = q.j;
  if (q.kind == TASK_PRE && (q.pre & 1) != 0) q.j = q.R;  // the diagonal block (j + 1, j + 1), also over k < j
  return q;
}

__device__ __forceinline__ float ld_shared(uint32_t at) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(at) : "memory");
  return v;
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
// (a call of its own: see the chain)
__device__ __noinline__ void eliminate_block(uint32_t off, uint32_t bars, int j, int nb, int32_t* status) {
  extern __shared__ uint8_t smem_raw[];
  int t;
  asm volatile("mov.u32 %0, %%tid.x;" : "=r"(t));
  Diag::eliminate<true>(t, reinterpret_cast<float*>(smem_raw + off), bars, (uint32_t)j & 1u, nullptr, 0, nb, NoOut{}, (int64_t)j * TB,
                        status);
}
// A thread's place: of the epilogue's threads (warps from EPI0 on) row i, columns 32 g .. + 31 of a tile.  Volatile: formed where it is
// called.
struct Place {
  int warp, lane, g, i;
  uint32_t data, tmem;
  uint8_t* ptr;
};
__device__ __forceinline__ Place place(uint8_t* smem, const volatile uint32_t* s_tmem) {
  Place q;
  int t;
  uint32_t zero;
  asm volatile("mov.u32 %0, %%tid.x;" : "=r"(t));
  asm volatile("mov.u32 %0, 0;" : "=r"(zero));
  q.warp = t >> 5;
  q.lane = t & 31;
  q.g = (q.warp - EPI0) >> 2;
  q.i = (q.warp & 3) * 32 + q.lane;
  const uint32_t raw = smem_u32(smem), up = (raw + zero + 1023u) & ~1023u;
  q.data = up;
  q.ptr = smem + (up - raw);
  q.tmem = *s_tmem;
  return q;
}
// waits for the product of two tiles (both its accumulators at `at` and at + TB): f(c, value) for the thread's 32 columns
template <typename F>
__device__ __forceinline__ bool read_sum(uint32_t tfull, uint32_t tempty, uint32_t parity, uint32_t at, int lane,
                                         volatile int* abort_flag, long long budget, F&& f) {
  const bool there = __all_sync(0xffffffffu, mbar_wait(tfull, parity, abort_flag, budget));
  tc_fence_after();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t hi[16], lo[16];
    tc_ld16(at + h * 16, hi);
    tc_ld16(at + TB + h * 16, lo);
    tc_wait_ld();
#pragma unroll
    for (int c = 0; c < 16; ++c) f(h * 16 + c, __uint_as_float(hi[c]) + __uint_as_float(lo[c]));
  }
  tc_fence_before();
  __syncwarp();
  if (lane == 0) arrive(tempty);
  return there;
}
// until a flag is set
__device__ __forceinline__ bool wait_flag(const uint32_t* f, volatile int* abort_flag, long long budget) {
  const long long t0 = clock64();
  while (ld_acquire(f) == 0u) {
    if (*abort_flag != 0 || clock64() - t0 > budget) {
      *abort_flag = 1;
      return false;
    }
  }
  return true;
}
// a block on the diagonal, where DiagTiles expects its tiles: zero above the diagonal, an identity beyond nb
__device__ __forceinline__ void stage_block(const Place& at, const float (&v)[32], int nb) {
  if (at.g > (at.warp & 3)) return;
  float* dst = reinterpret_cast<float*>(at.ptr) + Diag::staged_at(at.i, at.g * 32);
#pragma unroll
  for (int c = 0; c < 32; c += 4) {
    float u[4];
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      const int col = at.g * 32 + c + w;
      u[w] = col > at.i ? 0.f : at.i >= nb ? (col == at.i ? 1.f : 0.f) : v[c + w];
    }
    *reinterpret_cast<float4*>(dst + c) = make_float4(u[0], u[1], u[2], u[3]);
  }
}

// BATCH: gridDim.y systems.  (One system has a form of its own: registers are short.)
template <bool BATCH>
__global__ void __launch_bounds__(THREADS, 1)
solve_tc_kernel(const __grid_constant__ CUtensorMap tmP, const __grid_constant__ CUtensorMap tmY, const SolveParams p) {
  dependents_may_launch();
  if (p.skip != nullptr) {
    wait_for_predecessors();
    if (*p.skip != 0) return;
  }
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint32_t s_tmem;
  __shared__ volatile int s_system;
  __shared__ int s_abort, s_ticket[2];
  const uint32_t raw = smem_u32(smem_raw), data = (raw + 1023u) & ~1023u, bars = data + AREA;
  uint8_t* const data_ptr = smem_raw + (data - raw);
  auto full = [&](int h) { return bars + 8u * h; };              // a half chunk has landed
  auto empty = [&](int h) { return bars + 8u * (2 + h); };       // its products have read it
  auto tfull = [&](int b) { return bars + 8u * (4 + b); };       // an accumulator is complete
  auto tempty = [&](int b) { return bars + 8u * (6 + b); };      // and read
  const uint32_t xfull = bars + 8u * 8, aready = bars + 8u * 9;  // X(j, j) has landed; the left operand is written
  const uint32_t xfree = bars + 8u * 10;                         // chain: X(j, j) has left (barriers in this order there too)
  const uint32_t dbars = bars + 8u * NBARS;
  float* const row_max = reinterpret_cast<float*>(data_ptr + ROW_MAX_AT);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* abort_flag = &s_abort;
  if (threadIdx.x == 0) {
    s_abort = 0;
    for (int h = 0; h < 2; ++h) {
      mbar_init(full(h), 1);
      mbar_init(empty(h), 1);
      mbar_init(tfull(h), 1);
      mbar_init(tempty(h), EPI_WARPS);
    }
    mbar_init(xfull, 1);
    mbar_init(xfree, 1);
    mbar_init(aready, EPI_WARPS);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
  }
  for (uint32_t b = threadIdx.x; b < Diag::BARS; b += THREADS) mbar_init(dbars + 8u * b, 1);
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)), "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  wait_for_predecessors();

  // The system, in the order in which blocks come, which need not be that of their numbers: all blocks of a system are there before the
  // next one's first, so two running blocks are enough here too.  (In shared memory: registers are short.)
  if constexpr (BATCH) {
    if (threadIdx.x == 0) s_system = (int)(atomicAdd(p.flags + 1, 1u) / gridDim.x);
    __syncthreads();
  }
  const auto system = [&] { return BATCH ? (int)s_system : 0; };
  uint32_t* const ticket_of = p.flags + (int64_t)system() * p.flag_words;
  uint32_t* const flags = ticket_of + kFlags0;
  uint32_t* const pre_flags = flags + (int64_t)p.nblk * (p.nblk + p.mb);
  const int total = p.nblk * (p.nblk + 2 * p.mb), np = p.nblk * TB;
  // chunks, accumulators, written operands, loads of X(j, j) so far (the same in every role)
  uint32_t kc = 0, cc = 0, xc = 0, fc = 0;
  // epilogue threads: row i, columns 32 g .. + 31 of a tile
  const int g = (warp - EPI0) >> 2, i = (warp & 3) * 32 + lane;
  const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(g * 32);
  // the next product of two tiles: f(c, value) for this thread's 32 columns
  auto sum_of = [&](uint32_t cl, auto&& f) {
    return read_sum(tfull(cl & 1u), tempty(cl & 1u), (cl >> 1) & 1u, taddr + (cl & 1u) * 2 * TB, lane, abort_flag, p.budget, f);
  };
  if (threadIdx.x == 0) s_ticket[0] = (int)atomicAdd(ticket_of, 1u);
  __syncthreads();
  if (s_ticket[0] == 0) {
    // ------------------------------------------------------------------ the chain: all diagonal blocks, one after the other
    // Areas: X(j, j) lies where DiagTiles worked, the tile below it in the second slot; its sum comes in behind DiagTiles' arrays.  The
    // elimination takes nearly all registers, and what is spilled goes to the second-level cache, since shared memory has taken
    // the first (40 us a block with 500 bytes spilled inside it, 30 with 130).  So it is a call of its own, and everything but j
    // is formed anew behind it (Place).
    Place at = place(smem_raw, &s_tmem);
    if (at.warp >= EPI0) {
      float v[32];
#pragma unroll
      for (int c = 0; c < 32; ++c) {
        const int col = at.g * 32 + c;
        v[c] = at.i < p.nn && col <= at.i && col < p.nn ? p.A[(int64_t)system() * p.a_bs + (int64_t)at.i * p.lda + col] : 0.f;
      }
      stage_block(at, v, p.nn < TB ? p.nn : TB);
    }
    for (int j = 0; j < p.nblk; ++j) {
      if (given_up(abort_flag)) break;
      const int nb = p.nn - j * TB < TB ? p.nn - j * TB : TB;
      eliminate_block(at.data - smem_u32(smem_raw), at.data + AREA + 8u * NBARS, j, nb, p.status);
      at = place(smem_raw, &s_tmem);
      const bool more = j + 1 < p.nblk;
      const uint32_t par = (uint32_t)j & 1u, bars_j = at.data + AREA;
      const uint32_t tfull0 = bars_j + 8u * 4, tempty0 = bars_j + 8u * 6, xfull_j = bars_j + 8u * 8, aready_j = bars_j + 8u * 9,
                     xfree_j = bars_j + 8u * 10;
      uint32_t* const flags_j = p.flags + (int64_t)system() * p.flag_words + kFlags0;
      uint32_t* const pre_j = flags_j + (int64_t)p.nblk * (p.nblk + p.mb) + 2 * j;
      const float* const sums = p.pre + (int64_t)(2 * (system() * p.nblk + j)) * (TB * TB);
      const int row0 = system() * p.rows;
      if (at.warp == 0 && more && at.lane == 0 && wait_flag(pre_j, abort_flag, p.budget)) {     // (its tile of L is done first)
        asm volatile("fence.proxy.async;" ::: "memory");
        mbar_expect_tx(xfull_j, PRE_BYTES + TB * 4);
        bulk_load(at.data + PRE_AT, sums, PRE_BYTES, xfull_j);
        bulk_load(at.data + ROW_MAX_AT, p.pre_back + (int64_t)(system() * p.nblk + j) * TB, TB * 4, xfull_j);
      }
      __syncwarp();
      __syncthreads();                       // X is complete
      __syncwarp();
      if (at.warp >= EPI0) {
        float v[32];
        const int ns = (p.nn - j * TB + 31) / 32;
        if (at.g >= (at.warp & 3) && at.g < ns) {
          const uint32_t col = at.data + 4u * (uint32_t)((TB + at.g * 32) * Diag::P + at.i);
#pragma unroll
          for (int c = 0; c < 32; ++c) v[c] = ld_shared(col + 4u * c * Diag::P);
        } else {
          const int one = at.g >= ns ? at.i - at.g * 32 : -1;    // beyond the matrix: an identity
#pragma unroll
          for (int c = 0; c < 32; ++c) v[c] = c == one ? 1.f : 0.f;
        }
        epi_sync();                          // and read
        put_parts(at.ptr + (at.g >> 1) * OPER, at.i, (at.g & 1) * 4, v);
        if (more) {
          mbar_wait(xfull_j, par, abort_flag, p.budget);
          const float* src = reinterpret_cast<const float*>(at.ptr + PRE_AT);
#pragma unroll
          for (int c = 0; c < 32; c += 4) {
            const float4 u = *reinterpret_cast<const float4*>(src + pre_at(at.i, at.g * 8 + c / 4));
            v[c] = u.x; v[c + 1] = u.y; v[c + 2] = u.z; v[c + 3] = u.w;
          }
          epi_sync();                        // the sum lies where the operand is written
          put_parts(at.ptr + SLOT + (at.g >> 1) * OPER, at.i, (at.g & 1) * 4, v);
        }
      }
      fence_async_smem();
      if (given_up(abort_flag)) break;
      if (at.warp == 1 && more && at.lane == 0) {
        bool ok = mbar_wait(tempty0, par ^ 1u, abort_flag, p.budget);
        if (ok) {
          tc_fence_after();
          mma_by_x(at.tmem, at.data + SLOT, at.data);
          commit(tfull0);
          ok = mbar_wait(tempty0 + 8u, par ^ 1u, abort_flag, p.budget) && mbar_wait(aready_j, par, abort_flag, p.budget);
          if (ok) {
            tc_fence_after();
#pragma unroll 1
            for (int h = 0; h < 2; ++h) mma_half(at.tmem + 2 * TB, at.data + SLOT + h * OPER, at.data + SLOT + h * OPER, h);
            commit(tfull0 + 8u);
          }
        }
      } else if (at.warp == 2 && at.lane == 0) {
        store_tile(&tmP, np, j * TB, row0 + j * TB, at.data);
        arrive(xfree_j);
        bulk_wait_all();
        publish(flags_j + (int64_t)j * p.nblk + j);
      } else if (at.warp == 3 && more && at.lane == 0) {
        if (mbar_wait(aready_j, par, abort_flag, p.budget)) {
          store_tile(&tmP, np, j * TB, row0 + (j + 1) * TB, at.data + SLOT);
          bulk_wait_all();
          publish(flags_j + (int64_t)(j + 1) * p.nblk + j);
        }
      } else if (at.warp >= EPI0 && more) {
        const uint32_t taddr_j = at.tmem + ((uint32_t)((at.warp & 3) * 32) << 16) + (uint32_t)(at.g * 32);
        float d[32];
        const bool ok = read_sum(tfull0, tempty0, par, taddr_j, at.lane, abort_flag, p.budget, [&](int c, float u) { d[c] = u; });
        const float back = ld_shared(at.data + ROW_MAX_AT + 4u * (uint32_t)at.i);
        if (back != 1.f) {
#pragma unroll
          for (int c = 0; c < 32; ++c) d[c] *= back;
        }
        put_parts(at.ptr + SLOT + (at.g >> 1) * OPER, at.i, (at.g & 1) * 4, d);
        fence_async_smem();
        __syncwarp();
        if (ok && at.lane == 0) arrive(aready_j);
        // the sum of the next diagonal block, while its last product is formed
        wait_flag(pre_j + 1, abort_flag, p.budget);
        __syncwarp();
        const float4* src = reinterpret_cast<const float4*>(sums + TB * TB) + (at.warp - EPI0) * 32 + at.lane;
#pragma unroll
        for (int c = 0; c < 32; c += 4) {
          const float4 u = src[c / 4 * (EPI_WARPS * 32)];
          d[c] = u.x; d[c + 1] = u.y; d[c + 2] = u.z; d[c + 3] = u.w;
        }
        read_sum(tfull0 + 8u, tempty0 + 8u, par, taddr_j + 2 * TB, at.lane, abort_flag, p.budget, [&](int c, float u) { d[c] -= u; });
        mbar_wait(xfree_j, par, abort_flag, p.budget);
        stage_block(at, d, p.nn - (j + 1) * TB < TB ? p.nn - (j + 1) * TB : TB);
      }
      __syncwarp();
    }
    __syncthreads();
  } else
  for (int turn = 0;; turn ^= 1) {
    const int ticket = s_ticket[turn];
    int* const next_ticket = &s_ticket[turn ^ 1];      // written while others may still read the first
    if (ticket >= total) break;
    const Task tk = task_of(p, ticket);
    // chunks of the sum: q -> k; W with a leading system takes its last block's masked copy first
    const int nq = tk.k1 - tk.k0 + (tk.lead >= 0 ? 1 : 0);
    const int masked = tk.lead >= 0 ? tk.lead - tk.k0 : -1;       // the chunk that reads the masked copy
    auto k_of = [&](int q) { return tk.k0 + (masked >= 0 && q > masked ? q - 1 : q); };
    const bool same = tk.R == tk.j;      // both operands are the same tiles
    const int row0 = system() * p.rows;
    bool ok = true;

    if (warp == 0) {
      // ------------------------------------------------------------------ loads
      const uint32_t* fa = flags + (int64_t)tk.R * p.nblk;
      const uint32_t* fb = flags + (int64_t)tk.j * p.nblk;
      // until tile k of both rows is there (lane l looks at k + l); known: how far the look reached
      int known = tk.k0;
      auto wait_tiles = [&](int k, int k1, bool both) {
        if (k < known) return true;
        const long long t0 = clock64();
        for (;;) {
          const int kk = k + lane;
          const bool there = kk < k1 && ld_acquire(fa + kk) != 0u && (!both || ld_acquire(fb + kk) != 0u);
          const uint32_t b = __ballot_sync(0xffffffffu, there);
          if (b & 1u) {
            known = k + (b == 0xffffffffu ? 32 : __ffs(~b) - 1);
            break;
          }
          const bool out = *abort_flag != 0 || clock64() - t0 > p.budget;
          if (__any_sync(0xffffffffu, out)) {
            *abort_flag = 1;
            return false;
          }
          __nanosleep(20);
        }
        __syncwarp();        // lane 0 loads what other lanes have acquired: a vote orders no memory
        asm volatile("fence.proxy.async;" ::: "memory");
        return true;
      };
      uint32_t kl = kc;
      for (int q = 0; q < nq && ok; ++q, ++kl) {
        const int k = k_of(q);
        ok = wait_tiles(k, tk.k1, !same);
        if (ok && lane == 0) {
          for (int h = 0; h < 2 && ok; ++h) {
            if (!mbar_wait(empty(h), (kl & 1u) ^ 1u, abort_flag, p.budget)) { ok = false; break; }
            mbar_expect_tx(full(h), same ? OPER : SLOT);
            const uint32_t dst = data + h * SLOT;
#pragma unroll
            for (int z = 0; z < 3; ++z) {
              const int col = k * TB + h * 64;
              if (q == masked) tma_load_2d_local(dst + z * BOX, &tmY, z * TB + h * 64, (tk.R - p.nblk) * TB, full(h));
              else tma_load_2d_local(dst + z * BOX, &tmP, z * np + col, row0 + tk.R * TB, full(h));
              if (!same) tma_load_2d_local(dst + OPER + z * BOX, &tmP, z * np + col, row0 + tk.j * TB, full(h));
            }
          }
        }
        ok = __all_sync(0xffffffffu, ok);
      }
      if (tk.kind == TASK_T && ok) {
        // X(j, j), rows of K with the columns contiguous, once the last products have read the slots
        fa = flags + (int64_t)tk.j * p.nblk;
        known = -1;
        ok = wait_tiles(tk.j, tk.j + 1, false);
        if (ok && lane == 0) {
          for (int h = 0; h < 2 && ok; ++h) ok = mbar_wait(empty(h), (kl & 1u) ^ 1u, abort_flag, p.budget);
          if (ok) {
            mbar_expect_tx(xfull, SLOT);
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
              for (int z = 0; z < 3; ++z)
                tma_load_2d_local(data + SLOT + h * OPER + z * BOX, &tmP, z * np + tk.j * TB + h * 64, row0 + tk.j * TB, xfull);
          }
        }
      }
    } else if (warp == 1) {
      // ------------------------------------------------------------------ products
      if (lane == 0) {
        uint32_t kl = kc, cl = cc;
        for (int q = 0; q < nq && ok; ++q, ++kl, ++cl) {
          const uint32_t d = tmem + (cl & 1u) * 2 * TB;
          ok = mbar_wait(tempty(cl & 1u), ((cl >> 1) & 1u) ^ 1u, abort_flag, p.budget);
          for (int h = 0; h < 2 && ok; ++h) {
            ok = mbar_wait(full(h), kl & 1u, abort_flag, p.budget);
            if (!ok) break;
            tc_fence_after();
            const uint32_t a = data + h * SLOT;
            mma_half(d, a, same ? a : a + OPER, h);
            commit(empty(h));
          }
          if (ok) commit(tfull(cl & 1u));
        }
        if (tk.kind == TASK_T && ok) {
          const uint32_t d = tmem + (cl & 1u) * 2 * TB;
          ok = mbar_wait(tempty(cl & 1u), ((cl >> 1) & 1u) ^ 1u, abort_flag, p.budget) &&
               mbar_wait(aready, xc & 1u, abort_flag, p.budget) && mbar_wait(xfull, fc & 1u, abort_flag, p.budget);
          if (ok) {
            tc_fence_after();
            mma_by_x(d, data, data + SLOT);
            commit(tfull(cl & 1u));
          }
        }
        *next_ticket = (int)atomicAdd(ticket_of, 1u);
      }
    } else if (warp >= EPI0) {
      // ------------------------------------------------------------------ the running value, and what leaves
      const int col0 = tk.j * TB + g * 32;
      float s[32];
      {
        const int64_t row = tk.R < p.nblk ? (int64_t)tk.R * TB + i : (int64_t)p.nn + (int64_t)(tk.R - p.nblk) * TB + i;
        const bool have = tk.kind != TASK_W && tk.R >= tk.j &&
                          (tk.R < p.nblk ? row < p.nn : row < (int64_t)p.nn + p.m);
        const float* src = p.A + (int64_t)system() * p.a_bs + row * p.lda + col0;
        const int n_col = have ? (p.nn - col0 < 32 ? p.nn - col0 : 32) : 0;
        if (n_col == 32 && p.lda % 4 == 0) {
#pragma unroll
          for (int c = 0; c < 32; c += 4) {
            const float4 v = *reinterpret_cast<const float4*>(src + c);
            s[c] = v.x; s[c + 1] = v.y; s[c + 2] = v.z; s[c + 3] = v.w;
          }
        } else {
#pragma unroll
          for (int c = 0; c < 32; ++c) s[c] = c < n_col ? src[c] : 0.f;
        }
      }
      uint32_t cl = cc;
      for (int q = 0; q < nq && ok; ++q, ++cl) {
        if (q != masked) {
          ok = sum_of(cl, [&](int c, float v) { s[c] -= v; });
        } else {
          // the leading system's solution ends here
          const int64_t row = (int64_t)(tk.R - p.nblk) * TB + i;
          float* dst = p.lead + row * p.ld_lead + col0;
          const int n_out = row < p.m ? p.lead_k - col0 : 0;
          ok = sum_of(cl, [&](int c, float v) { if (c < n_out) dst[c] = v - s[c]; });
        }
      }
      if (tk.kind == TASK_T) {
        const float top = row_part_max(s);
        const float back = epi_any(tiny(top)) ? scale_tiny_row(s, top, row_max, g, i) : 1.f;
        uint8_t* const box = data_ptr + (g >> 1) * OPER;
        if (ok) {
          put_parts(box, i, (g & 1) * 4, s);
          fence_async_smem();
          __syncwarp();
          if (lane == 0) arrive(aready);
          ok = sum_of(cl, [&](int c, float v) { s[c] = v * back; });
        }
        if (ok) {
          put_parts(box, i, (g & 1) * 4, s);
          fence_async_smem();
        }
        epi_sync();
        const bool one = threadIdx.x == EPI0 * 32 && *abort_flag == 0;
        if (one) store_tile(&tmP, np, tk.j * TB, row0 + tk.R * TB, data);
        if (p.lead != nullptr && tk.R >= p.nblk && tk.j == (p.lead_k - 1) / TB) {
          // copy of the right-hand sides' last block of the leading system, zero beyond it
          epi_sync();
#pragma unroll
          for (int c = 0; c < 32; ++c) s[c] = col0 + c < p.lead_k ? s[c] : 0.f;
          put_parts(box, i, (g & 1) * 4, s);
          fence_async_smem();
          epi_sync();
          if (one) store_tile(&tmY, TB, 0, (tk.R - p.nblk) * TB, data);
        }
        if (one) {
          bulk_wait_all();
          publish(flags + (int64_t)tk.R * p.nblk + tk.j);
        }
      } else if (tk.kind == TASK_W) {
        const int64_t row = (int64_t)(tk.R - p.nblk) * TB + i;
        if (ok && row < p.m) {
          float* dst = p.W + (int64_t)system() * p.a_bs + row * p.ldw + col0;
          if (col0 + 32 <= p.nn && p.ldw % 4 == 0) {
#pragma unroll
            for (int c = 0; c < 32; c += 4)
              *reinterpret_cast<float4*>(dst + c) = make_float4(-s[c], -s[c + 1], -s[c + 2], -s[c + 3]);
          } else {
#pragma unroll
            for (int c = 0; c < 32; ++c)
              if (col0 + c < p.nn) dst[c] = -s[c];
          }
        }
      } else {
        // for the chain block (a diagonal block thread by thread, as it is read; the tile below one for a copy to shared memory, and what
        // its rows were divided by: as a rule one, and known behind the barrier that the flag needs anyway)
        float* dst = p.pre + (int64_t)(2 * system() * p.nblk + tk.pre) * (TB * TB);
        const auto put = [&] {
#pragma unroll
          for (int c = 0; c < 32; c += 4) {
            const int at = same ? (c / 4 * (EPI_WARPS * 32) + threadIdx.x - EPI0 * 32) * 4 : pre_at(i, g * 8 + c / 4);
            *reinterpret_cast<float4*>(dst + at) = make_float4(s[c], s[c + 1], s[c + 2], s[c + 3]);
          }
        };
        float* const back = p.pre_back + (int64_t)(system() * p.nblk + tk.j) * TB + i;
        put();
        if (!same && g == 0) *back = 1.f;
        const float top = row_part_max(s);
        if (epi_any(!same && tiny(top))) {
          const float f = scale_tiny_row(s, top, row_max, g, i);
          put();
          if (g == 0) *back = f;
          epi_sync();
        }
        if (threadIdx.x == EPI0 * 32 && *abort_flag == 0) publish(pre_flags + tk.pre);
      }
    }
    __syncwarp();            // (the block's barriers count whole warps)
    kc += (uint32_t)nq;
    cc += (uint32_t)nq + (tk.kind == TASK_T ? 1u : 0u);
    xc += tk.kind == TASK_T ? 1u : 0u;
    fc += tk.kind == TASK_T ? 1u : 0u;
    fence_async_smem();
    if (given_up(abort_flag)) break;
  }
  if (*abort_flag != 0) {
    // a wait ran out: copies and products in flight get time to end before shared and tensor memory are released
    if (threadIdx.x == 0) report_status(p.status, SP_ERR_TIMEOUT, (int32_t)blockIdx.x, 13);
    const long long t0 = clock64();
    while (clock64() - t0 < DRAIN) {}
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
}

}  // namespace

size_t solve_tc_flag_words(int64_t n, int64_t m) {
  const size_t nblk = (size_t)ceil_div(n, (int64_t)TB), mb = (size_t)ceil_div(m, (int64_t)TB);
  return kFlags0 + nblk * (nblk + mb) + 2 * nblk;
}

sp_status solve_tc(const float* A, int64_t nn, int64_t m, int64_t lda, float* W, int64_t ldw, const SolveOneBufs& b,
                   float* lead, int64_t ld_lead, int64_t lead_k, int32_t* status_dev, cudaStream_t stream, int batch, int64_t a_bs) {
  // (2^27 right-hand sides have parts of 300 GB at least; up to there rows, tasks and flags are counted in 32 bits)
  if (!solve_in_one(nn) || m < 1 || m > (1 << 27) || batch < 1 || batch > 65535 || (batch > 1 && lead != nullptr)) return SP_ERR_SHAPE;
  SolveParams p;
  memset(&p, 0, sizeof(p));
  p.A = A;
  p.lda = lda;
  p.nn = (int)nn;
  p.m = (int)m;
  p.nblk = (int)ceil_div(nn, (int64_t)TB);
  p.mb = (int)ceil_div(m, (int64_t)TB);
  // Columns that are worked on together: a row's tiles are then read for all of them at about the same time, once from memory.  1 / 2 / 4
  // columns, ms: 4096 unknowns, 3302 right-hand sides 1.25 / 1.24 / 1.31, 6553 / 4096 3.85 / 3.68 / 3.77, 8192 / 2048 4.41 / 4.09 /
  // 3.96, 11000 / 2048 9.09 / 8.32 / 8.37; smaller ones, whose parts the second-level cache holds, equal.
  p.group = p.nblk >= 60 ? 4 : p.nblk >= 40 ? 2 : 1;
  const int64_t np = (int64_t)p.nblk * TB, rows = np + (int64_t)p.mb * TB;
  p.P = reinterpret_cast<__nv_bfloat16*>(b.P);
  p.W = W;
  p.ldw = ldw;
  p.lead = lead;
  p.ld_lead = ld_lead;
  p.lead_k = (int)lead_k;
  p.pre = b.pre;
  p.pre_back = b.pre + (size_t)batch * 2 * p.nblk * TB * TB;
  p.flags = b.flags;
  p.status = status_dev;
  p.skip = skip_flag();
  p.a_bs = a_bs;
  p.rows = (int)rows;
  p.flag_words = (int)solve_tc_flag_words(nn, m);
  if (rows * batch > 0x7fffffff) return SP_ERR_SHAPE;
  p.budget = wait_budget_cycles() > 0 ? wait_budget_cycles() : WAIT_BUDGET;
  CUtensorMap tmP, tmY;
  if (!make_map(&tmP, false, b.P, 3 * np, rows * batch, 3 * np, 64, TB) ||
      !make_map(&tmY, false, lead ? b.Y : b.P, 3 * TB, (int64_t)p.mb * TB, 3 * TB, 64, TB))      // (read for `lead` alone)
    return SP_ERR_CUDA;
  static PerDeviceOnce attr_once;
  if (attr_once.run([] {
        const cudaError_t e = cudaFuncSetAttribute(solve_tc_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM);
        return e != cudaSuccess ? e : cudaFuncSetAttribute(solve_tc_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM);
      }) != cudaSuccess)
    return SP_ERR_CUDA;
  if (cudaMemsetAsync(b.flags, 0, (size_t)p.flag_words * batch * sizeof(uint32_t), stream) != cudaSuccess) return SP_ERR_CUDA;
  // (a system has two blocks at least: the chain waits for sums of the others)
  const int64_t tasks = (int64_t)p.nblk * (p.nblk + 2 * p.mb), share = sm_count() / batch, blocks = share > 2 ? share : 2;
  count_launch();
  launch(batch > 1 ? solve_tc_kernel<true> : solve_tc_kernel<false>, dim3((unsigned)(tasks < blocks ? tasks : blocks), (unsigned)batch),
         THREADS, SMEM, stream, tmP, tmY, p);
  return cudaGetLastError() == cudaSuccess ? SP_OK : SP_ERR_CUDA;
}

}  // namespace sp
