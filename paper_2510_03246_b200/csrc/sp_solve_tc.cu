// A regularised solve W = R G^-1 in ONE launch: fp32 Cholesky factorisation of G, forward substitution of the right-hand sides
// R, the inverse of the factor, and the product of both, as a graph of 128 x 128 tiles on the tensor cores.
//
// Tiles (row block r, column block j), all held as three bf16 parts (see sp_linalg_tc.cu) in one array P of np + m rows:
//   r > j  : L(r, j) of the factor;
//   r <= j : X(r, j) of X = inv(L)^T, whose rows are those of an identity carried along (X L^T = I);
//   r >= nblk: the forward-substituted right-hand sides Y.
// A tile is one task of one thread block.  It takes its entry of [G; I; R] less sum_k tile(r, k) L(j, k)^T over the k that exist to
// its left (left-looking: the running value stays in registers, nothing is read back and rewritten), and
//   D(j)    : factorises the block on the diagonal and inverts the factor (DiagTiles): X(j, j);
//   T(r, j) : multiplies by X(j, j) = inv(L_jj)^T;
//   W(r, j) : sum_k Y(r, k) X(j, k)^T over k >= j, the result (last, when all columns are there).
// So there is no backward sweep, a serial chain of its own, and what follows a diagonal block (its column's next tile, the next
// block's last update) waits for flags of its own tiles, not for launches.
//
// Tasks are taken by a counter in an order in which every task comes after those it reads.  A block that waits therefore waits for
// a task that a running block has: any number of resident blocks makes progress, beside whatever else runs on the GPU.
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
constexpr uint32_t NBARS = 10;
constexpr size_t SMEM = DATA + 1024 /*alignment*/ + (NBARS + Diag::BARS) * 8 + 4 * TB * sizeof(float) /*row maxima*/;
static_assert(Diag::SMEM - Diag::BARS * 8 <= DATA, "the diagonal block's arrays lie over the operand slots");
constexpr uint32_t TMEM_COLS = 4 * TB;                    // two pairs of accumulators in turn
constexpr long long WAIT_BUDGET = 4000000000LL;           // about two seconds
constexpr long long DRAIN = 200000000LL;
constexpr int kFlags0 = 32;                               // flags[0]: the task counter

struct SolveParams {
  const float* A;              // [nn + m, nn] fp32: lower triangle of the system, right-hand sides below
  int64_t lda;
  int nn, m, nblk, mb;
  __nv_bfloat16* P;
  int64_t ldp;                 // 3 np
  float* W;                    // [m, nn], may be the right-hand sides' own place
  int64_t ldw;
  float* lead;                 // optional [m, .]: the solution of the leading lead_k x lead_k system
  int64_t ld_lead;
  int lead_k;
  uint32_t* flags;
  int32_t* status;
  const int32_t* skip;
  long long budget;
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
__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, 512;" ::: "memory"); }
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

// X(j, j) of DiagTiles as parts: D points at its first element
struct PartsOut {
  __nv_bfloat16* D;
  int64_t ldp, np;
  __device__ __forceinline__ void row(int i, int col, const float (&a)[32], bool zero) const {
#pragma unroll
    for (int c = 0; c < 32; c += 8) {
      uint32_t o[4][3];
#pragma unroll
      for (int e = 0; e < 4; ++e) split3x2(zero ? 0.f : a[c + 2 * e], zero ? 0.f : a[c + 2 * e + 1], o[e]);
#pragma unroll
      for (int z = 0; z < 3; ++z)
        *reinterpret_cast<uint4*>(D + i * ldp + z * np + col + c) = make_uint4(o[0][z], o[1][z], o[2][z], o[3][z]);
    }
  }
  __device__ __forceinline__ void zeros(int rb, int s, int lane) const {
#pragma unroll
    for (int c = 0; c < 32; c += 8)
#pragma unroll
      for (int z = 0; z < 3; ++z)
        *reinterpret_cast<uint4*>(D + (s * 32 + lane) * ldp + z * np + rb * 32 + c) = make_uint4(0, 0, 0, 0);
  }
  __device__ __forceinline__ void tile(const float (&a)[32], const float*, bool, int rb, int s, int lane) const {
    row(rb * 32 + lane, s * 32, a, false);
  }
};

enum TaskKind : int { TASK_D = 0, TASK_T = 1, TASK_W = 2 };
struct Task {
  int kind, R, j;       // row block (in rows of P), column block
  int k0, k1;           // tiles to the left (W: of the sum)
  int lead;             // W: k of the leading system's last block (-1: none)
};
// D(0); then column by column: the tile below the diagonal and the next diagonal block first (the chain), the factor's other
// tiles, the right-hand sides, X.  nblk + mb tasks a column (one less in the last), then the W, longest sums first.
__device__ __forceinline__ Task task_of(const SolveParams& p, int t) {
  Task q;
  q.lead = -1;
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
  q.kind = TASK_T;
  q.j = t == 0 ? 0 : (t - 1) / C;
  const int idx = t == 0 ? 0 : (t - 1) % C, below = p.nblk - 1 - q.j, rest = below > 0 ? idx - (below + 1) : idx;
  if (t == 0) {
    q.kind = TASK_D;
    q.R = 0;
  } else if (rest >= 0) {
    q.R = rest < p.mb ? p.nblk + rest : rest - p.mb;
  } else if (idx == 1) {
    q.kind = TASK_D;
    q.R = ++q.j;
  } else {
    q.R = q.j + (idx == 0 ? 1 : idx);
  }
  q.k0 = q.R < q.j ? q.R : 0;
  q.k1 = q.j;
  return q;
}

__global__ void __launch_bounds__(THREADS, 1)
solve_tc_kernel(const __grid_constant__ CUtensorMap tmP, const __grid_constant__ CUtensorMap tmY, const SolveParams p) {
  dependents_may_launch();
  if (p.skip != nullptr) {
    wait_for_predecessors();
    if (*p.skip != 0) return;
  }
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort, s_ticket[2];
  const uint32_t raw = smem_u32(smem_raw), data = (raw + 1023u) & ~1023u, bars = data + DATA;
  uint8_t* const data_ptr = smem_raw + (data - raw);
  auto full = [&](int h) { return bars + 8u * h; };              // a half chunk has landed
  auto empty = [&](int h) { return bars + 8u * (2 + h); };       // its products have read it
  auto tfull = [&](int b) { return bars + 8u * (4 + b); };       // an accumulator is complete
  auto tempty = [&](int b) { return bars + 8u * (6 + b); };      // and read
  const uint32_t xfull = bars + 8u * 8, aready = bars + 8u * 9;  // X(j, j) has landed; the left operand is written
  const uint32_t dbars = bars + 8u * NBARS;
  float* const row_max = reinterpret_cast<float*>(data_ptr + DATA + (NBARS + Diag::BARS) * 8);   // [4][128]
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

  uint32_t* const flags = p.flags + kFlags0;
  const int total = p.nblk * (p.nblk + 2 * p.mb), np = p.nblk * TB;
  uint32_t kc = 0, cc = 0, xc = 0, dc = 0;   // chunks, accumulators, final products and diagonal blocks so far (the same in every role)
  if (threadIdx.x == 0) s_ticket[0] = (int)atomicAdd(p.flags, 1u);
  __syncthreads();
  for (int turn = 0;; turn ^= 1) {
    const int ticket = s_ticket[turn];
    int* const next_ticket = &s_ticket[turn ^ 1];      // written while others may still read the first
    if (ticket >= total) break;
    const Task tk = task_of(p, ticket);
    // chunks of the sum: q -> k; W with a leading system takes its last block's masked copy first
    const int nq = tk.k1 - tk.k0 + (tk.lead >= 0 ? 1 : 0);
    const int masked = tk.lead >= 0 ? tk.lead - tk.k0 : -1;       // the chunk that reads the masked copy
    auto k_of = [&](int q) { return tk.k0 + (masked >= 0 && q > masked ? q - 1 : q); };
    const int Brow = tk.kind == TASK_W ? tk.j : tk.kind == TASK_D ? tk.R : tk.j;
    bool ok = true;

    if (warp == 0) {
      // ------------------------------------------------------------------ loads
      const uint32_t* fa = flags + (int64_t)tk.R * p.nblk;
      const uint32_t* fb = flags + (int64_t)Brow * p.nblk;
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
        asm volatile("fence.proxy.async;" ::: "memory");
        return true;
      };
      uint32_t kl = kc;
      for (int q = 0; q < nq && ok; ++q, ++kl) {
        const int k = k_of(q);
        ok = wait_tiles(k, tk.k1, tk.kind != TASK_D);
        if (ok && lane == 0) {
          for (int h = 0; h < 2 && ok; ++h) {
            if (!mbar_wait(empty(h), (kl & 1u) ^ 1u, abort_flag, p.budget)) { ok = false; break; }
            mbar_expect_tx(full(h), tk.kind == TASK_D ? OPER : SLOT);
            const uint32_t dst = data + h * SLOT;
#pragma unroll
            for (int z = 0; z < 3; ++z) {
              const int col = k * TB + h * 64;
              if (q == masked) tma_load_2d_local(dst + z * BOX, &tmY, z * TB + h * 64, (tk.R - p.nblk) * TB, full(h));
              else tma_load_2d_local(dst + z * BOX, &tmP, z * np + col, tk.R * TB, full(h));
              if (tk.kind != TASK_D) tma_load_2d_local(dst + OPER + z * BOX, &tmP, z * np + col, Brow * TB, full(h));
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
                tma_load_2d_local(data + SLOT + h * OPER + z * BOX, &tmP, z * np + tk.j * TB + h * 64, tk.j * TB, xfull);
          }
        }
      }
    } else if (warp == 1) {
      // ------------------------------------------------------------------ products
      if (lane == 0) {
        const uint32_t idesc = instr_desc(true);
        uint32_t kl = kc, cl = cc;
        for (int q = 0; q < nq && ok; ++q, ++kl, ++cl) {
          const uint32_t d = tmem + (cl & 1u) * 2 * TB;
          ok = mbar_wait(tempty(cl & 1u), ((cl >> 1) & 1u) ^ 1u, abort_flag, p.budget);
          for (int h = 0; h < 2 && ok; ++h) {
            ok = mbar_wait(full(h), kl & 1u, abort_flag, p.budget);
            if (!ok) break;
            tc_fence_after();
            const uint32_t a = data + h * SLOT, b = tk.kind == TASK_D ? a : a + OPER;
#pragma unroll
            for (int s = 0; s < 6; ++s)
#pragma unroll
              for (int k = 0; k < 4; ++k)
                mma(s > 0 ? d + TB : d, make_smem_desc(a + part_a(s) * BOX + k * 32, true, 0),
                    make_smem_desc(b + part_b(s) * BOX + k * 32, true, 0), idesc, h > 0 || s > 1 || k > 0 ? 1u : 0u);
            commit(empty(h));
          }
          if (ok) commit(tfull(cl & 1u));
        }
        if (tk.kind == TASK_T && ok) {
          const uint32_t d = tmem + (cl & 1u) * 2 * TB, idx = instr_desc(false);
          ok = mbar_wait(tempty(cl & 1u), ((cl >> 1) & 1u) ^ 1u, abort_flag, p.budget) &&
               mbar_wait(aready, xc & 1u, abort_flag, p.budget) && mbar_wait(xfull, xc & 1u, abort_flag, p.budget);
          if (ok) {
            tc_fence_after();
#pragma unroll 1
            for (int s = 0; s < 6; ++s) {
              const int pa = part_a(s), pb = part_b(s);
#pragma unroll
              for (int k = 0; k < 8; ++k)
                mma(s > 0 ? d + TB : d, make_smem_desc(data + (k >> 2) * OPER + pa * BOX + (k & 3) * 32, true, 0),
                    make_smem_desc(data + SLOT + pb * BOX + k * 16 * 128, false, OPER), idx, s > 1 || k > 0 ? 1u : 0u);
            }
            commit(tfull(cl & 1u));
          }
        }
        if (tk.kind != TASK_D) *next_ticket = (int)atomicAdd(p.flags, 1u);
      }
    } else if (warp >= EPI0) {
      // ------------------------------------------------------------------ the running value, and what leaves
      const int e = warp - EPI0, g = e >> 2, i = (warp & 3) * 32 + lane;   // row i, columns 32 g .. + 31 of the tile
      const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(g * 32);
      const int col0 = tk.j * TB + g * 32;
      float s[32];
      {
        const int64_t row = tk.R < p.nblk ? (int64_t)tk.R * TB + i : (int64_t)p.nn + (int64_t)(tk.R - p.nblk) * TB + i;
        const bool have = tk.kind != TASK_W && tk.R >= tk.j &&
                          (tk.R < p.nblk ? row < p.nn : row < (int64_t)p.nn + p.m);
        const float* src = p.A + row * p.lda + col0;
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
      // the next product of two tiles: this thread's 32 values
      auto sum_of = [&](uint32_t cl, float (&v)[32]) {
        const bool there = mbar_wait(tfull(cl & 1u), (cl >> 1) & 1u, abort_flag, p.budget);
        if (!__all_sync(0xffffffffu, there)) return false;
        tc_fence_after();
        const uint32_t at = taddr + (cl & 1u) * 2 * TB;
        uint32_t hi[32];
        tc_ld32(at, hi);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t lo[16];
          tc_ld16(at + TB + h * 16, lo);
          tc_wait_ld();
#pragma unroll
          for (int c = 0; c < 16; ++c) v[h * 16 + c] = __uint_as_float(hi[h * 16 + c]) + __uint_as_float(lo[c]);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) arrive(tempty(cl & 1u));
        return true;
      };
      uint32_t cl = cc;
      for (int q = 0; q < nq && ok; ++q, ++cl) {
        float r[32];
        ok = sum_of(cl, r);
        if (!ok) break;
        if (q == masked) {
          // the leading system's solution ends here
          const int64_t row = (int64_t)(tk.R - p.nblk) * TB + i;
          if (row < p.m) {
            float* dst = p.lead + row * p.ld_lead + col0;
#pragma unroll
            for (int c = 0; c < 32; ++c)
              if (col0 + c < p.lead_k) dst[c] = r[c] - s[c];
          }
        } else {
#pragma unroll
          for (int c = 0; c < 32; ++c) s[c] -= r[c];
        }
      }
      // the three parts of this thread's values as a K-major operand in the first slot (also the layout in which they leave)
      const uint32_t box_row = (uint32_t)(g >> 1) * OPER + (uint32_t)i * 128u;
      auto put = [&](float (&v)[32]) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          uint32_t o[4][3];
#pragma unroll
          for (int w = 0; w < 4; ++w) split3x2(v[8 * u + 2 * w], v[8 * u + 2 * w + 1], o[w]);
          const uint32_t at = box_row + ((((uint32_t)(g & 1) * 4u + u) ^ (uint32_t)(i & 7)) << 4);
#pragma unroll
          for (int z = 0; z < 3; ++z)
            *reinterpret_cast<uint4*>(data_ptr + at + z * BOX) = make_uint4(o[0][z], o[1][z], o[2][z], o[3][z]);
        }
        fence_async_smem();
      };
      auto leave = [&](const CUtensorMap* map, int part_cols, int col, int row) {     // one thread
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int z = 0; z < 3; ++z) tma_store_2d(map, z * part_cols + col + h * 64, row, data + h * OPER + z * BOX);
        bulk_commit();
        bulk_wait_all();
      };
      if (tk.kind == TASK_T) {
        // Rows of tiny values are brought to the order of one by a power of two: below 2^-110 the low parts would be cut off.
        float top = 0.f, back = 1.f;
#pragma unroll
        for (int c = 0; c < 32; ++c) top = fmaxf(top, fabsf(s[c]));
        if (epi_any(top > 0.f && top < 0x1p-80f)) {
          row_max[g * TB + i] = top;
          epi_sync();
          top = fmaxf(fmaxf(row_max[i], row_max[TB + i]), fmaxf(row_max[2 * TB + i], row_max[3 * TB + i]));
          if (top > 0.f && top < 0x1p-80f) {
            const float up = top < 0x1p-104f ? 0x1p104f : 0x1p80f;
            back = 1.f / up;
#pragma unroll
            for (int c = 0; c < 32; ++c) s[c] *= up;
          }
        }
        if (ok) {
          put(s);
          __syncwarp();
          if (lane == 0) arrive(aready);
          ok = sum_of(cl, s);
#pragma unroll
          for (int c = 0; c < 32; ++c) s[c] *= back;
        }
        if (ok) put(s);
        epi_sync();
        const bool all = *abort_flag == 0;
        if (all && threadIdx.x == EPI0 * 32) leave(&tmP, np, tk.j * TB, tk.R * TB);
        if (p.lead != nullptr && tk.R >= p.nblk && tk.j == (p.lead_k - 1) / TB) {
          // copy of the right-hand sides' last block of the leading system, zero beyond it
          epi_sync();
#pragma unroll
          for (int c = 0; c < 32; ++c) s[c] = col0 + c < p.lead_k ? s[c] : 0.f;
          put(s);
          epi_sync();
          if (all && threadIdx.x == EPI0 * 32) leave(&tmY, TB, 0, (tk.R - p.nblk) * TB);
        }
        if (all && threadIdx.x == EPI0 * 32) publish(flags + (int64_t)tk.R * p.nblk + tk.j);
      } else if (tk.kind == TASK_W) {
        const int64_t row = (int64_t)(tk.R - p.nblk) * TB + i;
        if (ok && row < p.m) {
          float* dst = p.W + row * p.ldw + col0;
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
      } else if (g <= (warp & 3)) {
        // the block on the diagonal, where DiagTiles expects its tiles
        const int nb = p.nn - tk.j * TB < TB ? p.nn - tk.j * TB : TB;
        float* dst = reinterpret_cast<float*>(data_ptr) + Diag::staged_at(i, g * 32);
#pragma unroll
        for (int c = 0; c < 32; ++c) {
          const int col = g * 32 + c;
          s[c] = col > i ? 0.f : i >= nb ? (col == i ? 1.f : 0.f) : s[c];
        }
#pragma unroll
        for (int c = 0; c < 32; c += 4) *reinterpret_cast<float4*>(dst + c) = make_float4(s[c], s[c + 1], s[c + 2], s[c + 3]);
      }
    }
    __syncwarp();            // (the block's barriers count whole warps)
    kc += (uint32_t)nq;
    cc += (uint32_t)nq + (tk.kind == TASK_T ? 1u : 0u);
    xc += tk.kind == TASK_T ? 1u : 0u;
    if (tk.kind == TASK_D) {
      __syncthreads();
      if (*abort_flag == 0) {                    // (set before the barrier only: the same for every thread)
        const int nb = p.nn - tk.j * TB < TB ? p.nn - tk.j * TB : TB;
        const PartsOut out{p.P + (int64_t)tk.j * TB * p.ldp + tk.j * TB, p.ldp, np};
        Diag::eliminate<true>(reinterpret_cast<float*>(data_ptr), dbars, dc & 1u, nullptr, 0, nb, out, (int64_t)tk.j * TB, p.status);
        __syncthreads();
        if (threadIdx.x == 0) {
          publish(flags + (int64_t)tk.j * p.nblk + tk.j);
          *next_ticket = (int)atomicAdd(p.flags, 1u);
        }
        ++dc;                                    // (a narrower block is the last one: nothing waits on its barriers again)
      }
    }
    fence_async_smem();
    __syncthreads();
    if (*abort_flag != 0) break;
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
  return kFlags0 + nblk * (nblk + mb);
}

sp_status solve_tc(const float* A, int64_t nn, int64_t m, int64_t lda, float* W, int64_t ldw, const SolveOneBufs& b,
                   float* lead, int64_t ld_lead, int64_t lead_k, int32_t* status_dev, cudaStream_t stream) {
  if (!solve_in_one(nn) || m < 1 || m > (1 << 24)) return SP_ERR_SHAPE;
  SolveParams p;
  memset(&p, 0, sizeof(p));
  p.A = A;
  p.lda = lda;
  p.nn = (int)nn;
  p.m = (int)m;
  p.nblk = (int)ceil_div(nn, (int64_t)TB);
  p.mb = (int)ceil_div(m, (int64_t)TB);
  const int64_t np = (int64_t)p.nblk * TB, rows = np + (int64_t)p.mb * TB;
  p.P = reinterpret_cast<__nv_bfloat16*>(b.P);
  p.ldp = 3 * np;
  p.W = W;
  p.ldw = ldw;
  p.lead = lead;
  p.ld_lead = ld_lead;
  p.lead_k = (int)lead_k;
  p.flags = b.flags;
  p.status = status_dev;
  p.skip = skip_flag();
  p.budget = wait_budget_cycles() > 0 ? wait_budget_cycles() : WAIT_BUDGET;
  CUtensorMap tmP, tmY;
  if (!make_map(&tmP, false, b.P, 3 * np, rows, 3 * np, 64, TB) ||
      !make_map(&tmY, false, b.Y, 3 * TB, (int64_t)p.mb * TB, 3 * TB, 64, TB))
    return SP_ERR_CUDA;
  static PerDeviceOnce attr_once;
  if (attr_once.run([] { return cudaFuncSetAttribute(solve_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM); }) !=
      cudaSuccess)
    return SP_ERR_CUDA;
  if (cudaMemsetAsync(b.flags, 0, solve_tc_flag_words(nn, m) * sizeof(uint32_t), stream) != cudaSuccess) return SP_ERR_CUDA;
  const int64_t tasks = (int64_t)p.nblk * (p.nblk + 2 * p.mb), sms = sm_count();
  count_launch();
  launch(solve_tc_kernel, (unsigned)(tasks < sms ? tasks : sms), THREADS, SMEM, stream, tmP, tmY, p);
  return cudaGetLastError() == cudaSuccess ? SP_OK : SP_ERR_CUDA;
}

}  // namespace sp
