// Elementwise and row-wise kernels of the multi-head-attention auxiliary updates (Appendix A, "Computation on
// Multi-Head Attention layers", Method 2; Algorithm 2, SparseLLM2).  The contractions around them (logits, P V, the
// gradient products) are batched tensor-core GEMMs issued by the host code in sp_api.cu; everything here is bound by
// memory bandwidth: one warp per row of a [pairs, T, T] tensor, 16-byte accesses where the layout allows.
#include "sp_common.cuh"

namespace sp {
namespace {

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

constexpr int kRowWarps = 8;

// A row of logits in registers, lane l holding the keys l, l + 32, ...: NV of them cover rows of up to 32 NV keys (NV = 0: any
// length, the row is read again instead).  The three passes over a row (maximum, sum, values) then cost one read and one
// exponential per entry (T = 128: 9.5 -> 5.3 us for the backward).  Above 256 keys the registers cost more warps than the
// rereads, which the L1 answers (T = 1024: 717 us in registers).
template <int NV>
struct RowVals {
  float e[NV > 0 ? NV : 1];      // exp(s - max) once sum() has run
  float mx;
  __device__ __forceinline__ float at(const float* row, int lane, int i) const {
    if constexpr (NV > 0) return e[i];
    else return __expf(row[lane + 32 * i] - mx);
  }
  // loads the row and returns 1 / sum_u exp(s_u - max)
  __device__ __forceinline__ float prepare(const float* row, int lane, int lim) {
    mx = -INFINITY;
    float sum = 0.f;
    if constexpr (NV > 0) {
#pragma unroll
      for (int i = 0; i < NV; ++i) e[i] = lane + 32 * i < lim ? row[lane + 32 * i] : -INFINITY;
#pragma unroll
      for (int i = 0; i < NV; ++i) mx = fmaxf(mx, e[i]);
      mx = warp_max(mx);
#pragma unroll
      for (int i = 0; i < NV; ++i)
        if (lane + 32 * i < lim) {
          e[i] = __expf(e[i] - mx);
          sum += e[i];
        }
    } else {
      for (int u = lane; u < lim; u += 32) mx = fmaxf(mx, row[u]);
      mx = warp_max(mx);
      for (int u = lane; u < lim; u += 32) sum += __expf(row[u] - mx);
    }
    return 1.f / warp_sum(sum);
  }
};
// f(u, i) for the entries u = lane + 32 i < n
template <int NV, typename F>
__device__ __forceinline__ void for_row(int lane, int n, F&& f) {
  if constexpr (NV > 0) {
#pragma unroll
    for (int i = 0; i < NV; ++i)
      if (lane + 32 * i < n) f(lane + 32 * i, i);
  } else {
    for (int u = lane, i = 0; u < n; u += 32, ++i) f(u, i);
  }
}

// S[row, :] <- softmax over the keys of the row (in place).  rows = pairs * T; row r belongs to query t = r % T; with
// `causal` keys u > t get probability 0.  Optional bf16 copy.
template <int NV>
__global__ void __launch_bounds__(kRowWarps * 32) softmax_rows_kernel(float* S, int64_t rows, int T,
                                                                      int causal, __nv_bfloat16* Sb,
                                                                      int64_t plane) {
  kernel_begin();
  const int lane = threadIdx.x & 31;
  const int64_t r = (int64_t)blockIdx.x * kRowWarps + (threadIdx.x >> 5);
  if (r >= rows) return;
  float* row = S + r * T;
  const int lim = causal ? (int)(r % T) + 1 : T;
  RowVals<NV> v;
  const float inv = v.prepare(row, lane, lim);
  for_row<NV>(lane, T, [&](int u, int i) {
    const float p = u < lim ? v.at(row, lane, i) * inv : 0.f;
    row[u] = p;
    if (Sb) {
      const __nv_bfloat16 hi = __float2bfloat16_rn(p);
      Sb[r * T + u] = hi;
      if (plane > 0) Sb[plane + r * T + u] = __float2bfloat16_rn(p - __bfloat162float(hi));
    }
  });
}

// Gradient step of Eq. (85) on the attention probabilities of every (sequence, head) pair:
//   P <- P - eta_b (-2 alpha G1 + 2 beta (P - Phi)),  G1 = R V^T from the preceding product, eta_b per pair.
// gridDim.y and blockDim.y walk the pairs, a thread takes V neighbouring entries (V = 4: 16-byte accesses).
template <int V>
__global__ void __launch_bounds__(256) p_update_kernel(float* P, const float* Phi, const float* G1, const float* eta,
                                                       int64_t per_pair, int64_t pairs, float alpha, float beta,
                                                       __nv_bfloat16* Pb, int64_t plane) {
  kernel_begin();
  struct __align__(4 * V) F { float v[V]; };
  struct __align__(2 * V) H { __nv_bfloat16 v[V]; };
  struct In { F p, ph, g1; };
  const int64_t step = strip_rows();
  for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * V; i < per_pair;
       i += (int64_t)gridDim.x * blockDim.x * V) {
    const auto load = [&](int64_t b) {
      const int64_t e = b * per_pair + i;
      return In{*reinterpret_cast<const F*>(P + e), *reinterpret_cast<const F*>(Phi + e), *reinterpret_cast<const F*>(G1 + e)};
    };
    const auto finish = [&](int64_t b, const In& in, float et) {
      const int64_t e = b * per_pair + i;
      F pn;
      H hi, lo;
#pragma unroll
      for (int q = 0; q < V; ++q) {
        const float g = -2.f * alpha * in.g1.v[q] + 2.f * beta * (in.p.v[q] - in.ph.v[q]);
        pn.v[q] = in.p.v[q] - et * g;
        hi.v[q] = __float2bfloat16_rn(pn.v[q]);
        lo.v[q] = __float2bfloat16_rn(pn.v[q] - __bfloat162float(hi.v[q]));
      }
      *reinterpret_cast<F*>(P + e) = pn;
      if (Pb) {
        *reinterpret_cast<H*>(Pb + e) = hi;
        if (plane > 0) *reinterpret_cast<H*>(Pb + plane + e) = lo;
      }
    };
    // four pairs at a time: their loads are on their way before the first store
    for (int64_t b = strip_row(); b < pairs; b += 4 * step) {
      In x[4];
      float et[4];
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (b + q * step < pairs) {
          x[q] = load(b + q * step);
          et[q] = eta[b + q * step];
        }
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (b + q * step < pairs) finish(b + q * step, x[q], et[q]);
    }
  }
}

// Softmax and its backward for the softmax term of Eq. (87), one warp per row of logits S:
//   Phi = softmax(S),  E = Phi - P,  dS = 2 beta Phi (E - sum_u E Phi)  -> as bf16 to dSb, or (dSb == nullptr) in place.
// Beyond the causal limit zeros are written up to the end of the row's block of `tail` keys.
template <int NV>
__global__ void __launch_bounds__(kRowWarps * 32) softmax_backward_rows_kernel(float* S, const float* P,
                                                                               int64_t rows, int T, int causal, int tail,
                                                                               float beta,
                                                                               __nv_bfloat16* dSb) {
  kernel_begin();
  const int lane = threadIdx.x & 31;
  const int64_t r = (int64_t)blockIdx.x * kRowWarps + (threadIdx.x >> 5);
  if (r >= rows) return;
  float* row = S + r * T;
  const float* prow = P + r * T;
  const int lim = causal ? (int)(r % T) + 1 : T;
  RowVals<NV> v;
  const float inv = v.prepare(row, lane, lim);
  float p[NV > 0 ? NV : 1];
  float dot = 0.f;        // sum_u E Phi (Phi = 0 beyond the causal limit)
  for_row<NV>(lane, lim, [&](int u, int i) {
    const float ph = v.at(row, lane, i) * inv, pu = prow[u];
    if constexpr (NV > 0) p[i] = pu;
    dot = fmaf(ph - pu, ph, dot);
  });
  dot = warp_sum(dot);
  const auto put = [&](int u, float g) {
    if (dSb) dSb[r * T + u] = __float2bfloat16_rn(g);
    else row[u] = g;
  };
  const int end = causal && tail < T ? min(T, ((lim - 1) / tail + 1) * tail) : T;
  if constexpr (NV > 0) {
    for_row<NV>(lane, end, [&](int u, int i) {
      const float ph = u < lim ? v.at(row, lane, i) * inv : 0.f;
      put(u, u < lim ? 2.f * beta * ph * (ph - p[i] - dot) : 0.f);
    });
  } else {
    const auto value = [&](int u) {
      const float ph = __expf(row[u] - v.mx) * inv;
      return 2.f * beta * ph * (ph - prow[u] - dot);
    };
    int u = lane;
    for (; u + 96 < lim; u += 128) {       // four entries at a time: their loads before the first store
      float g[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) g[q] = value(u + 32 * q);
#pragma unroll
      for (int q = 0; q < 4; ++q) put(u + 32 * q, g[q]);
    }
    for (; u < lim; u += 32) put(u, value(u));
    for (; u < end; u += 32) put(u, 0.f);
  }
}

// Sum of squares of the [T, d_h] slice of every (sequence, head) pair of up to two token-major [tokens, d] tensors;
// one block per pair, fixed summation order.  out[b] = sum x^2 (+ sum y^2), b = seq * H + head.
__global__ void __launch_bounds__(256) pair_sumsq_kernel(const float* x, const float* y,
                                                         int64_t ld, int T, int d_h, int H, double* out) {
  kernel_begin();
  __shared__ double sm[256];
  const int b = blockIdx.x, seq = b / H, head = b % H;
  const int64_t base = (int64_t)seq * T * ld + (int64_t)head * d_h;
  double acc = 0.0;
  const int total = T * d_h;
  // eight entries in flight, added in order; a head width that divides 256 keeps a thread in its column
  const bool one_col = 256 % d_h == 0;
  const int64_t o0 = base + (int64_t)(threadIdx.x / d_h) * ld + threadIdx.x % d_h, step = (int64_t)(256 / d_h) * ld;
  for (int e0 = threadIdx.x, j = 0; e0 < total; e0 += 8 * 256, j += 8) {
    float v[8], w[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int e = e0 + q * 256;
      const int64_t o = one_col ? o0 + (j + q) * step : base + (int64_t)(e / d_h) * ld + (e % d_h);
      v[q] = e < total ? x[o] : 0.f;
      w[q] = y && e < total ? y[o] : 0.f;
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      acc += (double)v[q] * v[q];
      if (y) acc += (double)w[q] * w[q];
    }
  }
  sm[threadIdx.x] = acc;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) sm[threadIdx.x] += sm[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[b] = sm[0];
}

// Step sizes from the sums above: mode 0 (Eq. 85): eta = 1 / (2 (alpha s + beta));
// mode 1 (Eq. 87): eta = eta_z / (2 alpha + beta s / d_h).
__global__ void step_size_kernel(const double* s, int n, int mode, double alpha, double beta, double eta_z,
                                 int d_h, float* eta) {
  kernel_begin();
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= n) return;
  eta[b] = mode == 0 ? (float)(1.0 / (2.0 * (alpha * s[b] + beta)))
                     : (float)(eta_z / (2.0 * alpha + beta * s[b] / (double)d_h));
}

// Gradient step of Eq. (87) on the projection outputs, token-major [tokens, d]:
//   Z <- Z - eta_b (G + 2 alpha (Z - Tg)) for Z in {Zq, Zk}, b = (token / T) * H + column / d_h;
// optional bf16 hi / lo planes of the new values (operands of the next logits product).  A thread takes V neighbouring
// columns of one head (V = 4: 16-byte accesses).
template <int V>
__global__ void __launch_bounds__(256) z_update_kernel(float* Zq, float* Zk, const float* Gq, const float* Gk,
                                                       const float* Tq, const float* Tk, const float* eta, int64_t tokens, int d, int T,
                                                       int d_h, float alpha, __nv_bfloat16* Zqs,
                                                       __nv_bfloat16* Zks, int64_t plane) {
  kernel_begin();
  struct __align__(4 * V) F { float v[V]; };
  struct __align__(2 * V) B { __nv_bfloat16 v[V]; };
  const int H = d / d_h, c = (int)(blockIdx.x * blockDim.x + threadIdx.x) * V;
  if (c >= d) return;
  const int head = c / d_h;
  for (int64_t tok = strip_row(); tok < tokens; tok += strip_rows()) {
    const int64_t e = tok * d + c;
    const float et = eta[(tok / T) * H + head];
    const auto in = [&](const float* p) { return *reinterpret_cast<const F*>(p + e); };
    const auto step = [&](const F& z, const F& g, const F& t, float* Z, __nv_bfloat16* S) {
      F n;
      B hi, lo;
#pragma unroll
      for (int q = 0; q < V; ++q) {
        n.v[q] = z.v[q] - et * (g.v[q] + 2.f * alpha * (z.v[q] - t.v[q]));
        hi.v[q] = __float2bfloat16_rn(n.v[q]);
        lo.v[q] = __float2bfloat16_rn(n.v[q] - __bfloat162float(hi.v[q]));
      }
      *reinterpret_cast<F*>(Z + e) = n;
      if (S) {
        *reinterpret_cast<B*>(S + e) = hi;
        *reinterpret_cast<B*>(S + plane + e) = lo;
      }
    };
    const F zq = in(Zq), gq = in(Gq), tq = in(Tq), zk = in(Zk), gk = in(Gk), tk = in(Tk);   // (all on their way before a store)
    step(zq, gq, tq, Zq, Zqs);
    step(zk, gk, tk, Zk, Zks);
  }
}

// hi / lo bf16 planes of a dense fp32 tensor of `total` elements: dst[e] = bf16(x), dst[plane + e] = bf16(x - hi).
__global__ void __launch_bounds__(256) split_planes_kernel(const float* x, int64_t total,
                                                           __nv_bfloat16* dst, int64_t plane) {
  kernel_begin();
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  for (int64_t e0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e0 < total; e0 += 4 * step) {
    float v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = e0 + q * step < total ? x[e0 + q * step] : 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int64_t e = e0 + q * step;
      if (e >= total) break;
      const __nv_bfloat16 hi = __float2bfloat16_rn(v[q]);
      dst[e] = hi;
      if (plane > 0) dst[plane + e] = __float2bfloat16_rn(v[q] - __bfloat162float(hi));
    }
  }
}

// bf16 hi / lo planes of the selected heads' [T, T] blocks: grid (pieces of a block, slots, sequences), 16-byte reads.
__global__ void __launch_bounds__(256) split_heads_kernel(const float* P, int64_t n_seq, int64_t H, int64_t per_pair,
                                                          const __grid_constant__ HeadList heads,
                                                          __nv_bfloat16* dst, int64_t plane) {
  kernel_begin();
  struct __align__(8) B { __nv_bfloat162 v[2]; };
  for (int64_t seq = blockIdx.z; seq < n_seq; seq += gridDim.z) {
    const float* src = P + (seq * H + heads.h[blockIdx.y]) * per_pair;
    __nv_bfloat16* out = dst + (seq * gridDim.y + blockIdx.y) * per_pair;
    const int64_t step = (int64_t)gridDim.x * 1024;
    for (int64_t e0 = ((int64_t)blockIdx.x * 256 + threadIdx.x) * 4; e0 < per_pair; e0 += 4 * step) {
      float4 x[4];
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (e0 + q * step < per_pair) x[q] = *reinterpret_cast<const float4*>(src + e0 + q * step);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int64_t e = e0 + q * step;
        if (e >= per_pair) break;
        B hi, lo;
        hi.v[0] = __floats2bfloat162_rn(x[q].x, x[q].y);
        hi.v[1] = __floats2bfloat162_rn(x[q].z, x[q].w);
        lo.v[0] = __floats2bfloat162_rn(x[q].x - __low2float(hi.v[0]), x[q].y - __high2float(hi.v[0]));
        lo.v[1] = __floats2bfloat162_rn(x[q].z - __low2float(hi.v[1]), x[q].w - __high2float(hi.v[1]));
        *reinterpret_cast<B*>(out + e) = hi;
        *reinterpret_cast<B*>(out + plane + e) = lo;
      }
    }
  }
}

// The selected heads' columns of a token-major tensor as hi / lo parts: grid (tokens, slots)
__global__ void split_head_cols_kernel(const float* A, int64_t tokens, int64_t d, int d_h,
                                       const __grid_constant__ HeadList heads, __nv_bfloat16* dst, int64_t ld,
                                       int64_t lo_off) {
  kernel_begin();
  const int per_block = blockDim.x / d_h > 0 ? blockDim.x / d_h : 1;
  const int64_t t0 = (int64_t)blockIdx.x * per_block;
  for (int e = threadIdx.x; e < per_block * d_h; e += blockDim.x) {
    const int64_t t = t0 + e / d_h;
    const int c = e % d_h;
    if (t >= tokens) continue;
    const float v = A[t * d + (int64_t)heads.h[blockIdx.y] * d_h + c];
    const __nv_bfloat16 hi = __float2bfloat16_rn(v);
    __nv_bfloat16* out = dst + ((int64_t)blockIdx.y * tokens + t) * ld + c;
    out[0] = hi;
    out[lo_off] = __float2bfloat16_rn(v - __bfloat162float(hi));
  }
}

__global__ void __launch_bounds__(1024) add_ridge_batched_kernel(float* G, int64_t bs, int64_t n, double rho,
                                                                 int rel) {
  kernel_begin();
  __shared__ double sm[32];
  G += (int64_t)blockIdx.x * bs;
  double s = 0.0;
  if (rel)
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) s += (double)G[i * n + i];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sm[w];
    sm[0] = rel ? rho * t / (double)n : rho;
  }
  __syncthreads();
  const double r = sm[0];
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) G[i * n + i] = (float)((double)G[i * n + i] + r);
}

__global__ void __launch_bounds__(256) place_heads_kernel(const float* src, int64_t bs, int64_t d,
                                                          const __grid_constant__ HeadList heads, float* W,
                                                          int64_t ldw) {
  kernel_begin();
  const float* in = src + (int64_t)blockIdx.y * bs + (int64_t)blockIdx.x * d;
  float* out = W + ((int64_t)heads.h[blockIdx.y] * gridDim.x + blockIdx.x) * ldw;
  for (int64_t c = threadIdx.x; c < d; c += 1024) {
    float v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = c + 256 * q < d ? in[c + 256 * q] : 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (c + 256 * q < d) out[c + 256 * q] = v[q];
  }
}

template <typename T>
__global__ void set_identity_kernel(T* A, int64_t n, int64_t ld) {
  kernel_begin();
  const int64_t total = n * n;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / n, j = e % n;
    A[i * ld + j] = i == j ? 1.f : 0.f;
  }
}

unsigned grid_1d(int64_t total, int threads) {
  int64_t b = (total + threads - 1) / threads;
  const int64_t cap = (int64_t)sm_count() * 16;
  if (b > cap) b = cap;
  if (b < 1) b = 1;
  return (unsigned)b;
}

}  // namespace

cudaError_t mha_softmax_rows(float* S, int64_t pairs, int T, bool causal, void* Sb, int64_t plane,
                             cudaStream_t stream) {
  const int64_t rows = pairs * T;
  if (rows == 0) return cudaSuccess;
  ProfScope prof(PK_ELEMENTWISE, 0.0, (double)rows * T * 8.0, stream);
  count_launch();
  const unsigned grid = (unsigned)ceil_div(rows, (int64_t)kRowWarps);
  const auto run = [&](auto kernel) {
    launch(kernel, grid, kRowWarps * 32, 0, stream, S, rows, T, causal ? 1 : 0, reinterpret_cast<__nv_bfloat16*>(Sb), plane);
  };
  if (T <= 128) run(softmax_rows_kernel<4>);
  else if (T <= 256) run(softmax_rows_kernel<8>);
  else run(softmax_rows_kernel<0>);
  return cudaGetLastError();
}

cudaError_t mha_p_update(float* P, const float* Phi, const float* G1, const float* eta, int64_t pairs, int T,
                         double alpha, double beta, void* Pb, int64_t plane, cudaStream_t stream) {
  const int64_t total = pairs * T * T;
  if (total == 0) return cudaSuccess;
  ProfScope prof(PK_ELEMENTWISE, 0.0, (double)total * 16.0, stream);
  count_launch();
  const int64_t per_pair = (int64_t)T * T;
  const auto al = [](const void* p, uintptr_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; };
  const bool vec = per_pair % 4 == 0 && plane % 4 == 0 && al(P, 16) && al(Phi, 16) && al(G1, 16) && al(Pb, 8);
  const int V = vec ? 4 : 1;
  const dim3 block = strip_block(ceil_div(per_pair, (int64_t)V));
  int64_t gx = ceil_div(per_pair, (int64_t)block.x * V), gy = ceil_div(pairs, (int64_t)block.y);
  if (gy > 65535) gy = 65535;
  const int64_t cap = (int64_t)sm_count() * 16;
  if (gx > cap) gx = cap;
  if (gx * gy > cap) gy = cap / gx > 0 ? cap / gx : 1;
  const dim3 grid((unsigned)gx, (unsigned)gy);
  __nv_bfloat16* pb = reinterpret_cast<__nv_bfloat16*>(Pb);
  if (vec) launch(p_update_kernel<4>, grid, block, 0, stream, P, Phi, G1, eta, per_pair, pairs, (float)alpha, (float)beta, pb, plane);
  else launch(p_update_kernel<1>, grid, block, 0, stream, P, Phi, G1, eta, per_pair, pairs, (float)alpha, (float)beta, pb, plane);
  return cudaGetLastError();
}

cudaError_t mha_softmax_backward_rows(float* S, const float* P, int64_t pairs, int T, bool causal, int tail, double beta,
                                      void* dSb, cudaStream_t stream) {
  const int64_t rows = pairs * T;
  if (rows == 0) return cudaSuccess;
  ProfScope prof(PK_ELEMENTWISE, 0.0, (double)rows * T * 12.0, stream);
  count_launch();
  const unsigned grid = (unsigned)ceil_div(rows, (int64_t)kRowWarps);
  const auto run = [&](auto kernel) {
    launch(kernel, grid, kRowWarps * 32, 0, stream, S, P, rows, T, causal ? 1 : 0, tail, (float)beta,
                                                reinterpret_cast<__nv_bfloat16*>(dSb));
  };
  if (T <= 128) run(softmax_backward_rows_kernel<4>);
  else if (T <= 256) run(softmax_backward_rows_kernel<8>);
  else run(softmax_backward_rows_kernel<0>);
  return cudaGetLastError();
}

cudaError_t mha_step_sizes(const float* x, const float* y, int64_t ld, int64_t n_seq, int T, int d_h, int H, int mode,
                           double alpha, double beta, double eta_z, double* sums, float* eta, cudaStream_t stream) {
  const int n = (int)(n_seq * H);
  if (n == 0) return cudaSuccess;
  ProfScope prof(PK_ELEMENTWISE, 0.0, 0.0, stream);
  count_launch(2);
  launch(pair_sumsq_kernel, n, 256, 0, stream, x, y, ld, T, d_h, H, sums);
  launch(step_size_kernel, (n + 255) / 256, 256, 0, stream, sums, n, mode, alpha, beta, eta_z, d_h, eta);
  return cudaGetLastError();
}

cudaError_t mha_z_update(float* Zq, float* Zk, const float* Gq, const float* Gk, const float* Tq, const float* Tk,
                         const float* eta, int64_t tokens, int d, int T, int d_h, double alpha, void* Zqs, void* Zks,
                         int64_t plane, cudaStream_t stream) {
  const int64_t total = tokens * d;
  if (total == 0) return cudaSuccess;
  ProfScope prof(PK_ELEMENTWISE, 0.0, (double)total * 32.0, stream);
  count_launch();
  const auto al = [](const void* p, uintptr_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; };
  const bool vec = d_h % 4 == 0 && plane % 4 == 0 && al(Zq, 16) && al(Zk, 16) && al(Gq, 16) && al(Gk, 16) && al(Tq, 16) &&
                   al(Tk, 16) && al(Zqs, 8) && al(Zks, 8);
  const int V = vec ? 4 : 1;
  const dim3 block = strip_block(ceil_div(d, V));
  const int64_t gx = ceil_div(d, (int)block.x * V), row_blocks = ceil_div(tokens, (int64_t)block.y);
  int64_t gy = ceil_div((int64_t)sm_count() * 8, gx);
  if (gy > row_blocks) gy = row_blocks;
  const auto run = [&](auto kernel) {
    launch(kernel, dim3((unsigned)gx, (unsigned)gy), block, 0, stream, Zq, Zk, Gq, Gk, Tq, Tk, eta, tokens, d, T, d_h, (float)alpha,
                                                                 reinterpret_cast<__nv_bfloat16*>(Zqs),
                                                                 reinterpret_cast<__nv_bfloat16*>(Zks), plane);
  };
  if (vec) run(z_update_kernel<4>);
  else run(z_update_kernel<1>);
  return cudaGetLastError();
}

template <typename T>
cudaError_t set_identity(T* A, int64_t n, int64_t ld, cudaStream_t stream) {
  if (n == 0) return cudaSuccess;
  count_launch();
  launch(set_identity_kernel<T>, grid_1d(n * n, 256), 256, 0, stream, A, n, ld);
  return cudaGetLastError();
}
template cudaError_t set_identity<float>(float*, int64_t, int64_t, cudaStream_t);
template cudaError_t set_identity<double>(double*, int64_t, int64_t, cudaStream_t);

cudaError_t split_planes(const float* x, int64_t total, void* dst, int64_t plane, cudaStream_t stream) {
  if (total == 0) return cudaSuccess;
  ProfScope prof(PK_ELEMENTWISE, 0.0, (double)total * 8.0, stream);
  count_launch();
  launch(split_planes_kernel, grid_1d(total, 256), 256, 0, stream, x, total, reinterpret_cast<__nv_bfloat16*>(dst), plane);
  return cudaGetLastError();
}

cudaError_t mha_split_heads(const float* P, int64_t n_seq, int64_t H, int64_t per_pair, const HeadList& heads, void* dst,
                            int64_t plane, cudaStream_t stream) {
  if (n_seq * heads.n * per_pair == 0) return cudaSuccess;
  if (per_pair % 4 != 0) return cudaErrorInvalidValue;
  ProfScope prof(PK_ELEMENTWISE, 0.0, (double)n_seq * heads.n * per_pair * 8.0, stream);
  count_launch();
  int64_t gx = ceil_div(per_pair, (int64_t)1024);
  const int64_t cap = ceil_div((int64_t)sm_count() * 32, n_seq * heads.n);
  if (gx > cap) gx = cap;
  const unsigned gz = (unsigned)(n_seq < 65535 ? n_seq : 65535);
  launch(split_heads_kernel, dim3((unsigned)gx, (unsigned)heads.n, gz), 256, 0, stream, 
      P, n_seq, H, per_pair, heads, reinterpret_cast<__nv_bfloat16*>(dst), plane);
  return cudaGetLastError();
}

cudaError_t mha_split_head_cols(const float* A, int64_t tokens, int64_t d, int64_t d_h, const HeadList& heads, void* dst,
                                int64_t ld, int64_t lo_off, cudaStream_t stream) {
  if (tokens * heads.n == 0) return cudaSuccess;
  ProfScope prof(PK_ELEMENTWISE, 0.0, (double)tokens * heads.n * d_h * 8.0, stream);
  count_launch();
  const int64_t per_block = 256 / d_h > 0 ? 256 / d_h : 1;
  launch(split_head_cols_kernel, dim3((unsigned)ceil_div(tokens, per_block), (unsigned)heads.n), 256, 0, stream, 
      A, tokens, d, (int)d_h, heads, reinterpret_cast<__nv_bfloat16*>(dst), ld, lo_off);
  return cudaGetLastError();
}

cudaError_t add_ridge_batched(float* G, int64_t bs, int64_t n, int batch, double rho, bool rel, cudaStream_t stream) {
  if (n == 0 || batch == 0) return cudaSuccess;
  ProfScope prof(PK_ELEMENTWISE, 0.0, 0.0, stream);
  count_launch();
  launch(add_ridge_batched_kernel, (unsigned)batch, 1024, 0, stream, G, bs, n, rho, rel ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t mha_place_heads(const float* src, int64_t bs, int64_t d_h, int64_t d, const HeadList& heads, float* W,
                            int64_t ldw, cudaStream_t stream) {
  if (heads.n == 0 || d_h == 0) return cudaSuccess;
  ProfScope prof(PK_ELEMENTWISE, 0.0, (double)heads.n * d_h * d * 8.0, stream);
  count_launch();
  launch(place_heads_kernel, dim3((unsigned)d_h, (unsigned)heads.n), 256, 0, stream, src, bs, d, heads, W, ldw);
  return cudaGetLastError();
}

}  // namespace sp
