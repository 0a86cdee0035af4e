// Dense-row forward on CUDA cores: one CTA per query row, every visible key visited, with a scratch of one score row per CTA.
// It is what entmax_attn_fwd_static runs (its fixed scratch holds no more).  Also holds the prologue kernel (ASEntmax scale
// table, cleared counters), the scale gradient kernel and the gradient store kernel.
//
// Threshold solve: f(tau) = sum_j [y_j - tau]_+^e - 1 with y = (alpha-1) s and e = 1/(alpha-1) >= 1 is
// convex and decreasing (Eq. 1 of the paper with the sum-to-one condition).  Newton steps started at
// the lower end of the paper's bracket, tau0 = y_max - 1 (App. A), therefore never overshoot the root
// and converge monotonically; no bisection safeguard is needed.
#include "common.cuh"

namespace entmax {

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kMaxNewton = 400;

__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}
__device__ __forceinline__ float warp_max(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
  return x;
}

// red: kWarps*2 floats of shared memory.  Every thread gets both block sums.
__device__ __forceinline__ float2 block_sum2(float a, float b, float* red) {
  a = warp_sum(a);
  b = warp_sum(b);
  int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) { red[w] = a; red[kWarps + w] = b; }
  __syncthreads();
  float ra = 0.f, rb = 0.f;
#pragma unroll
  for (int i = 0; i < kWarps; ++i) { ra += red[i]; rb += red[kWarps + i]; }
  return make_float2(ra, rb);
}
__device__ __forceinline__ float block_max(float a, float* red) {
  a = warp_max(a);
  int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = a;
  __syncthreads();
  float r = red[0];
#pragma unroll
  for (int i = 1; i < kWarps; ++i) r = fmaxf(r, red[i]);
  return r;
}

struct RowCtx {
  int grow, bh, b, h, i, nv;
  float c, a, g;
  float slope;  // ALiBi slope in dot-product units (m_h / sm_scale), 0 without ALiBi
  size_t base;  // element offset of (b, h, 0, 0)
};

__device__ __forceinline__ RowCtx make_row(const Problem& p, const float* scale, int grow) {
  RowCtx r;
  r.grow = grow;
  r.bh = grow / p.N;
  r.i = grow - r.bh * p.N;
  r.b = r.bh / p.H;
  r.h = r.bh - r.b * p.H;
  r.nv = p.causal ? r.i + 1 : p.N;
  r.c = scale[(size_t)r.b * p.scale_sb + (size_t)r.h * p.N + r.i];
  r.g = r.c * p.sm_scale;
  r.a = (p.alpha - 1.0f) * r.g;
  r.slope = p.alibi ? p.alibi[r.h] / p.sm_scale : 0.f;
  r.base = (size_t)r.b * p.sb + (size_t)r.h * p.sh;
  return r;
}

// y_j = a_i <q_i,k_j> for every visible key into ybuf; returns the row maximum (block-wide).
template <typename T, int D>
__device__ __forceinline__ float score_pass(const Problem& p, const RowCtx& r, const T* k, const float (&qs)[D / 32],
                                            float* ybuf, float* red) {
  constexpr int PER = D / 32;
  int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  float wmax = -INFINITY;
  for (int j = w; j < r.nv; j += kWarps) {
    float ks[PER];
    load_slice<PER>(k + r.base + (size_t)j * p.sn + l * PER, ks);
    float dot = 0.f;
#pragma unroll
    for (int t = 0; t < PER; ++t) dot = fmaf(qs[t], ks[t], dot);
    dot = warp_sum(dot);
    // ALiBi: the logit is sm_scale * (dot - slope |i - j|) with slope = m_h / sm_scale
    if (r.slope != 0.f) dot -= r.slope * fabsf((float)(j - r.i));
    float y = r.a * dot;
    if (l == 0) ybuf[j] = y;
    wmax = fmaxf(wmax, y);
  }
  return block_max(wmax, red);
}

__device__ __forceinline__ float newton_tau(const Problem& p, const float* ybuf, int nv, float ymax, float* red) {
  TauIter st = tau_iter_start(ymax);
  for (int it = 0; it < kMaxNewton; ++it) {
    float s0 = 0.f, s1 = 0.f;
    for (int j = threadIdx.x; j < nv; j += kThreads) {
      float y = ybuf[j] - st.tau;
      if (y > 0.f) {
        float ye, ye1;
        pow_pair(y, p.expo_class, p.expo, ye, ye1);
        s0 += ye;
        s1 += ye1;
      }
    }
    float2 s = block_sum2(s0, s1, red);
    if (!tau_iter_update(st, s.x, s.y, p.expo_class, p.expo, 1e-7f)) break;
  }
  return st.tau;
}

template <typename T, int D>
__global__ void __launch_bounds__(kThreads) dense_fwd_kernel(Problem p, const T* __restrict__ q, const T* __restrict__ k,
                                                             const T* __restrict__ v, const float* __restrict__ scale,
                                                             T* __restrict__ o, float* __restrict__ tau_out,
                                                             float* scratch, size_t scratch_floats) {
  pdl_begin();
  constexpr int PER = D / 32;
  __shared__ float red[2 * kWarps];
  __shared__ float opart[kWarps][D];
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  const int total = p.B * p.H * p.N;
  float* ybuf = scratch + (size_t)blockIdx.x * scratch_floats;
  for (int ridx = blockIdx.x; ridx < total; ridx += gridDim.x) {
    const RowCtx r = make_row(p, scale, ridx);
    float qs[PER];
    load_slice<PER>(q + r.base + (size_t)r.i * p.sn + l * PER, qs);
    const float ymax = score_pass<T, D>(p, r, k, qs, ybuf, red);
    const float tau = newton_tau(p, ybuf, r.nv, ymax, red);
    float acc[PER];
#pragma unroll
    for (int t = 0; t < PER; ++t) acc[t] = 0.f;
    for (int j = w; j < r.nv; j += kWarps) {
      const float y = ybuf[j] - tau;
      if (y > 0.f) {
        float pe, pe1;
        pow_pair(y, p.expo_class, p.expo, pe, pe1);
        float vs[PER];
        load_slice<PER>(v + r.base + (size_t)j * p.sn + l * PER, vs);
#pragma unroll
        for (int t = 0; t < PER; ++t) acc[t] = fmaf(pe, vs[t], acc[t]);
      }
    }
#pragma unroll
    for (int t = 0; t < PER; ++t) opart[w][l * PER + t] = acc[t];
    __syncthreads();
    if (threadIdx.x < D / PER) {
      float out[PER];
#pragma unroll
      for (int t = 0; t < PER; ++t) {
        float s = 0.f;
#pragma unroll
        for (int ww = 0; ww < kWarps; ++ww) s += opart[ww][threadIdx.x * PER + t];
        out[t] = s;
      }
      store_slice<PER>(o + r.base + (size_t)r.i * p.sn + threadIdx.x * PER, out);
    }
    if (threadIdx.x == 0) tau_out[r.grow] = tau;
    __syncthreads();
  }
}

// dbeta_h, dgamma_h, ddelta_h from the per-row scale gradients: c_i = delta + beta L^gamma with L = ln n_i
// (rows with n_i = 1 have c_i = delta), so d/ddelta = 1, d/dbeta = L^gamma, d/dgamma = beta L^gamma ln L.
// fp64 throughout.  What bounds it is the fp64 logarithms and exponentials (one L^gamma per head and position, after the
// batch has been summed), so the positions of a head are spread over as many CTAs as it takes to reach every SM; each
// leaves three partial sums, and the CTA that finishes last adds them in a fixed order (reproducible).  One CTA per head
// and a pow per (batch, head, position) took 178 us at 16 heads x 32768 and 350 us at 8 x 65536; this takes 14 and 18 us.
constexpr int kScaleGradThreads = 256;
__device__ __forceinline__ double block_sum_fp64(double x, double* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
  __syncthreads();
  double r = 0.0;
#pragma unroll
  for (int w = 0; w < kScaleGradThreads / 32; ++w) r += red[w];
  return r;
}
__global__ void __launch_bounds__(kScaleGradThreads) scale_grad_kernel(Problem p, const float* __restrict__ beta,
                                                                       const float* __restrict__ gamma,
                                                                       const float* __restrict__ dc_rows,
                                                                       double* __restrict__ partial, int32_t* counter,
                                                                       float* __restrict__ dbeta,
                                                                       float* __restrict__ dgamma,
                                                                       float* __restrict__ ddelta) {
  pdl_begin();
  __shared__ double red[kScaleGradThreads / 32];
  __shared__ int last;
  const int h = blockIdx.x;                        // (heads along x: the other dimensions of a grid end at 65535)
  const double b = beta[h], g = gamma[h];
  double sb = 0.0, sg = 0.0, sd = 0.0;
  for (int i = blockIdx.y * kScaleGradThreads + threadIdx.x; i < p.N; i += gridDim.y * kScaleGradThreads) {
    double dc = 0.0;
    for (int bb = 0; bb < p.B; ++bb) dc += dc_rows[((size_t)bb * p.H + h) * p.N + i];
    const int n = (p.n_mode || !p.causal) ? p.N : i + 1;
    sd += dc;
    if (n > 1) {
      const double lnL = log(log((double)n));
      const double t = dc * exp(g * lnL);
      sb += t;
      sg += t * b * lnL;
    }
  }
  sb = block_sum_fp64(sb, red);
  sg = block_sum_fp64(sg, red);
  sd = block_sum_fp64(sd, red);
  if (threadIdx.x == 0) {
    double* mine = partial + 3 * ((size_t)h * gridDim.y + blockIdx.y);
    mine[0] = sb;
    mine[1] = sg;
    mine[2] = sd;
    __threadfence();
    last = atomicAdd(counter, 1) == (int)(gridDim.x * gridDim.y) - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int t = threadIdx.x; t < 3 * p.H; t += kScaleGradThreads) {
    const int hh = t / 3, which = t - 3 * hh;
    double sum = 0.0;
    for (unsigned c = 0; c < gridDim.y; ++c) sum += __ldcg(partial + 3 * ((size_t)hh * gridDim.y + c) + which);
    (which == 0 ? dbeta : which == 1 ? dgamma : ddelta)[hh] = (float)sum;
  }
}

// c_i = delta_h + beta_h (ln n_i)^gamma_h in fp64, rounded once to fp32 (Eq. "asentmax").  A thread takes one position of
// kScaleHeads heads: the two logarithms do not depend on the head, one exponential per head is left (a pow per entry took
// 9.3 us at 16 heads x 32768, this 5.4 us).  The same launch clears the call's counters and flags (`clear`, n_clear words),
// which used to be memsets of their own: about 2 us of stream time each.
constexpr int kScaleHeads = 4;
__global__ void __launch_bounds__(256) prologue_kernel(Problem p, const float* __restrict__ beta,
                                                       const float* __restrict__ gamma, const float* __restrict__ delta,
                                                       float* __restrict__ scale, int32_t* __restrict__ clear, int n_clear,
                                                       int32_t* __restrict__ status) {
  pdl_begin();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (blockIdx.y == 0)
    for (int t = i; t < n_clear; t += gridDim.x * blockDim.x) clear[t] = 0;
  if (!scale || i >= p.N) return;
  const int n = (p.n_mode || !p.causal) ? p.N : i + 1;
  const double lnL = p.has_scale && n > 1 ? log(log((double)n)) : 0.0;
  for (int h0 = blockIdx.y * kScaleHeads; h0 < p.H; h0 += gridDim.y * kScaleHeads) {
#pragma unroll
    for (int t = 0; t < kScaleHeads; ++t) {
      const int h = h0 + t;
      if (h >= p.H) break;
      float c = 1.0f;
      if (p.has_scale) {
        double cd = (double)delta[h];
        if (n > 1) cd += (double)beta[h] * exp((double)gamma[h] * lnL);
        c = (float)cd;
        if (!isfinite(c) && status) atomicOr(status + ENTMAX_ATTN_STATUS_FLAGS, ENTMAX_ATTN_FLAG_BAD_SCALE);
      }
      scale[(size_t)h * p.N + i] = c;
    }
  }
}

// The fp32 accumulators of dK and dV in the problem's type and layout.  Bound by memory: four 16-byte loads in flight per
// thread, and the row of an element by 32-bit arithmetic, or not at all where the output is contiguous (three 64-bit
// divisions for every four elements made 86 us of 4 x 16 x 8192 x 64, now 55, and 20 of 8 x 12 x 1024 x 64, now 11).
template <typename T>
__global__ void __launch_bounds__(256) store_grad_kernel(Problem p, const float* __restrict__ acc_dk,
                                                         const float* __restrict__ acc_dv, T* __restrict__ dk,
                                                         T* __restrict__ dv) {
  pdl_begin();
  constexpr int kFlight = 4;
  const float* __restrict__ acc = blockIdx.y ? acc_dv : acc_dk;
  T* __restrict__ out = blockIdx.y ? dv : dk;
  const int row_shift = p.D == 64 ? 4 : 5;         // 16-byte pieces of a row
  const size_t total4 = ((size_t)p.B * p.H * p.N) << row_shift;
  const bool packed = p.sn == p.D && p.sh == (int64_t)p.N * p.D && p.sb == (int64_t)p.H * p.N * p.D;
  const size_t step = (size_t)gridDim.x * (256 * kFlight);
  for (size_t t0 = (size_t)blockIdx.x * (256 * kFlight) + threadIdx.x; t0 < total4; t0 += step) {
    float x[kFlight][4];
#pragma unroll
    for (int u = 0; u < kFlight; ++u)
      if (t0 + u * 256 < total4) load_slice<4>(acc + 4 * (t0 + u * 256), x[u]);
#pragma unroll
    for (int u = 0; u < kFlight; ++u) {
      const size_t t = t0 + u * 256;
      if (t >= total4) break;
      size_t at = 4 * t;
      if (!packed) {
        const unsigned row = (unsigned)(t >> row_shift), col = 4 * (unsigned)(t & ((1u << row_shift) - 1u));
        const unsigned bh = row / (unsigned)p.N, i = row - bh * p.N, b = bh / (unsigned)p.H, h = bh - b * p.H;
        at = b * p.sb + h * p.sh + i * p.sn + col;
      }
      store_slice<4>(out + at, x[u]);
    }
  }
}

}  // namespace

cudaError_t launch_prologue(const Problem& p, const float* beta, const float* gamma, const float* delta, float* scale,
                            int32_t* clear, size_t n_clear, int32_t* status, cudaStream_t stream) {
  const int most = scale ? p.N : (int)(n_clear < 256 * 148 ? n_clear : 256 * 148);
  const int groups = scale ? (p.H + kScaleHeads - 1) / kScaleHeads : 1;
  const dim3 grid((most + 255) / 256, groups < 65535 ? groups : 65535);
  launch_kernel(prologue_kernel, grid, 256, 0, stream, p, beta, gamma, delta, scale, clear, (int)n_clear, status);
  return cudaGetLastError();
}

cudaError_t launch_dense_fwd(const Problem& p, const void* q, const void* k, const void* v, const float* scale, void* o,
                             float* tau, float* scratch, size_t scratch_floats, int ctas, cudaStream_t stream) {
#define ENTMAX_LAUNCH(T, D)                                                                                      \
  launch_kernel(dense_fwd_kernel<T, D>, ctas, kThreads, 0, stream, p, (const T*)q, (const T*)k, (const T*)v, scale, (T*)o, \
                                                        tau, scratch, scratch_floats)
  if (p.dtype == ENTMAX_ATTN_DTYPE_FP32) {
    if (p.D == 64) ENTMAX_LAUNCH(float, 64); else ENTMAX_LAUNCH(float, 128);
  } else {
    if (p.D == 64) ENTMAX_LAUNCH(__nv_bfloat16, 64); else ENTMAX_LAUNCH(__nv_bfloat16, 128);
  }
#undef ENTMAX_LAUNCH
  return cudaGetLastError();
}

cudaError_t launch_scale_grad(const Problem& p, const float* beta, const float* gamma, const float* dc_rows,
                              double* partial, int32_t* counter, float* dbeta, float* dgamma, float* ddelta,
                              cudaStream_t stream) {
  // CTAs per head: enough for four per SM over all heads, none without a position of its own
  int ctas = (148 * 4 + p.H - 1) / p.H;
  const int most = (p.N + kScaleGradThreads - 1) / kScaleGradThreads;
  if (ctas > most) ctas = most;
  launch_kernel(scale_grad_kernel, dim3(p.H, ctas), kScaleGradThreads, 0, stream, p, beta, gamma, dc_rows, partial, counter, dbeta,
                                                                       dgamma, ddelta);
  return cudaGetLastError();
}

cudaError_t launch_store_grad(const Problem& p, const float* acc_dk, const float* acc_dv, void* dk, void* dv,
                              cudaStream_t stream) {
  const size_t total4 = (size_t)p.B * p.H * p.N * p.D / 4;
  const int blocks = (int)((total4 + 1023) / 1024 < 148 * 8 ? (total4 + 1023) / 1024 : 148 * 8);
  if (p.dtype == ENTMAX_ATTN_DTYPE_FP32) launch_kernel(store_grad_kernel<float>, dim3(blocks, 2), 256, 0, stream, p, acc_dk, acc_dv, (float*)dk, (float*)dv);
  else launch_kernel(store_grad_kernel<__nv_bfloat16>, dim3(blocks, 2), 256, 0, stream, p, acc_dk, acc_dv, (__nv_bfloat16*)dk, (__nv_bfloat16*)dv);
  return cudaGetLastError();
}

}  // namespace entmax
