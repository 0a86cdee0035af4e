// ASEntmax's content-dependent scale (Sec. 4.1 of the paper): per query token and head
//   beta = softplus(<x, w_beta_h>),  gamma = s tanh(<x, w_gamma_h>),  c = delta_h + beta (log n)^gamma
// evaluated from the layer input x, and the chain rule from dL/dc back to w_beta, w_gamma, delta and x.
// The attention calls take c as a per-query table (entmax_attn_fwd_rowscale) and return dL/dc
// (entmax_attn_bwd_rowscale); these two kernels close the loop around them.  Skinny contractions (2 H columns): fp32 FMA
// work bounded by how often the operands are read; x is read once per call in the forward kernel, the backward kernel
// recomputes the projections.
#include <cmath>
#include <initializer_list>

#include "common.cuh"

namespace entmax {

namespace {

constexpr int kProjThreads = 256;
constexpr int kProjWarps = kProjThreads / 32;
constexpr int kTok = 4;                       // tokens a warp projects at a time
constexpr int kHeads = 4;                     // heads per round: kTok * kHeads * 2 = 32 sums, one per lane in the end
constexpr int kChunk = kProjWarps * kTok;     // tokens per CTA in the backward kernel
constexpr int kMaxHeads = 64;
static_assert(kTok * kHeads * 2 == 32, "one sum per lane");

struct ProjArgs {
  int B, H, N, dm;
  int causal, n_mode;
  float s;
};

// VEC consecutive elements of x or of a float32 row (VEC = 1, 2 or 4; aligned to their size)
template <int VEC>
__device__ __forceinline__ void load_vec(const float* p, float (&v)[VEC]) {
  if constexpr (VEC == 1) v[0] = *p;
  else load_slice<VEC>(p, v);
}
template <int VEC>
__device__ __forceinline__ void load_vec(const __nv_bfloat16* p, float (&v)[VEC]) {
  if constexpr (VEC == 1) v[0] = __bfloat162float(*p);
  else load_slice<VEC>(p, v);
}
template <int VEC>
__device__ __forceinline__ void store_vec(float* p, const float (&v)[VEC]) {
  if constexpr (VEC == 1) *p = v[0];
  else store_slice<VEC>(p, v);
}
template <int VEC>
__device__ __forceinline__ void store_vec(__nv_bfloat16* p, const float (&v)[VEC]) {
  if constexpr (VEC == 1) *p = __float2bfloat16_rn(v[0]);
  else store_slice<VEC>(p, v);
}

// The projections of kTok tokens for kHeads heads by one warp: lanes take columns of d_model, every weight a lane loads
// serves all the tokens (one token and one head at a time re-read x for every head and a weight for every token: 81 us for
// 6002 tokens x 768 x 12 heads, now 20), and the 32 sums are reduced together, halving the number of values a lane
// carries with every exchange (31 shuffles instead of 160).  Lane 4 t + hh ends with <x_t, w_beta> of head h0 + hh, lane
// 16 + 4 t + hh with <x_t, w_gamma>.  Tokens and heads past the end are read as the last valid ones.
template <typename T, int VEC>
__device__ __forceinline__ float project_block(const T* x, long tok0, long tokens, const float* wb, const float* wg, int h0,
                                               int H, int dm, int lane) {
  float acc[32];
#pragma unroll
  for (int u = 0; u < 32; ++u) acc[u] = 0.f;
  const T* xr[kTok];
  const float* wr[2 * kHeads];
#pragma unroll
  for (int t = 0; t < kTok; ++t) xr[t] = x + (tok0 + t < tokens ? tok0 + t : tokens - 1) * dm;
#pragma unroll
  for (int hh = 0; hh < kHeads; ++hh) {
    const size_t row = (size_t)(h0 + hh < H ? h0 + hh : H - 1) * dm;
    wr[hh] = wb + row;
    wr[kHeads + hh] = wg + row;
  }
  for (int c = lane * VEC; c < dm; c += 32 * VEC) {
    float xv[kTok][VEC];
#pragma unroll
    for (int t = 0; t < kTok; ++t) load_vec<VEC>(xr[t] + c, xv[t]);
#pragma unroll
    for (int u = 0; u < 2 * kHeads; ++u) {
      float wv[VEC];
      load_vec<VEC>(wr[u] + c, wv);
#pragma unroll
      for (int t = 0; t < kTok; ++t)
#pragma unroll
        for (int e = 0; e < VEC; ++e) {
          float& s = acc[(u / kHeads) * 16 + t * kHeads + (u % kHeads)];
          s = fmaf(xv[t][e], wv[e], s);
        }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const bool upper = (lane & o) != 0;
#pragma unroll
    for (int u = 0; u < o; ++u) {
      const float give = upper ? acc[u] : acc[u + o];
      const float keep = upper ? acc[u + o] : acc[u];
      acc[u] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  return acc[0];
}

// beta, gamma, c and the factors of the chain rule, in double (once per token and head: the cost is nothing, and
// c then agrees with the per-head scale table, which is evaluated the same way)
struct ScalePoint {
  double beta, gamma, c, dc_dpb, dc_dpg;
};
__device__ __forceinline__ ScalePoint scale_point(double pb, double pg, double delta, double s, long n_i) {
  ScalePoint r;
  r.beta = pb > 0.0 ? pb + log1p(exp(-pb)) : log1p(exp(pb));
  const double th = tanh(pg);
  r.gamma = s * th;
  r.c = delta;
  r.dc_dpb = 0.0;
  r.dc_dpg = 0.0;
  if (n_i > 1) {
    const double lnL = log(log((double)n_i)), Lg = exp(r.gamma * lnL);
    r.c = delta + r.beta * Lg;
    r.dc_dpb = Lg / (1.0 + exp(-pb));                          // d beta / d pre = sigmoid
    r.dc_dpg = r.beta * Lg * lnL * s * (1.0 - th * th);     // d gamma / d pre = s (1 - tanh^2)
  }
  return r;
}

template <typename T, int VEC>
__global__ void __launch_bounds__(kProjThreads) scale_proj_fwd_kernel(ProjArgs a, const T* __restrict__ x,
                                                                      const float* __restrict__ w_beta,
                                                                      const float* __restrict__ w_gamma,
                                                                      const float* __restrict__ delta,
                                                                      float* __restrict__ c_rows) {
  pdl_begin();
  const int lane = threadIdx.x & 31;
  const long tokens = (long)a.B * a.N;
  const int rounds = (a.H + kHeads - 1) / kHeads;
  const long work = (tokens + kTok - 1) / kTok * rounds;
  for (long w = (long)blockIdx.x * kProjWarps + (threadIdx.x >> 5); w < work; w += (long)gridDim.x * kProjWarps) {
    const long blk = w / rounds;
    const int h0 = (int)(w - blk * rounds) * kHeads;
    const float s = project_block<T, VEC>(x, blk * kTok, tokens, w_beta, w_gamma, h0, a.H, a.dm, lane);
    const float pg = __shfl_down_sync(0xffffffffu, s, 16);
    const long tok = blk * kTok + lane / kHeads;
    const int h = h0 + lane % kHeads;
    if (lane < 16 && tok < tokens && h < a.H) {
      const long b = tok / a.N, i = tok - b * a.N;
      const long n_i = (a.n_mode || !a.causal) ? a.N : i + 1;
      c_rows[((size_t)b * a.H + h) * a.N + i] = (float)scale_point(s, pg, delta[h], a.s, n_i).c;
    }
  }
}

// One CTA per kChunk tokens: first the chain-rule factors of every (token, head) of the chunk into shared memory, laid out
// [head][token] so that a broadcast 16-byte read serves four tokens; then every thread owns COLS columns of d_model: dx
// for eight tokens at a time (a weight read once per eight tokens), dw for kHeads heads at a time in registers, added by one
// reduction per (head, column) and CTA.  ddelta is summed over the warp's tokens first (an atomic per token and head on H
// addresses was most of the 361 us this took for 6002 tokens x 768 x 12 heads; now 62).
template <typename T, int VEC, int COLS>
__global__ void __launch_bounds__(kProjThreads) scale_proj_bwd_kernel(ProjArgs a, const T* __restrict__ x,
                                                                      const float* __restrict__ w_beta,
                                                                      const float* __restrict__ w_gamma,
                                                                      const float* __restrict__ dc_rows,
                                                                      float* __restrict__ dw_beta,
                                                                      float* __restrict__ dw_gamma,
                                                                      float* __restrict__ ddelta, T* __restrict__ dx) {
  pdl_begin();
  extern __shared__ float4 sm4[];
  float* g_s = reinterpret_cast<float*>(sm4);      // [2][H][kChunk]: dL/d(pre beta), dL/d(pre gamma)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long tokens = (long)a.B * a.N;
  const long tok0 = (long)blockIdx.x * kChunk;
  const int n_tok = (int)(tokens - tok0 < kChunk ? tokens - tok0 : kChunk);
  for (int h0 = 0; h0 < a.H; h0 += kHeads) {
    const float s = project_block<T, VEC>(x, tok0 + warp * kTok, tokens, w_beta, w_gamma, h0, a.H, a.dm, lane);
    const float pg = __shfl_down_sync(0xffffffffu, s, 16);
    const int tl = warp * kTok + lane / kHeads, h = h0 + lane % kHeads;
    float gd = 0.f;
    if (lane < 16 && h < a.H) {
      float gb = 0.f, gg = 0.f;                    // tokens past the end contribute zeros
      if (tl < n_tok) {
        const long tok = tok0 + tl, b = tok / a.N, i = tok - b * a.N;
        const long n_i = (a.n_mode || !a.causal) ? a.N : i + 1;
        gd = dc_rows[((size_t)b * a.H + h) * a.N + i];
        const ScalePoint pt = scale_point(s, pg, 0.0, a.s, n_i);
        gb = (float)(gd * pt.dc_dpb);
        gg = (float)(gd * pt.dc_dpg);
      }
      g_s[h * kChunk + tl] = gb;
      g_s[(a.H + h) * kChunk + tl] = gg;
    }
    if (ddelta) {
      // the warp's four tokens of a head: lanes hh, hh + 4, hh + 8, hh + 12
      gd += __shfl_xor_sync(0xffffffffu, gd, 4);
      gd += __shfl_xor_sync(0xffffffffu, gd, 8);
      if (lane < kHeads && h < a.H) atomicAdd(ddelta + h, gd);
    }
  }
  __syncthreads();
  for (int col = threadIdx.x * COLS; col < a.dm; col += kProjThreads * COLS) {
    if (dx) {
#pragma unroll 1
      for (int t0 = 0; t0 < n_tok; t0 += 8) {
        float acc[8][COLS];
#pragma unroll
        for (int t = 0; t < 8; ++t)
#pragma unroll
          for (int e = 0; e < COLS; ++e) acc[t][e] = 0.f;
#pragma unroll 2
        for (int h = 0; h < a.H; ++h) {
          float wv[2][COLS];
          load_vec<COLS>(w_beta + (size_t)h * a.dm + col, wv[0]);
          load_vec<COLS>(w_gamma + (size_t)h * a.dm + col, wv[1]);
#pragma unroll
          for (int which = 0; which < 2; ++which) {
            const float4* gp = reinterpret_cast<const float4*>(g_s + (which * a.H + h) * kChunk + t0);
            const float4 g0 = gp[0], g1 = gp[1];
            const float gv[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
#pragma unroll
            for (int t = 0; t < 8; ++t)
#pragma unroll
              for (int e = 0; e < COLS; ++e) acc[t][e] = fmaf(gv[t], wv[which][e], acc[t][e]);
          }
        }
#pragma unroll
        for (int t = 0; t < 8; ++t)
          if (t0 + t < n_tok) store_vec<COLS>(dx + (tok0 + t0 + t) * a.dm + col, acc[t]);
      }
    }
#pragma unroll 1
    for (int h0 = 0; h0 < a.H; h0 += kHeads) {
      float acc[2 * kHeads][COLS];
#pragma unroll
      for (int u = 0; u < 2 * kHeads; ++u)
#pragma unroll
        for (int e = 0; e < COLS; ++e) acc[u][e] = 0.f;
#pragma unroll 2
      for (int t0 = 0; t0 < kChunk; t0 += 4) {
        float xv[4][COLS];
#pragma unroll
        for (int t = 0; t < 4; ++t) load_vec<COLS>(x + (t0 + t < n_tok ? tok0 + t0 + t : tok0) * a.dm + col, xv[t]);
#pragma unroll
        for (int u = 0; u < 2 * kHeads; ++u) {
          const int h = h0 + u % kHeads < a.H ? h0 + u % kHeads : a.H - 1;
          const float4 g4 = *reinterpret_cast<const float4*>(g_s + ((u / kHeads) * a.H + h) * kChunk + t0);
#pragma unroll
          for (int e = 0; e < COLS; ++e)
            acc[u][e] = fmaf(g4.x, xv[0][e], fmaf(g4.y, xv[1][e], fmaf(g4.z, xv[2][e], fmaf(g4.w, xv[3][e], acc[u][e]))));
        }
      }
#pragma unroll
      for (int u = 0; u < 2 * kHeads; ++u) {
        if (h0 + u % kHeads >= a.H) continue;
        float* dst = (u < kHeads ? dw_beta : dw_gamma) + (size_t)(h0 + u % kHeads) * a.dm + col;
        if constexpr (COLS == 2) red_add_v2(dst, acc[u][0], acc[u][1]);
        else atomicAdd(dst, acc[u][0]);
      }
    }
  }
}

// vectors of four in the projections and pairs of columns in the chain rule need rows that start on 16 bytes
bool rows_aligned(const ProjArgs& a, std::initializer_list<const void*> ptrs) {
  if (a.dm % 4 != 0) return false;
  for (const void* p : ptrs)
    if (p && !aligned16(p)) return false;
  return true;
}

int check_proj(const entmax_attn_proj_params* p, ProjArgs* a) {
  if (!p) return ENTMAX_ATTN_EINVAL_NULL;
  if (p->batch < 1 || p->heads < 1 || p->heads > kMaxHeads || p->seq < 1 || p->d_model < 1) return ENTMAX_ATTN_EINVAL_SHAPE;
  if ((long long)p->batch * p->heads * p->seq > 0x7fffffffLL / 2) return ENTMAX_ATTN_EINVAL_SHAPE;
  if (p->x_dtype != ENTMAX_ATTN_DTYPE_BF16 && p->x_dtype != ENTMAX_ATTN_DTYPE_FP32) return ENTMAX_ATTN_EINVAL_DTYPE;
  if (!(p->gamma_range > 0.f) || !std::isfinite(p->gamma_range)) return ENTMAX_ATTN_EINVAL_ALPHA;
  a->B = p->batch; a->H = p->heads; a->N = p->seq; a->dm = p->d_model;
  a->causal = p->causal ? 1 : 0;
  a->n_mode = p->n_mode ? 1 : 0;
  a->s = p->gamma_range;
  return ENTMAX_ATTN_OK;
}

}  // namespace

}  // namespace entmax

using namespace entmax;

extern "C" {

int entmax_attn_scale_proj_fwd(const entmax_attn_proj_params* params, const void* x, const float* w_beta,
                               const float* w_gamma, const float* delta, float* c_rows, void* cuda_stream) {
  ProjArgs a;
  int rc = check_proj(params, &a);
  if (rc != ENTMAX_ATTN_OK) return rc;
  if (!x || !w_beta || !w_gamma || !delta || !c_rows) return ENTMAX_ATTN_EINVAL_NULL;
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  const long tokens = (long)a.B * a.N;
  const long work = (tokens + kTok - 1) / kTok * ((a.H + kHeads - 1) / kHeads);
  long ctas = (work + kProjWarps - 1) / kProjWarps;
  if (ctas > 148L * 16) ctas = 148L * 16;
  const bool vec = rows_aligned(a, {x, w_beta, w_gamma});
#define ENTMAX_PROJ_FWD(T, VEC)                                                                                  \
  launch_kernel(scale_proj_fwd_kernel<T, VEC>, (int)ctas, kProjThreads, 0, stream, a, static_cast<const T*>(x), w_beta, w_gamma, delta, \
                                                                        c_rows)
  if (params->x_dtype == ENTMAX_ATTN_DTYPE_FP32) {
    if (vec) ENTMAX_PROJ_FWD(float, 4); else ENTMAX_PROJ_FWD(float, 1);
  } else {
    if (vec) ENTMAX_PROJ_FWD(__nv_bfloat16, 4); else ENTMAX_PROJ_FWD(__nv_bfloat16, 1);
  }
#undef ENTMAX_PROJ_FWD
  cudaError_t err = cudaGetLastError();
  return err == cudaSuccess ? ENTMAX_ATTN_OK : fail_cuda(err);
}

int entmax_attn_scale_proj_bwd(const entmax_attn_proj_params* params, const void* x, const float* w_beta,
                               const float* w_gamma, const float* d_scale_rows, float* dw_beta, float* dw_gamma,
                               float* ddelta, void* dx, void* cuda_stream) {
  ProjArgs a;
  int rc = check_proj(params, &a);
  if (rc != ENTMAX_ATTN_OK) return rc;
  if (!x || !w_beta || !w_gamma || !d_scale_rows || !dw_beta || !dw_gamma) return ENTMAX_ATTN_EINVAL_NULL;
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  cudaError_t err = cudaMemsetAsync(dw_beta, 0, sizeof(float) * (size_t)a.H * a.dm, stream);
  if (err == cudaSuccess) err = cudaMemsetAsync(dw_gamma, 0, sizeof(float) * (size_t)a.H * a.dm, stream);
  if (err == cudaSuccess && ddelta) err = cudaMemsetAsync(ddelta, 0, sizeof(float) * (size_t)a.H, stream);
  if (err != cudaSuccess) return fail_cuda(err);
  const long tokens = (long)a.B * a.N;
  const int ctas = (int)((tokens + kChunk - 1) / kChunk);
  const size_t smem = sizeof(float) * 2 * kChunk * a.H;
  const bool vec = rows_aligned(a, {x, w_beta, w_gamma, dw_beta, dw_gamma, dx});
#define ENTMAX_PROJ_BWD(T, VEC, COLS)                                                                                 \
  launch_kernel(scale_proj_bwd_kernel<T, VEC, COLS>, ctas, kProjThreads, smem, stream, a, static_cast<const T*>(x), w_beta, w_gamma, \
                                                                            d_scale_rows, dw_beta, dw_gamma, ddelta,      \
                                                                            static_cast<T*>(dx))
  if (params->x_dtype == ENTMAX_ATTN_DTYPE_FP32) {
    if (vec) ENTMAX_PROJ_BWD(float, 4, 2); else ENTMAX_PROJ_BWD(float, 1, 1);
  } else {
    if (vec) ENTMAX_PROJ_BWD(__nv_bfloat16, 4, 2); else ENTMAX_PROJ_BWD(__nv_bfloat16, 1, 1);
  }
#undef ENTMAX_PROJ_BWD
  err = cudaGetLastError();
  return err == cudaSuccess ? ENTMAX_ATTN_OK : fail_cuda(err);
}

}  // extern "C"
