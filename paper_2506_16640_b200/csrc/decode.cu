// Decode-shape forward: a few new query rows per sequence against a long key/value cache, sequences of
// different lengths in one batch.  Query t of sequence b sits at position pos = kv_len[b] - q_len + t,
// sees the keys j <= pos, and gets Eq. 1 on its ASEntmax-scaled logits like any row of the full problem
// (n_i = pos + 1).  The path is bound by reading K once from HBM:
//   decode_scores_tc_kernel   (decode_scores_sm100.cu) streams K through TMA and tcgen05, writes
//                             y = a_t (q.k + bias), a_t = (alpha-1) c_t sm_scale, to a score row in the
//                             workspace and the maximum of every 32 keys;
//   decode_solve_kernel       one CTA per query row: y_max, the candidates above the lower end of the bracket
//                             of App. A (tau >= y_max - 1; only 128-key tiles whose maximum lies above it are read),
//                             Newton from the left on them (e-norm step), then
//                             p = [y - tau]_+^e and O = sum_j p_j v_j as a gather of the support's V rows.
// V is read only on the support.  Rows with more candidates than the CTA's list holds run the same
// Newton iteration and output loop over the whole score row instead.
// All sums are taken in a fixed order: repeated calls give identical bits.
#include "common.cuh"
#include "decode.cuh"

namespace entmax {

namespace {

constexpr int kListSlots = 2048;   // candidate slots of a solve CTA, split evenly among its threads
constexpr int kMaxNewtonD = 64;

// PER consecutive bf16 values (PER = 2 or 4), as they lie in memory and as floats
template <int PER>
__device__ __forceinline__ void load_packed_row(const __nv_bfloat16* p, uint32_t (&w)[PER / 2]) {
  if constexpr (PER == 4) {
    const uint2 raw = *reinterpret_cast<const uint2*>(p);
    w[0] = raw.x;
    w[1] = raw.y;
  } else {
    w[0] = *reinterpret_cast<const uint32_t*>(p);
  }
}
__device__ __forceinline__ float packed_at(const uint32_t* w, int e) {
  return __uint_as_float((e & 1) ? (w[e >> 1] & 0xffff0000u) : (w[e >> 1] << 16));
}

// Sum over the CTA in a fixed order; every thread returns the same value.  `slot` alternates between
// calls so that one barrier per call is enough.
template <int kSolveThreads>
__device__ __forceinline__ float2 block_sum2(float x, float y, float2 (*red)[kSolveThreads / 32], int slot) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    x += __shfl_xor_sync(0xffffffffu, x, o);
    y += __shfl_xor_sync(0xffffffffu, y, o);
  }
  if ((threadIdx.x & 31) == 0) red[slot][threadIdx.x >> 5] = make_float2(x, y);
  __syncthreads();
  float2 s = make_float2(0.f, 0.f);
#pragma unroll
  for (int w = 0; w < kSolveThreads / 32; ++w) {
    s.x += red[slot][w].x;
    s.y += red[slot][w].y;
  }
  return s;
}

// A row with more candidates than the list holds: the same iteration and output sum over the whole score row.  The CTA's warps
// leave their shares of O in opart; returns the threshold and (its bits) the support size.  (Out of line, so that it costs the
// usual path no registers.)  The gather takes the warp's ballot of 64 keys and four V rows at a time: as a loop over single
// keys every step waited for its score, 457 us of 16 heads x 32768 keys at c = 1 (8 of 16 rows run over), now 108.
template <int D, int kSolveThreads>
__device__ __noinline__ float2 solve_on_score_row(const float* y_row, int nv, float ymax, int expo_class, float expo,
                                                  const __nv_bfloat16* v_head, int64_t v_stride,
                                                  float2 (*red)[kSolveThreads / 32], int* scan, float (*opart)[D]) {
  constexpr int kWarps = kSolveThreads / 32;
  constexpr int PER = D / 32;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  TauIter st = tau_iter_start(ymax);
  for (int it = 0; it < kMaxNewtonD; ++it) {
    float s0 = 0.f, s1 = 0.f;
    for (int j0 = tid; j0 < nv; j0 += 4 * kSolveThreads) {
      float d[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int j = j0 + u * kSolveThreads;
        d[u] = j < nv ? y_row[j] - st.tau : -INFINITY;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (d[u] > 0.f) {
          float ye, ye1;
          pow_pair(d[u], expo_class, expo, ye, ye1);
          s0 += ye;
          s1 += ye1;
        }
    }
    const float2 s = block_sum2<kSolveThreads>(s0, s1, red, it & 1);
    if (!tau_iter_update(st, s.x, s.y, expo_class, expo, 1e-7f)) break;
  }
  const float tau = st.tau;
  const __nv_bfloat16* vbase = v_head + lane * PER;
  float acc[PER];
#pragma unroll
  for (int e = 0; e < PER; ++e) acc[e] = 0.f;
  int local = 0;
  // a warp looks at 64 keys together and gathers the V rows of those in the support four at a time
  for (int j0 = warp * 64; j0 < nv; j0 += kWarps * 64) {
    float d[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int j = j0 + 32 * u + lane;
      d[u] = j < nv ? y_row[j] - tau : -INFINITY;
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      float ye = 0.f, ye1;
      if (d[u] > 0.f) pow_pair(d[u], expo_class, expo, ye, ye1);
      unsigned m = __ballot_sync(0xffffffffu, d[u] > 0.f);
      local += __popc(m);
      while (m) {
        float p[4];
        uint32_t vw[4][PER / 2];
#pragma unroll
        for (int z = 0; z < 4; ++z) {
          const int src = m ? __ffs(m) - 1 : 0;
          p[z] = __shfl_sync(0xffffffffu, ye, src);
#pragma unroll
          for (int e = 0; e < PER / 2; ++e) vw[z][e] = 0u;
          if (m) load_packed_row<PER>(vbase + (size_t)(j0 + 32 * u + src) * v_stride, vw[z]);
          m &= m - 1;
        }
#pragma unroll
        for (int z = 0; z < 4; ++z)
#pragma unroll
          for (int e = 0; e < PER; ++e) acc[e] = fmaf(p[z], packed_at(vw[z], e), acc[e]);
      }
    }
  }
  if (lane == 0) scan[warp] = local;
#pragma unroll
  for (int e = 0; e < PER; ++e) opart[warp][lane * PER + e] = acc[e];
  __syncthreads();
  int support = 0;
  for (int w = 0; w < kWarps; ++w) support += scan[w];
  return make_float2(tau, __int_as_float(support));
}

// (register cap: without it three CTAs of 512 threads no longer fit an SM, 77.8 us against 76.8 on 8 x 16 x 16384, four queries)
template <int D, int kSolveThreads>
__global__ void __launch_bounds__(kSolveThreads, kSolveThreads == 512 ? 3 : 1) decode_solve_kernel(DecodeArgs a, const __nv_bfloat16* __restrict__ v,
                                                                    const float* __restrict__ scores,
                                                                    const float* __restrict__ tile_max,
                                                                    __nv_bfloat16* __restrict__ o,
                                                                    float* __restrict__ tau_out,
                                                                    int32_t* __restrict__ support_out,
                                                                    int32_t* __restrict__ status) {
  pdl_begin();
  constexpr int kWarps = kSolveThreads / 32;
  constexpr int kPerThread = kListSlots / kSolveThreads;
  constexpr int kCap = kListSlots;
  constexpr int PER = D / 32;
  __shared__ float cand_y[kCap];      // per-thread slots, then the compact list's p values
  __shared__ int cand_j[kCap];
  __shared__ float list_y[kCap];      // candidates compacted in (thread, slot) order
  __shared__ int list_j[kCap];
  __shared__ float2 red[2][kWarps];
  __shared__ float wmax[kWarps];
  __shared__ int scan[kWarps];
  __shared__ float opart[kWarps][D];
  __shared__ int s_overflow;
  __shared__ float s_tau;
  __shared__ int s_support;
  const int row = blockIdx.x;                       // (b * H + h) * QL + t
  const int t = row % a.QL, bh = row / a.QL, h = bh % a.H, b = bh / a.H;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int len = seq_len(a, b, nullptr);
  const int nv = len - a.QL + t + 1;                // visible keys
  const float* y_row = scores + (size_t)row * a.score_stride;
  if (tid == 0) s_overflow = 0;
  // ---- y_max from the tile maxima
  float m = -INFINITY;
  const int tiles = (nv + 127) / 128;
  const float4* row_max = reinterpret_cast<const float4*>(tile_max) + (size_t)row * a.n_tiles;
  for (int c = tid; c < tiles; c += kSolveThreads) {
    const float4 x = row_max[c];
    m = fmaxf(m, fmaxf(fmaxf(x.x, x.y), fmaxf(x.z, x.w)));
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
  if (lane == 0) wmax[warp] = m;
  __syncthreads();
  float ymax = wmax[0];
#pragma unroll
  for (int w = 1; w < kWarps; ++w) ymax = fmaxf(ymax, wmax[w]);
  // ---- candidates: y > y_max - 1 (App. A: tau >= y_max - 1), kept per thread in key order
  const float floor_y = ymax - 1.0f;
  int cnt = 0;
  {
    // Tile t is warp t mod kWarps's, a lane 4 of its 128 keys; 32 of the warp's tiles are tested at a time and those that
    // hold a candidate read, four at a time (a thread meets its keys in increasing order).  The kernel took 12 us on 16 rows
    // of 32768 keys with the whole rows read, 9 now; 18 and 14 on 512 rows of 16384.
    const float4* y_row4 = reinterpret_cast<const float4*>(y_row);
    for (int k0 = 0; warp + k0 * kWarps < tiles; k0 += 32) {
      const int mine = warp + (k0 + lane) * kWarps;
      bool any = false;
      if (mine < tiles) {
        const float4 x = row_max[mine];
        any = fmaxf(fmaxf(x.x, x.y), fmaxf(x.z, x.w)) > floor_y;
      }
      unsigned todo = __ballot_sync(0xffffffffu, any);
      while (todo) {
        int at[4];
        float4 yv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          at[u] = -1;
          yv[u] = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
          if (todo) {
            at[u] = (warp + (k0 + __ffs(todo) - 1) * kWarps) * 32 + lane;
            todo &= todo - 1;
            if (4 * at[u] < nv) yv[u] = y_row4[at[u]];
          }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float ye[4] = {yv[u].x, yv[u].y, yv[u].z, yv[u].w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int j = 4 * at[u] + e;
            if (j < nv && ye[e] > floor_y) {
              if (cnt < kPerThread) {
                cand_y[tid * kPerThread + cnt] = ye[e];
                cand_j[tid * kPerThread + cnt] = j;
              }
              ++cnt;
            }
          }
        }
      }
    }
  }
  if (cnt > kPerThread) s_overflow = 1;
  // ---- compact the candidates in (thread, slot) order
  int incl = cnt < kPerThread ? cnt : kPerThread;
  const int mine = incl;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int up = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += up;
  }
  if (lane == 31) scan[warp] = incl;
  __syncthreads();
  const bool dense = s_overflow != 0;
  int base = 0, n_cand = 0;
  for (int w = 0; w < kWarps; ++w) {
    if (w < warp) base += scan[w];
    n_cand += scan[w];
  }
  if (!dense) {
    const int at = base + incl - mine;
    for (int c = 0; c < mine; ++c) {
      list_y[at + c] = cand_y[tid * kPerThread + c];
      list_j[at + c] = cand_j[tid * kPerThread + c];
    }
  }
  __syncthreads();
  if (dense && tid == 0 && status) atomicAdd(status + ENTMAX_ATTN_STATUS_DENSE_ROWS, 1);
  // ---- Newton from the left on f(tau) = sum [y - tau]_+^e - 1, e-norm step
  TauIter st;
  st.tau = st.lo = floor_y;      // y_max - 1, the bracket's lower end (App. A)
  st.hi = ymax;
  const __nv_bfloat16* v_head = v + (size_t)b * a.ksb + (size_t)h * a.ksh;
  float tau = floor_y;
  int support = 0;
  if (!dense) {
    // the first warp alone: shuffles only, no CTA barriers inside the iteration
    if (warp == 0) {
      for (int it = 0; it < kMaxNewtonD; ++it) {
        float s0 = 0.f, s1 = 0.f;
        for (int c = lane; c < n_cand; c += 32) {
          const float d = list_y[c] - st.tau;
          if (d > 0.f) {
            float ye, ye1;
            pow_pair(d, a.expo_class, a.expo, ye, ye1);
            s0 += ye;
            s1 += ye1;
          }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
          s0 += __shfl_xor_sync(0xffffffffu, s0, off);
          s1 += __shfl_xor_sync(0xffffffffu, s1, off);
        }
        if (!tau_iter_update(st, s0, s1, a.expo_class, a.expo, 1e-7f)) break;
      }
      tau = st.tau;
      // p of every candidate (0 outside the support), in list order
      int local = 0;
      for (int c = lane; c < n_cand; c += 32) {
        const float d = list_y[c] - tau;
        float ye = 0.f, ye1;
        if (d > 0.f) {
          pow_pair(d, a.expo_class, a.expo, ye, ye1);
          ++local;
        }
        cand_y[c] = ye;
      }
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) local += __shfl_xor_sync(0xffffffffu, local, off);
      if (lane == 0) {
        s_tau = tau;
        s_support = local;
      }
    }
    __syncthreads();
    tau = s_tau;
    support = s_support;
    // ---- O = sum_j p_j v_j
    float acc[PER];
#pragma unroll
    for (int e = 0; e < PER; ++e) acc[e] = 0.f;
    for (int c = warp; c < n_cand; c += kWarps) {
      const float p = cand_y[c];
      if (p > 0.f) {
        uint32_t vw[PER / 2];
        load_packed_row<PER>(v_head + (size_t)list_j[c] * a.ksn + lane * PER, vw);
#pragma unroll
        for (int e = 0; e < PER; ++e) acc[e] = fmaf(p, packed_at(vw, e), acc[e]);
      }
    }
#pragma unroll
    for (int e = 0; e < PER; ++e) opart[warp][lane * PER + e] = acc[e];
  } else {
    const float2 solved = solve_on_score_row<D, kSolveThreads>(y_row, nv, ymax, a.expo_class, a.expo, v_head, a.ksn, red, scan,
                                                              opart);
    tau = solved.x;
    support = __float_as_int(solved.y);
  }
  __syncthreads();
  if (tid < D) {
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) s += opart[w][tid];
    o[(size_t)row * D + tid] = __float2bfloat16(s);
  }
  if (tid == 0) {
    tau_out[row] = tau;
    if (support_out) support_out[row] = support;
  }
}

struct DecodeLayout {
  size_t tile_max, scores, total;
  size_t score_stride;
  int chunk_tiles, n_chunks, n_tiles;
};

// A CTA of the score kernel takes 1024 keys where that makes four waves' worth of CTAs at least.  Below that a wave more
// or less, and each CTA's start (barriers, TMEM, the first K tile from HBM: about a tile's time), are what the kernel
// waits for: the number of CTAs per (sequence, head) is the one that needs the fewest tile times, wave by wave of the
// 2 x 148 resident CTAs, and the kernel deals a sequence's tiles to them evenly, however full the cache is.
// 16 heads x 32768 keys, 128 columns: 1024 CTAs of four tiles 31 us, 18 CTAs per head of up to 15 tiles 26 us.
DecodeLayout decode_layout(int B, int H, int QL, int NC) {
  DecodeLayout l;
  const size_t rows = (size_t)B * H * QL;
  const long long bh = (long long)B * H;
  l.n_tiles = (NC + 127) / 128;
  l.chunk_tiles = 8;
  l.n_chunks = (l.n_tiles + 7) / 8;
  if (bh * l.n_chunks < 4 * 148) {
    l.chunk_tiles = 0;
    long long best = 0;
    for (int w = 1; w <= 4; ++w) {
      long long n = w * 296 / bh;
      if (n > l.n_tiles) n = l.n_tiles;
      if (n < 1) continue;
      const long long cost = w * ((l.n_tiles + n - 1) / n + 1);
      if (best == 0 || cost < best) {
        best = cost;
        l.n_chunks = (int)n;
      }
    }
  }
  l.score_stride = ((size_t)NC + 31) / 32 * 32;
  size_t off = 0;
  auto take = [&off](size_t bytes) { size_t at = off; off = (off + bytes + 255) / 256 * 256; return at; };
  l.tile_max = take(rows * l.n_tiles * 4 * sizeof(float));
  l.scores = take(rows * l.score_stride * sizeof(float));
  l.total = off;
  return l;
}

int check_decode_params(const entmax_attn_decode_params* p, DecodeArgs* a) {
  if (!p) return ENTMAX_ATTN_EINVAL_NULL;
  if (p->batch < 1 || p->heads < 1 || p->q_len < 1 || p->q_len > ENTMAX_ATTN_DECODE_MAX_Q) return ENTMAX_ATTN_EINVAL_SHAPE;
  if (p->kv_capacity < p->q_len) return ENTMAX_ATTN_EINVAL_SHAPE;
  if (p->head_dim != 64 && p->head_dim != 128) return ENTMAX_ATTN_EINVAL_SHAPE;
  if ((long long)p->batch * p->heads * p->q_len > 0x7fffffffLL / 4) return ENTMAX_ATTN_EINVAL_SHAPE;
  if (!(p->alpha > 1.0f) || !(p->alpha <= kAlphaMax)) return ENTMAX_ATTN_EINVAL_ALPHA;
  if (!(p->sm_scale >= 0.f) || !(p->sm_scale < INFINITY)) return ENTMAX_ATTN_EINVAL_ALPHA;
  a->B = p->batch; a->H = p->heads; a->QL = p->q_len; a->NC = p->kv_capacity; a->D = p->head_dim;
  a->alpha_m1 = p->alpha - 1.0f;
  a->sm_scale = p->sm_scale == 0.f ? 1.0f / sqrtf((float)p->head_dim) : p->sm_scale;
  a->expo = 1.0f / (p->alpha - 1.0f);
  a->expo_class = p->alpha == 2.0f ? kExpo1 : p->alpha == 1.5f ? kExpo2 : p->alpha == 1.25f ? kExpo4 : kExpoGeneral;
  if (p->kv_stride_b == 0 && p->kv_stride_h == 0 && p->kv_stride_n == 0) {
    a->ksn = p->head_dim;
    a->ksh = (int64_t)p->kv_capacity * p->head_dim;
    a->ksb = (int64_t)p->heads * p->kv_capacity * p->head_dim;
  } else {
    a->ksb = p->kv_stride_b; a->ksh = p->kv_stride_h; a->ksn = p->kv_stride_n;
    if (a->ksn < p->head_dim || a->ksh < 1 || a->ksb < 1) return ENTMAX_ATTN_EINVAL_SHAPE;
    if (a->ksn % 8 || a->ksh % 8 || a->ksb % 8) return ENTMAX_ATTN_EINVAL_SHAPE;
  }
  return ENTMAX_ATTN_OK;
}

}  // namespace

}  // namespace entmax

using namespace entmax;

extern "C" size_t entmax_attn_decode_workspace_bytes(const entmax_attn_decode_params* params) {
  DecodeArgs a;
  if (check_decode_params(params, &a) != ENTMAX_ATTN_OK) return 0;
  return decode_layout(a.B, a.H, a.QL, a.NC).total;
}

extern "C" int entmax_attn_decode_fwd(const entmax_attn_decode_params* params, const void* q, const void* k,
                                      const void* v, const int32_t* kv_len, const float* beta, const float* gamma,
                                      const float* delta, const float* alibi_slopes, void* o, float* tau,
                                      int32_t* support_size, void* workspace, size_t workspace_bytes,
                                      int32_t* device_status, void* cuda_stream) {
  DecodeArgs a;
  int rc = check_decode_params(params, &a);
  if (rc != ENTMAX_ATTN_OK) return rc;
  if (!q || !k || !v || !o || !tau) return ENTMAX_ATTN_EINVAL_NULL;
  const int given = (beta != nullptr) + (gamma != nullptr) + (delta != nullptr);
  if (given != 0 && given != 3) return ENTMAX_ATTN_EINVAL_NULL;
  auto aligned = [](const void* p, uintptr_t m) { return (reinterpret_cast<uintptr_t>(p) & (m - 1)) == 0; };
  if (!aligned(q, 16) || !aligned(k, 16) || !aligned(v, 16) || !aligned(o, 16) || !aligned(tau, 4)) return ENTMAX_ATTN_EINVAL_ALIGN;
  if ((kv_len && !aligned(kv_len, 4)) || (alibi_slopes && !aligned(alibi_slopes, 4)) ||
      (support_size && !aligned(support_size, 4)))
    return ENTMAX_ATTN_EINVAL_ALIGN;
  const DecodeLayout lay = decode_layout(a.B, a.H, a.QL, a.NC);
  if (!workspace || !aligned(workspace, 256) || workspace_bytes < lay.total) return ENTMAX_ATTN_EINVAL_WORKSPACE;
  a.kv_len = kv_len;
  a.alibi = alibi_slopes;
  a.beta = beta; a.gamma = gamma; a.delta = delta;
  a.chunk_tiles = lay.chunk_tiles;
  a.n_chunks = lay.n_chunks;
  a.n_tiles = lay.n_tiles;
  a.score_stride = lay.score_stride;
  int dev = 0, major = 0;
  cudaError_t err = cudaGetDevice(&dev);
  if (err == cudaSuccess) err = cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
  if (err != cudaSuccess) return fail_cuda(err);
  if (major != 10) return ENTMAX_ATTN_EUNSUPPORTED;          // the score kernel needs tcgen05 / TMA
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  uint8_t* ws = static_cast<uint8_t*>(workspace);
  float* tile_max = reinterpret_cast<float*>(ws + lay.tile_max);
  float* scores = reinterpret_cast<float*>(ws + lay.scores);
  if (device_status) {
    err = cudaMemsetAsync(device_status, 0, sizeof(int32_t) * ENTMAX_ATTN_STATUS_WORDS, stream);
    if (err != cudaSuccess) return fail_cuda(err);
  }
  const int rows = a.B * a.H * a.QL;
  err = launch_decode_scores_tc(a, q, k, scores, tile_max, device_status, stream);
  if (err != cudaSuccess) return fail_cuda(err);
  const __nv_bfloat16* vb = static_cast<const __nv_bfloat16*>(v);
  __nv_bfloat16* ob = static_cast<__nv_bfloat16*>(o);
  // long rows: more threads per row (more loads in flight); many short rows: smaller CTAs
#define ENTMAX_SOLVE(D, T) \
  launch_kernel(decode_solve_kernel<D, T>, rows, T, 0, stream, a, vb, scores, tile_max, ob, tau, support_size, device_status)
  if (a.NC >= 16384) {
    if (a.D == 64) ENTMAX_SOLVE(64, 512); else ENTMAX_SOLVE(128, 512);
  } else {
    if (a.D == 64) ENTMAX_SOLVE(64, 256); else ENTMAX_SOLVE(128, 256);
  }
#undef ENTMAX_SOLVE
  err = cudaGetLastError();
  return err == cudaSuccess ? ENTMAX_ATTN_OK : fail_cuda(err);
}
