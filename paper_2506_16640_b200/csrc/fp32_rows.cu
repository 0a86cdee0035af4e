// float32 problems on CUDA cores (fp32 FMA dot products: the tighter threshold tolerance of float32 inputs is out of
// reach of bf16 tensor-core operands).
//
// A CTA takes R consecutive query rows of one (batch, head) in two phases:
//   scores   y_ij = a_i <q_i, k_j> for the R rows against tiles of kKeys keys: the K tile in shared memory (rows padded by
//            16 bytes, so that eight lanes reading 16 bytes of eight different keys hit all banks), a thread holding eight
//            rows x one or two keys in registers; written to the CTA's score rows in global scratch (they stay in L2).
//            One CTA per row with a warp per key, which this replaces, spent five shuffles and a load of K on every 64
//            multiply-adds and read all of K once per row.
//   rows     one warp per row: forward, the bracket of App. A (tau >= y_max - 1) cuts the row down to its candidates,
//            compacted into shared memory (the K tile's space), Newton on those, output as a gather over the support;
//            backward, the support y > tau is compacted, dP by eight lanes per key, the entmax Jacobian, dQ as a gather
//            and dK, dV by vector reductions.
// What bounds it: the score phase runs at the rate shared memory feeds the FMA pipes (16 bytes of LDS bandwidth per 16
// multiply-adds of a warp); at short lengths, the latency of the row phase.  Measured with 2 x 4 heads x 777 x 64, causal:
// forward 250 -> 37 us, backward 430 -> 38 us; 2 heads x 128 x 64 forward 17 -> 11 us.
#include "common.cuh"

namespace entmax {

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kKeys = 256;              // keys of a K tile
constexpr int kChunkD = 64;             // columns of a K tile (head_dim 128 takes two tiles per key block)
constexpr int kPitch = kChunkD + 4;     // floats from one key of the tile to the next
constexpr int kTileFloats = kKeys * kPitch;
constexpr int kMaxNewton = 400;
constexpr int kFwdCap = kTileFloats / (2 * kWarps);   // candidates (y, j) a warp can hold in the K tile's space
constexpr int kBwdCap = kTileFloats / (3 * kWarps);   // support entries (y, j, dP)
static_assert(kFwdCap >= 256 && kBwdCap >= 256, "row lists");

template <int D, int R>
constexpr int smem_bytes() { return (kTileFloats + R * D) * (int)sizeof(float); }
// CTAs an SM holds (228 KB of shared memory, 1 KB of it reserved per CTA): three, two for sixteen rows of 128
template <int D, int R>
constexpr int resident_ctas() { return 3 * (smem_bytes<D, R>() + 1024) <= 233472 ? 3 : 2; }

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

struct RowTile {
  int bh, b, h, i0, n_rows, nv_max;     // rows i0 .. i0 + n_rows - 1; keys 0 .. nv_max - 1 are visible to some of them
  size_t base;                          // element offset of (b, h, 0, 0)
};
// Work item t: on causal problems the row tiles that see the most keys come first, the heads interleaved.
template <int R>
__device__ __forceinline__ RowTile row_tile(const Problem& p, int t) {
  const int n_bh = p.B * p.H, tiles = (p.N + R - 1) / R;
  RowTile r;
  r.bh = t % n_bh;
  r.b = r.bh / p.H;
  r.h = r.bh - r.b * p.H;
  r.i0 = (tiles - 1 - t / n_bh) * R;
  r.n_rows = min(R, p.N - r.i0);
  r.nv_max = p.causal ? r.i0 + r.n_rows : p.N;
  r.base = (size_t)r.b * p.sb + (size_t)r.h * p.sh;
  return r;
}

// Scores of the tile's rows into ybuf (row pitch `pitch` floats).  q_s: [R][D] floats, k_s: [kKeys][kPitch] floats.
template <int D, int R>
__device__ __forceinline__ void score_tile(const Problem& p, const RowTile& rt, const float* __restrict__ q,
                                           const float* __restrict__ k, const float* __restrict__ scale, float* q_s,
                                           float* k_s, float* ybuf, int pitch) {
  constexpr int KPT = R / 8;            // keys per thread: 8 rows x KPT keys
  constexpr int kRowGroups = R / 8, kKeyGroups = kWarps / kRowGroups;
  static_assert(kKeyGroups * 32 * KPT == kKeys, "a K tile is one key group per warp and row group");
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row0 = (w % kRowGroups) * 8, key0 = (w / kRowGroups) * 32 * KPT + lane;
  for (int t = threadIdx.x; t < R * D / 4; t += kThreads) {
    const int r = t / (D / 4), c = t % (D / 4);
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r < rt.n_rows) x = *reinterpret_cast<const float4*>(q + rt.base + (size_t)(rt.i0 + r) * p.sn + 4 * c);
    *reinterpret_cast<float4*>(q_s + r * D + 4 * c) = x;
  }
  const float slope = p.alibi ? p.alibi[rt.h] / p.sm_scale : 0.f;
  float a[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const int i = rt.i0 + row0 + r;
    a[r] = row0 + r < rt.n_rows
               ? (p.alpha - 1.0f) * (scale[(size_t)rt.b * p.scale_sb + (size_t)rt.h * p.N + i] * p.sm_scale) : 0.f;
  }
  for (int j0 = 0; j0 < rt.nv_max; j0 += kKeys) {
    float acc[8][KPT];
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
      for (int u = 0; u < KPT; ++u) acc[r][u] = 0.f;
#pragma unroll 1
    for (int dc = 0; dc < D; dc += kChunkD) {
      __syncthreads();                  // the previous tile has been used (and, the first time, Q is in shared memory)
      for (int t = threadIdx.x; t < kKeys * kChunkD / 4; t += kThreads) {
        const int j = t / (kChunkD / 4), c = t % (kChunkD / 4);
        if (j0 + j < rt.nv_max)
          *reinterpret_cast<float4*>(k_s + j * kPitch + 4 * c) =
              *reinterpret_cast<const float4*>(k + rt.base + (size_t)(j0 + j) * p.sn + dc + 4 * c);
      }
      __syncthreads();
      if (j0 + (w / kRowGroups) * 32 * KPT < rt.nv_max) {
#pragma unroll 4
        for (int c = 0; c < kChunkD; c += 4) {
          float4 kv[KPT];
#pragma unroll
          for (int u = 0; u < KPT; ++u) kv[u] = *reinterpret_cast<const float4*>(k_s + (key0 + 32 * u) * kPitch + c);
#pragma unroll
          for (int r = 0; r < 8; ++r) {
            const float4 qv = *reinterpret_cast<const float4*>(q_s + (row0 + r) * D + dc + c);
#pragma unroll
            for (int u = 0; u < KPT; ++u)
              acc[r][u] = fmaf(qv.w, kv[u].w, fmaf(qv.z, kv[u].z, fmaf(qv.y, kv[u].y, fmaf(qv.x, kv[u].x, acc[r][u]))));
          }
        }
      }
    }
#pragma unroll
    for (int u = 0; u < KPT; ++u) {
      const int j = j0 + key0 + 32 * u;
      if (j < rt.nv_max) {
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          float dot = acc[r][u];
          // ALiBi: the logit is sm_scale * (dot - slope |i - j|) with slope = m_h / sm_scale
          if (slope != 0.f) dot -= slope * fabsf((float)(j - (rt.i0 + row0 + r)));
          ybuf[(size_t)(row0 + r) * pitch + j] = a[r] * dot;
        }
      }
    }
  }
  __syncthreads();                      // the scores are in place, the K tile's space is free
}

// Keys [from, nv) of a score row with y > cut, compacted into (ly, lj) in key order, whole blocks of 128 keys at a time
// until the row ends or fewer than 128 slots are left.  Returns the entry count; `from` moves to the next key to look at.
__device__ __forceinline__ int compact_row(const float* y, int nv, float cut, int cap, float* ly, int* lj, int lane,
                                           int& from) {
  int cnt = 0;
  for (; from < nv && cnt + 128 <= cap; from += 128) {
    const int j = from + 4 * lane;
    float4 v = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
    if (j < nv) v = *reinterpret_cast<const float4*>(y + j);
    const float e[4] = {v.x, j + 1 < nv ? v.y : -INFINITY, j + 2 < nv ? v.z : -INFINITY, j + 3 < nv ? v.w : -INFINITY};
    int n = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) n += e[u] > cut ? 1 : 0;
    if (!__any_sync(0xffffffffu, n > 0)) continue;
    int pos = n;                        // inclusive prefix sum over the lanes
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, pos, o);
      if (lane >= o) pos += t;
    }
    const int total = __shfl_sync(0xffffffffu, pos, 31);
    pos += cnt - n;
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (e[u] > cut) {
        ly[pos] = e[u];
        lj[pos] = j + u;
        ++pos;
      }
    cnt += total;
  }
  __syncwarp();
  return cnt;
}

template <int D, int R>
__global__ void __launch_bounds__(kThreads, resident_ctas<D, R>()) fp32_fwd_kernel(Problem p, const float* __restrict__ q,
                                                               const float* __restrict__ k, const float* __restrict__ v,
                                                               const float* __restrict__ scale, float* __restrict__ o,
                                                               float* __restrict__ tau_out, int32_t* __restrict__ row_cnt,
                                                               int32_t* __restrict__ dense_cnt, Entry* __restrict__ entries,
                                                               float* scratch, int pitch, int items) {
  pdl_begin();
  constexpr int PER = D / 32;
  extern __shared__ float4 sm4[];
  float* k_s = reinterpret_cast<float*>(sm4);
  float* q_s = k_s + kTileFloats;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* ybuf = scratch + (size_t)blockIdx.x * R * pitch;
  float* ly = k_s + w * 2 * kFwdCap;
  int* lj = reinterpret_cast<int*>(ly + kFwdCap);
  for (int t = blockIdx.x; t < items; t += gridDim.x) {
    const RowTile rt = row_tile<R>(p, t);
    score_tile<D, R>(p, rt, q, k, scale, q_s, k_s, ybuf, pitch);
    for (int r = w; r < rt.n_rows; r += kWarps) {
      const int i = rt.i0 + r, nv = p.causal ? i + 1 : p.N;
      const int grow = rt.bh * p.N + i;
      const float* y = ybuf + (size_t)r * pitch;
      float ymax = -INFINITY;
      for (int j = 4 * lane; j < nv; j += 128) {
        const float4 x = *reinterpret_cast<const float4*>(y + j);
        ymax = fmaxf(ymax, x.x);
        if (j + 1 < nv) ymax = fmaxf(ymax, x.y);
        if (j + 2 < nv) ymax = fmaxf(ymax, x.z);
        if (j + 3 < nv) ymax = fmaxf(ymax, x.w);
      }
      ymax = warp_max(ymax);
      // everything that can have p > 0 (tau >= y_max - 1); more than the list holds: the row itself is walked instead
      int from = 0;
      const int cnt = compact_row(y, nv, ymax - 1.0f, kFwdCap, ly, lj, lane, from);
      const bool listed = from >= nv;
      const float* src = listed ? ly : y;
      const int n = listed ? cnt : nv;
      TauIter st = tau_iter_start(ymax);
      for (int it = 0; it < kMaxNewton; ++it) {
        float s0 = 0.f, s1 = 0.f;
        for (int e = lane; e < n; e += 32) {
          const float d = src[e] - st.tau;
          if (d > 0.f) {
            float ye, ye1;
            pow_pair(d, p.expo_class, p.expo, ye, ye1);
            s0 += ye;
            s1 += ye1;
          }
        }
        if (!tau_iter_update(st, warp_sum(s0), warp_sum(s1), p.expo_class, p.expo, 1e-7f)) break;
      }
      const float tau = st.tau;
      float acc[PER];
#pragma unroll
      for (int u = 0; u < PER; ++u) acc[u] = 0.f;
      Entry* list = entries + (size_t)grow * kListCap;
      const float* vbase = v + rt.base + lane * PER;
      int supp = 0;
      for (int e0 = 0; e0 < n; e0 += 32) {
        const int e = e0 + lane;
        const float ye = e < n ? src[e] : -INFINITY;
        const int je = listed ? (e < n ? lj[e] : 0) : e;
        float pe = 0.f, pe1;
        const bool in = ye - tau > 0.f;
        if (in) pow_pair(ye - tau, p.expo_class, p.expo, pe, pe1);
        unsigned m = __ballot_sync(0xffffffffu, in);
        if (in) {
          const int pos = supp + __popc(m & ((1u << lane) - 1u));
          if (pos < kListCap) {
            list[pos].y = ye;
            list[pos].j = je;
          }
        }
        supp += __popc(m);
        while (m) {
          // four keys at a time, so that their loads are in flight together
          int kj[4];
          float pj[4], vs[4][PER];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int src_lane = m ? __ffs(m) - 1 : 0;
            pj[u] = __shfl_sync(0xffffffffu, pe, src_lane);
            kj[u] = __shfl_sync(0xffffffffu, je, src_lane);
            if (!m) {
              pj[u] = 0.f;
              kj[u] = 0;
            }
            m &= m - 1;
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) load_slice<PER>(vbase + (size_t)kj[u] * p.sn, vs[u]);
#pragma unroll
          for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int c = 0; c < PER; ++c) acc[c] = pj[u] != 0.f ? fmaf(pj[u], vs[u][c], acc[c]) : acc[c];
        }
      }
      store_slice<PER>(o + rt.base + (size_t)i * p.sn + lane * PER, acc);
      if (lane == 0) {
        tau_out[grow] = tau;
        row_cnt[grow] = supp <= kListCap ? supp : -2;
        // a support too long for the list: its size alone is kept (same place and form as the dense-tile kernel's)
        if (supp > kListCap) {
          dense_cnt[2 * (size_t)grow] = supp;
          dense_cnt[2 * (size_t)grow + 1] = 0;
        }
      }
      __syncwarp();
    }
    __syncthreads();                    // the lists are in the space of the next item's K tile
  }
}

// acc_dk, acc_dv: fp32 [B,H,N,D] contiguous, zero on entry
template <int D, int R>
__global__ void __launch_bounds__(kThreads, resident_ctas<D, R>()) fp32_bwd_kernel(Problem p, const float* __restrict__ q,
                                                               const float* __restrict__ k, const float* __restrict__ v,
                                                               const float* __restrict__ d_o, const float* __restrict__ scale,
                                                               const float* __restrict__ tau_in, float* __restrict__ dq,
                                                               float* __restrict__ acc_dk, float* __restrict__ acc_dv,
                                                               float* __restrict__ dc_rows, float* scratch, int pitch,
                                                               int items) {
  pdl_begin();
  constexpr int PL = D / 8;             // elements of a row per lane, eight lanes per key, in chunks of four
  extern __shared__ float4 sm4[];
  float* k_s = reinterpret_cast<float*>(sm4);
  float* q_s = k_s + kTileFloats;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int grp = lane >> 3, sl = lane & 7;
  float* ybuf = scratch + (size_t)blockIdx.x * R * pitch;
  float* ly = k_s + w * 3 * kBwdCap;
  int* lj = reinterpret_cast<int*>(ly + kBwdCap);
  float* ld = ly + 2 * kBwdCap;
  auto load8 = [&](const float* row, float (&x)[PL]) {
#pragma unroll
    for (int c = 0; c < PL / 4; ++c) {
      const float4 t = *reinterpret_cast<const float4*>(row + 32 * c + 4 * sl);
      x[4 * c] = t.x; x[4 * c + 1] = t.y; x[4 * c + 2] = t.z; x[4 * c + 3] = t.w;
    }
  };
  for (int t = blockIdx.x; t < items; t += gridDim.x) {
    const RowTile rt = row_tile<R>(p, t);
    score_tile<D, R>(p, rt, q, k, scale, q_s, k_s, ybuf, pitch);
    for (int r = w; r < rt.n_rows; r += kWarps) {
      const int i = rt.i0 + r, nv = p.causal ? i + 1 : p.N;
      const int grow = rt.bh * p.N + i;
      const float* y = ybuf + (size_t)r * pitch;
      const float tau = tau_in[grow];
      const float c_i = scale[(size_t)rt.b * p.scale_sb + (size_t)rt.h * p.N + i];
      const float g = c_i * p.sm_scale;
      float gs[PL];
      load8(d_o + rt.base + (size_t)i * p.sn, gs);
      // the support in stretches of at most kBwdCap entries (nearly always one), with dP of every entry
      int from = 0, cnt = 0;
      auto stretch = [&]() {
        cnt = compact_row(y, nv, tau, kBwdCap, ly, lj, lane, from);
        for (int e0 = 0; e0 < cnt; e0 += 8) {
          float dp[2] = {0.f, 0.f};
          float vs[2][PL];
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int e = e0 + 4 * u + grp;
            load8(v + rt.base + (size_t)lj[e < cnt ? e : 0] * p.sn, vs[u]);
          }
#pragma unroll
          for (int u = 0; u < 2; ++u) {
#pragma unroll
            for (int c = 0; c < PL; ++c) dp[u] = fmaf(gs[c], vs[u][c], dp[u]);
#pragma unroll
            for (int off = 1; off < 8; off <<= 1) dp[u] += __shfl_xor_sync(0xffffffffu, dp[u], off);
            const int e = e0 + 4 * u + grp;
            if (sl == 0 && e < cnt) ld[e] = dp[u];
          }
        }
        __syncwarp();
      };
      float su = 0.f, sud = 0.f;
      bool whole = true;
      while (from < nv) {
        stretch();
        whole = whole && from >= nv;
        for (int e = lane; e < cnt; e += 32) {
          float pe, u;
          pow_pair(ly[e] - tau, p.expo_class, p.expo, pe, u);
          su += u;
          sud += u * ld[e];
        }
        __syncwarp();
      }
      su = warp_sum(su);
      sud = warp_sum(sud);
      const float rho = su > 0.f ? sud / su : 0.f;
      float qs[PL], acc[PL], dc = 0.f;
      load8(q + rt.base + (size_t)i * p.sn, qs);
#pragma unroll
      for (int c = 0; c < PL; ++c) acc[c] = 0.f;
      const size_t arow = (size_t)rt.bh * p.N;
      if (!whole) from = 0;
      for (bool first = true; first || from < nv; first = false) {
        if (!whole) stretch();
        for (int e0 = 0; e0 < cnt; e0 += 4) {
          const int e = e0 + grp;
          if (e < cnt) {
            const float ye = ly[e];
            const int j = lj[e];
            float pe, u;
            pow_pair(ye - tau, p.expo_class, p.expo, pe, u);
            const float ds = u * (ld[e] - rho), gds = g * ds;
            if (sl == 0) dc = fmaf(ds, ye, dc);       // sum_j dS_ij y_ij
            float ks[PL];
            load8(k + rt.base + (size_t)j * p.sn, ks);
            float* dkr = acc_dk + (arow + j) * D + 4 * sl;
            float* dvr = acc_dv + (arow + j) * D + 4 * sl;
#pragma unroll
            for (int c = 0; c < PL / 4; ++c) {
#pragma unroll
              for (int z = 0; z < 4; ++z) acc[4 * c + z] = fmaf(gds, ks[4 * c + z], acc[4 * c + z]);
              red_add_v4(dkr + 32 * c, gds * qs[4 * c], gds * qs[4 * c + 1], gds * qs[4 * c + 2], gds * qs[4 * c + 3]);
              red_add_v4(dvr + 32 * c, pe * gs[4 * c], pe * gs[4 * c + 1], pe * gs[4 * c + 2], pe * gs[4 * c + 3]);
            }
          }
        }
        __syncwarp();
      }
#pragma unroll
      for (int c = 0; c < PL; ++c) {
        acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], 8);
        acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], 16);
      }
      if (grp == 0) {
        float* dqr = dq + rt.base + (size_t)i * p.sn + 4 * sl;
#pragma unroll
        for (int c = 0; c < PL / 4; ++c)
          *reinterpret_cast<float4*>(dqr + 32 * c) = make_float4(acc[4 * c], acc[4 * c + 1], acc[4 * c + 2], acc[4 * c + 3]);
      }
      if (dc_rows) {
        // dL/dc_i = sum_j dS_ij z_ij, z_ij = y_ij / ((alpha-1) c_i)  (y = (alpha-1) c z)
        dc = warp_sum(dc);
        const float denom = (p.alpha - 1.0f) * c_i;
        if (lane == 0) dc_rows[grow] = denom != 0.f ? dc / denom : 0.f;
      }
    }
    __syncthreads();
  }
}

// Rows per CTA: eight (one per warp) while sixteen would leave SMs without a CTA
bool eight_rows(const Problem& p) { return (long)p.B * p.H * ((p.N + 15) / 16) < 148; }

// Long problems, whose score rows leave fewer CTAs than the SMs hold: these start only after the kernel before them.  Beside
// its last CTAs they would be placed two on one SM and none on another, and stay there for the whole problem (32768 x 64, one
// head: forward 12.2 ms, placed early 13.5 to 15.2; 3 x 40000 x 128 76 and 90).  Where the grid fills the machine an early
// start gains (2 x 8 x 2048 x 64: 316 us against 326).
bool plain_launch(long items, int ctas) { return items > ctas && ctas < 148 * 3; }

template <int D, int R>
cudaError_t launch_fwd(const Problem& p, const float* q, const float* k, const float* v, const float* scale, float* o,
                       float* tau, int32_t* row_cnt, int32_t* dense_cnt, Entry* entries, float* scratch, int ctas,
                       cudaStream_t stream) {
  constexpr int bytes = smem_bytes<D, R>();
  const long items = (long)p.B * p.H * ((p.N + R - 1) / R);
  cudaError_t err = cudaFuncSetAttribute(fp32_fwd_kernel<D, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (err != cudaSuccess) return err;
  if (plain_launch(items, ctas))
    fp32_fwd_kernel<D, R><<<ctas, kThreads, bytes, stream>>>(p, q, k, v, scale, o, tau, row_cnt, dense_cnt, entries, scratch,
                                                             fp32_scratch_pitch(p), (int)items);
  else
    launch_kernel(fp32_fwd_kernel<D, R>, (int)(items < ctas ? items : ctas), kThreads, bytes, stream, p, q, k, v, scale, o, tau, row_cnt, dense_cnt,
                  entries, scratch, fp32_scratch_pitch(p), (int)items);
  return cudaGetLastError();
}
template <int D, int R>
cudaError_t launch_bwd(const Problem& p, const float* q, const float* k, const float* v, const float* d_o, const float* scale,
                       const float* tau, float* dq, float* acc_dk, float* acc_dv, float* dc_rows, float* scratch, int ctas,
                       cudaStream_t stream) {
  constexpr int bytes = smem_bytes<D, R>();
  const long items = (long)p.B * p.H * ((p.N + R - 1) / R);
  cudaError_t err = cudaFuncSetAttribute(fp32_bwd_kernel<D, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (err != cudaSuccess) return err;
  if (plain_launch(items, ctas))
    fp32_bwd_kernel<D, R><<<ctas, kThreads, bytes, stream>>>(p, q, k, v, d_o, scale, tau, dq, acc_dk, acc_dv, dc_rows, scratch,
                                                             fp32_scratch_pitch(p), (int)items);
  else
    launch_kernel(fp32_bwd_kernel<D, R>, (int)(items < ctas ? items : ctas), kThreads, bytes, stream, p, q, k, v, d_o, scale, tau, dq, acc_dk, acc_dv,
                  dc_rows, scratch, fp32_scratch_pitch(p), (int)items);
  return cudaGetLastError();
}

}  // namespace

int fp32_scratch_pitch(const Problem& p) { return (p.N + 31) / 32 * 32; }
int fp32_scratch_rows(const Problem& p) { return eight_rows(p) ? 8 : 16; }
// 3 x 148 CTAs while their score rows stay within 256 MB, never fewer than one per SM.  (Also where the SMs hold fewer: what
// waits for a free place evens out the items' lengths.  2 x 4 x 777 x 128 causal: 64 us, with 2 x 148 CTAs 81.)
int fp32_scratch_ctas(const Problem& p) {
  const int rows = fp32_scratch_rows(p);
  const long items = (long)p.B * p.H * ((p.N + rows - 1) / rows);
  const long per = (long)rows * fp32_scratch_pitch(p) * 4;
  long ctas = (256L << 20) / per;
  ctas = ctas > 148 * 3 ? 148 * 3 : ctas < 148 ? 148 : ctas;
  return (int)(items < ctas ? items : ctas);
}

cudaError_t launch_fp32_fwd(const Problem& p, const float* q, const float* k, const float* v, const float* scale, float* o,
                            float* tau, int32_t* row_cnt, int32_t* dense_cnt, Entry* entries, float* scratch, int ctas,
                            cudaStream_t stream) {
#define ENTMAX_FP32_FWD(D, R) launch_fwd<D, R>(p, q, k, v, scale, o, tau, row_cnt, dense_cnt, entries, scratch, ctas, stream)
  if (p.D == 64) return eight_rows(p) ? ENTMAX_FP32_FWD(64, 8) : ENTMAX_FP32_FWD(64, 16);
  return eight_rows(p) ? ENTMAX_FP32_FWD(128, 8) : ENTMAX_FP32_FWD(128, 16);
#undef ENTMAX_FP32_FWD
}

cudaError_t launch_fp32_bwd(const Problem& p, const float* q, const float* k, const float* v, const float* d_o,
                            const float* scale, const float* tau, float* dq, float* acc_dk, float* acc_dv, float* dc_rows,
                            float* scratch, int ctas, cudaStream_t stream) {
#define ENTMAX_FP32_BWD(D, R) launch_bwd<D, R>(p, q, k, v, d_o, scale, tau, dq, acc_dk, acc_dv, dc_rows, scratch, ctas, stream)
  if (p.D == 64) return eight_rows(p) ? ENTMAX_FP32_BWD(64, 8) : ENTMAX_FP32_BWD(64, 16);
  return eight_rows(p) ? ENTMAX_FP32_BWD(128, 8) : ENTMAX_FP32_BWD(128, 16);
#undef ENTMAX_FP32_BWD
}

}  // namespace entmax
