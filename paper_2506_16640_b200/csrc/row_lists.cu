// Per-row kernels of the bf16 path that work on the sparse candidate lists left by the tensor-core
// score sweep (see common.cuh).
//
// Forward: exact threshold on the candidates (Eq. 1 with the sum-to-one condition), probabilities, and
// O_i = sum_j p_ij v_j as a gather over the support only -- every zero of P is skipped, not just
// all-zero tiles.  A thread solves a row (lists of up to 32 entries, in registers), then lanes share the gathers of a row.
// Backward: the entmax Jacobian dS = u (dP - <u,dP>/sum u), u = p^(2-alpha), on the support, dQ by
// gathering K rows, dK / dV by vector atomics into fp32 accumulators.
#include "common.cuh"

namespace entmax {

namespace {

constexpr int kWarpsPerCta = 8;
constexpr int kSlots = kListCap / 32;
constexpr int kMaxNewton = 400;

// Butterfly sum, strides ascending as in sub_sum below.
__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}
__device__ __forceinline__ float warp_max(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
  return x;
}

// reductions over aligned groups of W lanes (W = 8 or 16); the sum takes ascending strides like warp_sum
template <int W>
__device__ __forceinline__ float sub_sum(float x) {
#pragma unroll
  for (int o = 1; o < W; o <<= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// A lane's share of a row of D elements, W lanes per row: PL = D / W elements.  They are taken as chunks of four
// that interleave across the lanes (chunk c of lane sl = elements [4 W c + 4 sl, +4)), so that what the W lanes
// move in one instruction is contiguous: 16-byte reductions of neighbouring lanes fall into the same 32-byte
// sector instead of half-filling one each, loads and stores stay coalesced.  (PL < 4: one contiguous piece.)
template <int PL, int W>
__device__ __forceinline__ void store_share(__nv_bfloat16* row, int sl, const float (&x)[PL]) {
  if constexpr (PL < 4) {
    store_slice<PL>(row + sl * PL, x);
  } else {
#pragma unroll
    for (int c = 0; c < PL / 4; ++c) {
      const float t[4] = {x[4 * c], x[4 * c + 1], x[4 * c + 2], x[4 * c + 3]};
      store_slice<4>(row + 4 * W * c + 4 * sl, t);
    }
  }
}
template <int PL, int W>
__device__ __forceinline__ void add_share(float* row, int sl, const float (&x)[PL]) {
  if constexpr (PL < 4) {
    atomic_add_slice<PL>(row + sl * PL, x);
  } else {
#pragma unroll
    for (int c = 0; c < PL / 4; ++c) red_add_v4(row + 4 * W * c + 4 * sl, x[4 * c], x[4 * c + 1], x[4 * c + 2], x[4 * c + 3]);
  }
}

// A lane's share of a row as it lies in memory (interleaved as above), two elements to a register: half the
// registers of its floats, so that several rows can be in flight.
template <int PL>
struct PackedShare {
  uint32_t w[PL / 2];
};
template <int PL, int W>
__device__ __forceinline__ void load_packed(const __nv_bfloat16* row, int sl, PackedShare<PL>& x) {
  if constexpr (PL < 4) {
    x.w[0] = *reinterpret_cast<const uint32_t*>(row + 2 * sl);
  } else {
#pragma unroll
    for (int c = 0; c < PL / 4; ++c) {
      const uint2 r = *reinterpret_cast<const uint2*>(row + 4 * W * c + 4 * sl);
      x.w[2 * c] = r.x;
      x.w[2 * c + 1] = r.y;
    }
  }
}
template <int PL>
__device__ __forceinline__ float packed_at(const PackedShare<PL>& x, int e) {
  return __uint_as_float((e & 1) ? (x.w[e >> 1] & 0xffff0000u) : (x.w[e >> 1] << 16));
}

// Row solve.  The lists the sweep leaves are deterministic (a row's candidates and their order depend on the 32 rows its warp
// scanned together and on nothing that varies from call to call), so a threshold iterated on the whole list is reproducible to
// the bit.
constexpr float kBoundMargin = 4e-6f;   // rounding of the bound the sweep ended with

// Threshold of Eq. 1 on the n <= K list entries of one row, by one thread with the entries in registers (n = 0: a lane without
// a row, which only takes part in the votes); the list is left compacted to the support, y in Eq. 1's units.  Newton from the
// left starting at the bound the sweep ended with (e < 1: bracketed, tau_iter_update).  Sums over a row need no shuffles this
// way: eight to thirty-two lanes per row spent two chains of them on every iteration, or sorted the list first (alpha = 1.25,
// 16 x 20011 x 128: 580 + 92 us with the long rows -> 227 + 66; alpha = 1.5, 16 x 32768 x 128: 222 + 105 -> 255 + 32 by this
// step alone, 168 + 22 with the gathers of the kernels below as they are now).
template <int K, int EC>
__device__ __forceinline__ int solve_row(const Problem& p, Entry* list, int n, float a, float bound, float& tau) {
  float y[K];
  float ymax = -INFINITY;
#pragma unroll
  for (int e = 0; e < K; e += 2) {
    float4 q = make_float4(-INFINITY, 0.f, -INFINITY, 0.f);
    if (e < n) q = *reinterpret_cast<const float4*>(list + e);     // {y, j, y, j}
    y[e] = e < n ? a * q.x : -INFINITY;
    y[e + 1] = e + 1 < n ? a * q.z : -INFINITY;
    ymax = fmaxf(ymax, fmaxf(y[e], y[e + 1]));
  }
  TauIter st = tau_iter_start(ymax);
  st.tau = st.lo = fmaxf(st.lo, bound);
  bool done = n == 0;
  for (int it = 0; it < kMaxNewton; ++it) {
    float s0[2] = {0.f, 0.f}, s1[2] = {0.f, 0.f};
#pragma unroll
    for (int e = 0; e < K; ++e) {
      const float d = fmaxf(y[e] - st.tau, 0.f);
      float ye, ye1;
      pow_pair_c<EC>(d, d > 0.f, p.expo, ye, ye1);
      s0[e & 1] += ye;
      s1[e & 1] += ye1;
    }
    if (!done) done = !tau_iter_update(st, s0[0] + s0[1], s1[0] + s1[1], p.expo_class, p.expo, 1e-7f);
    if (__all_sync(0xffffffffu, done)) break;
  }
  tau = st.tau;
  int cnt = 0;
#pragma unroll
  for (int e = 0; e < K; ++e) {
    if (e < n && y[e] > tau) {
      Entry en;
      en.y = y[e];
      en.j = list[e].j;
      list[cnt++] = en;
    }
  }
  return cnt;
}

// O_i of 32 / W rows at once, W lanes per row, from the supports solve_row left (cnt <= W entries; a row without any, whose
// y_max - 1 rounds to y_max, gets zeros; not active: no row, cnt = 0).
template <int D, int W, int EC>
__device__ __forceinline__ void gather_rows(const Problem& p, const __nv_bfloat16* __restrict__ v,
                                            const Entry* __restrict__ entries, __nv_bfloat16* __restrict__ o, int grow,
                                            bool active, int cnt, float tau, int lane) {
  constexpr int PL = D / W;                        // elements of a V / O row per lane
  constexpr int kBatch = 4;                        // V rows in flight
  const int sl = lane & (W - 1);
  const int base = lane & (32 - W);
  const int bh = grow / p.N, i = grow - bh * p.N, b = bh / p.H, h = bh - b * p.H;
  float pe = 0.f;
  int j = 0;
  if (sl < cnt) {
    const Entry en = entries[(size_t)grow * kListCap + sl];
    float pe1;
    pow_pair_c<EC>(en.y - tau, true, p.expo, pe, pe1);
    j = en.j;
  }
  float acc[PL];
#pragma unroll
  for (int t = 0; t < PL; ++t) acc[t] = 0.f;
  const size_t hbase = (size_t)b * p.sb + (size_t)h * p.sh;
#pragma unroll 1
  for (int t0 = 0; t0 < W; t0 += kBatch) {
    if (!__any_sync(0xffffffffu, t0 < cnt)) break;
    PackedShare<PL> vs[kBatch];
    float pj[kBatch];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      pj[u] = __shfl_sync(0xffffffffu, pe, base + t0 + u);
      const int kj = __shfl_sync(0xffffffffu, j, base + t0 + u);
#pragma unroll
      for (int e = 0; e < PL / 2; ++e) vs[u].w[e] = 0u;
      if (t0 + u < cnt) load_packed<PL, W>(v + hbase + (size_t)kj * p.sn, sl, vs[u]);
    }
#pragma unroll
    for (int u = 0; u < kBatch; ++u)
#pragma unroll
      for (int e = 0; e < PL; ++e) acc[e] = fmaf(pj[u], packed_at(vs[u], e), acc[e]);
  }
  if (active) store_share<PL, W>(o + hbase + (size_t)i * p.sn, sl, acc);
}

// One row with the whole warp, up to 32 S list entries: threshold, support, output.
template <int D, int S, int EC>
__device__ __forceinline__ void long_row(const Problem& p, const __nv_bfloat16* __restrict__ v, Entry* list, int n, float a,
                                         float bound, __nv_bfloat16* __restrict__ o, float* __restrict__ tau_slot,
                                         int32_t* __restrict__ cnt_slot, size_t hbase, int i, int lane) {
  constexpr int PER = D / 32;
  float y[S];
  int jj[S];
  float ymax = -INFINITY;
#pragma unroll
  for (int s = 0; s < S; ++s) {
    const int e = lane + 32 * s;
    y[s] = -INFINITY;
    jj[s] = 0;
    if (e < n) {
      const Entry en = list[e];
      y[s] = a * en.y;
      jj[s] = en.j;
    }
    ymax = fmaxf(ymax, y[s]);
  }
  ymax = warp_max(ymax);
  __syncwarp();   // every entry is in registers before the list is overwritten
  TauIter st = tau_iter_start(ymax);
  st.tau = st.lo = fmaxf(st.lo, bound);
  for (int it = 0; it < kMaxNewton; ++it) {
    float s0 = 0.f, s1 = 0.f;
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const float d = fmaxf(y[s] - st.tau, 0.f);
      float ye, ye1;
      pow_pair_c<EC>(d, d > 0.f, p.expo, ye, ye1);
      s0 += ye;
      s1 += ye1;
    }
    s0 = warp_sum(s0);
    s1 = warp_sum(s1);
    if (!tau_iter_update(st, s0, s1, p.expo_class, p.expo, 1e-7f)) break;
  }
  const float tau = st.tau;
  float acc[PER];
#pragma unroll
  for (int t = 0; t < PER; ++t) acc[t] = 0.f;
  int kept = 0;
#pragma unroll
  for (int s = 0; s < S; ++s) {
    const float d = fmaxf(y[s] - tau, 0.f);
    float pe, pe1;
    pow_pair_c<EC>(d, d > 0.f, p.expo, pe, pe1);
    unsigned m = __ballot_sync(0xffffffffu, d > 0.f);
    if (d > 0.f) {
      const int pos = kept + __popc(m & ((1u << lane) - 1u));
      list[pos].y = y[s];
      list[pos].j = jj[s];
    }
    kept += __popc(m);
    while (m) {
      // eight V rows in flight
      PackedShare<PER> vs[8];
      float pj[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int src = m ? __ffs(m) - 1 : 0;
        const int kj = __shfl_sync(0xffffffffu, jj[s], src);
        pj[u] = __shfl_sync(0xffffffffu, pe, src);
        if (!m) pj[u] = 0.f;
#pragma unroll
        for (int t = 0; t < PER / 2; ++t) vs[u].w[t] = 0u;
        if (m) load_packed<PER, 32>(v + hbase + (size_t)kj * p.sn, lane, vs[u]);
        m &= m - 1;
      }
#pragma unroll
      for (int u = 0; u < 8; ++u)
#pragma unroll
        for (int t = 0; t < PER; ++t) acc[t] = fmaf(pj[u], packed_at(vs[u], t), acc[t]);
    }
  }
  store_share<PER, 32>(o + hbase + (size_t)i * p.sn, lane, acc);
  if (lane == 0) {
    *tau_slot = tau;
    *cnt_slot = kept;
  }
}

// Rows with more than kLongRow list entries take the whole warp for a long time each (two-stage solves, gathers over
// dozens of keys) and come in runs -- the start of every causal head, where all visible keys are candidates.  A
// warp that met sixteen of them in its block would work through them one after the other while the rest of the grid
// has finished, so they are only listed here (from the far end of the dense-row list, which has a slot for every
// row) and a second launch gives each of them a warp of its own.  kLongCounter: their count, in the counter block
// that starts at fb_count.
constexpr int kLongCounter = 56;
constexpr int kLongRow = 32;   // list entries from which a row counts as long
__device__ __forceinline__ void push_long_rows(unsigned mask, int grow, int total, int32_t* fb_count, int32_t* fb_list,
                                               int lane) {
  if (mask == 0u) return;
  const int leader = __ffs(mask) - 1;
  int base = 0;
  if (lane == leader) base = atomicAdd(fb_count + kLongCounter, __popc(mask));
  base = __shfl_sync(0xffffffffu, base, leader);
  if ((mask >> lane) & 1u) fb_list[total - 1 - (base + __popc(mask & ((1u << lane) - 1u)))] = grow;
}

// The rows of a warp that go to the dense-tile path (mask over the warp's lanes, lane l holding row `grow`): one status
// update for all of them -- a counter bumped once per row is a chain of dependent L2 atomics on one address --, their
// 128-row Q tiles listed once (tile_flag arbitrates; of the lanes that name the same tile only the lowest asks) and, where
// tile_mask is given, the rows marked in it.
__device__ __forceinline__ void push_dense_tiles(const Problem& p, unsigned mask, int grow, uint32_t* tile_mask,
                                                 int32_t* tile_flag, int32_t* tile_list, int32_t* tile_count,
                                                 int32_t* status, int lane) {
  if (mask == 0u) return;
  if (status && lane == __ffs(mask) - 1) atomicAdd(status + ENTMAX_ATTN_STATUS_DENSE_ROWS, __popc(mask));
  if ((mask >> lane) & 1u) {
    const int tiles_per_head = (p.N + 127) / 128;
    const int bh = grow / p.N, i = grow - bh * p.N;
    const int id = bh * tiles_per_head + i / 128, r = i % 128;
    const unsigned same = __match_any_sync(mask, id);
    if (lane == __ffs(same) - 1 && atomicExch(tile_flag + id, 1) == 0) tile_list[atomicAdd(tile_count, 1)] = id;
    if (tile_mask) {
      const unsigned word = __match_any_sync(mask, 4 * id + (r >> 5));
      const unsigned bits = __reduce_or_sync(word, 1u << (r & 31));
      if (lane == __ffs(word) - 1) atomicOr(tile_mask + 4 * (size_t)id + (r >> 5), bits);
    }
  }
}

// The rows row_fwd_kernel listed as long (push_long_rows): one warp per row.
template <int D, int EC>
__global__ void __launch_bounds__(kWarpsPerCta * 32, 4) row_fwd_long_kernel(Problem p, const __nv_bfloat16* __restrict__ v,
                                                                         const float* __restrict__ scale,
                                                                         int32_t* __restrict__ row_cnt,
                                                                         const int32_t* __restrict__ list_cnt,
                                                                         const float* __restrict__ list_thr,
                                                                         Entry* __restrict__ entries,
                                                                         __nv_bfloat16* __restrict__ o,
                                                                         float* __restrict__ tau_out,
                                                                         const int32_t* __restrict__ fb_count,
                                                                         const int32_t* __restrict__ fb_list) {
  pdl_begin();
  const int lane = threadIdx.x & 31;
  const int total = p.B * p.H * p.N;
  const int n_long = fb_count[kLongCounter];
  for (int t = blockIdx.x * kWarpsPerCta + (threadIdx.x >> 5); t < n_long; t += gridDim.x * kWarpsPerCta) {
    const int grow = fb_list[total - 1 - t];
    const int n = list_cnt[2 * (size_t)grow];
    const int bh = grow / p.N, i = grow - bh * p.N, b = bh / p.H, h = bh - b * p.H;
    const float a = (p.alpha - 1.0f) * (scale[(size_t)b * p.scale_sb + (size_t)h * p.N + i] * p.sm_scale);
    float bound = list_thr[grow];
    bound -= kBoundMargin * fmaxf(1.0f, fabsf(bound));
    Entry* list = entries + (size_t)grow * kListCap;
    const size_t hbase = (size_t)b * p.sb + (size_t)h * p.sh;
    if (n <= 64) long_row<D, 2, EC>(p, v, list, n, a, bound, o, tau_out + grow, row_cnt + grow, hbase, i, lane);
    else if (n <= 128) long_row<D, 4, EC>(p, v, list, n, a, bound, o, tau_out + grow, row_cnt + grow, hbase, i, lane);
    else long_row<D, kSlots, EC>(p, v, list, n, a, bound, o, tau_out + grow, row_cnt + grow, hbase, i, lane);
  }
}

// (register cap: as for row_bwd_kernel.  Without one the solve takes 127 registers and two CTAs fill an SM: 47 us against 37
// now on 8 x 12 x 1024 x 64, 152 against 120 on 4 x 16 x 8192 x 64; at head_dim 128 227 against 212 on 16 x 20011)
template <int D, int EC>
__global__ void __launch_bounds__(kWarpsPerCta * 32, D == 64 ? 4 : 3) row_fwd_kernel(Problem p, const __nv_bfloat16* __restrict__ v,
                                                                    const float* __restrict__ scale,
                                                                    int32_t* __restrict__ row_cnt,
                                                                    const int32_t* __restrict__ list_cnt,
                                                                    const float* __restrict__ list_thr,
                                                                    Entry* __restrict__ entries,
                                                                    __nv_bfloat16* __restrict__ o,
                                                                    float* __restrict__ tau_out, int32_t* fb_count,
                                                                    int32_t* fb_list, int32_t* tile_flag,
                                                                    int32_t* tile_list, int32_t* tile_count,
                                                                    int32_t* status, int rpw) {
  pdl_begin();
  const int lane = threadIdx.x & 31;
  const int total = p.B * p.H * p.N;
  const int blocks = (total + rpw - 1) / rpw;
  for (int blk = blockIdx.x * kWarpsPerCta + (threadIdx.x >> 5); blk < blocks; blk += gridDim.x * kWarpsPerCta) {
    // A warp takes rpw (32, 16 or 8) consecutive rows; lane l looks at row rpw*blk + l and solves it.  The rows' outputs are
    // then gathered by support size: four rows at a time with eight lanes each (up to 8 entries), two with sixteen (up to
    // 16), one with the whole warp.
    const int my_row = lane < rpw ? rpw * blk + lane : total;
    int n = 0;
    if (my_row < total) n = list_cnt[2 * (size_t)my_row];
    {
      // rows without a usable list go to the dense-tile path, all of the warp's at once, the ones with long lists to a
      // launch of their own
      const unsigned mdense = __ballot_sync(0xffffffffu, my_row < total && n < 1);
      push_dense_tiles(p, mdense, my_row, nullptr, tile_flag, tile_list, tile_count, status, lane);
      if ((mdense >> lane) & 1u) row_cnt[my_row] = -2;
      const unsigned mlong = __ballot_sync(0xffffffffu, n > kLongRow);
      push_long_rows(mlong, my_row, total, fb_count, fb_list, lane);
      if (n < 0 || n > kLongRow) n = 0;
    }
    float a = 1.0f, bound = -INFINITY, tau = 0.f;
    if (n > 0) {
      const int bh = my_row / p.N, i = my_row - bh * p.N, b = bh / p.H, h = bh - b * p.H;
      a = (p.alpha - 1.0f) * (scale[(size_t)b * p.scale_sb + (size_t)h * p.N + i] * p.sm_scale);
      bound = list_thr[my_row];
      bound -= kBoundMargin * fmaxf(1.0f, fabsf(bound));
    }
    Entry* list = entries + (size_t)(my_row < total ? my_row : 0) * kListCap;
    const int n_max = __reduce_max_sync(0xffffffffu, n);
    int cnt = 0;
    if (n_max > 16) cnt = solve_row<32, EC>(p, list, n, a, bound, tau);
    else if (n_max > 8) cnt = solve_row<16, EC>(p, list, n, a, bound, tau);
    else if (n_max > 0) cnt = solve_row<8, EC>(p, list, n, a, bound, tau);
    if (n > 0) {
      tau_out[my_row] = tau;
      row_cnt[my_row] = cnt;
    }
    __syncwarp();   // the supports are ordered before the other lanes' loads
    unsigned m8 = __ballot_sync(0xffffffffu, n > 0 && cnt <= 8);
    unsigned m16 = __ballot_sync(0xffffffffu, cnt > 8 && cnt <= 16);
    unsigned m32 = __ballot_sync(0xffffffffu, cnt > 16);
    while (m8) {
      const unsigned src = __fns(m8, 0, (lane >> 3) + 1);        // the row of this group of eight lanes
      const bool active = src < 32u;
      const int c = __shfl_sync(0xffffffffu, cnt, active ? src : 0);
      const float t = __shfl_sync(0xffffffffu, tau, active ? src : 0);
      gather_rows<D, 8, EC>(p, v, entries, o, active ? rpw * blk + (int)src : 0, active, active ? c : 0, t, lane);
#pragma unroll
      for (int z = 0; z < 4; ++z) m8 &= m8 - 1;
    }
    while (m16) {
      const unsigned src = __fns(m16, 0, (lane >> 4) + 1);
      const bool active = src < 32u;
      const int c = __shfl_sync(0xffffffffu, cnt, active ? src : 0);
      const float t = __shfl_sync(0xffffffffu, tau, active ? src : 0);
      gather_rows<D, 16, EC>(p, v, entries, o, active ? rpw * blk + (int)src : 0, active, active ? c : 0, t, lane);
      m16 &= m16 - 1;
      m16 &= m16 - 1;
    }
    while (m32) {
      const int src = __ffs(m32) - 1;
      m32 &= m32 - 1;
      const int c = __shfl_sync(0xffffffffu, cnt, src);
      const float t = __shfl_sync(0xffffffffu, tau, src);
      gather_rows<D, 32, EC>(p, v, entries, o, rpw * blk + src, true, c, t, lane);
    }
  }
}

// Backward of one row with the whole warp, for rows with at most 32 S list entries: entry e on lane e mod 32, the row's
// elements split over the 32 lanes.  Bound by the latency of the gathers: four V rows, then four K rows are in flight
// (packed), and four sums share one butterfly.  Float rows and a reduction each -> now: 2 x 12 x 3001 x 64 73 -> 60 us,
// 8 x 65536 x 64 (retrieval) 182 -> 137, 16 x 32768 x 128 36 -> 27.  Eight rows in flight need more registers, and with
// three CTAs on an SM instead of four lose more than they gain: 82 and 215 us.
template <int D, int S>
__device__ __forceinline__ void bwd_row_wide(const Problem& p, const __nv_bfloat16* __restrict__ q,
                                             const __nv_bfloat16* __restrict__ k, const __nv_bfloat16* __restrict__ v,
                                             const __nv_bfloat16* __restrict__ d_o, const float* __restrict__ scale,
                                             const float* __restrict__ tau_in, const Entry* __restrict__ entries,
                                             __nv_bfloat16* __restrict__ dq, float* __restrict__ acc_dk,
                                             float* __restrict__ acc_dv, float* __restrict__ dc_rows, int grow, int n,
                                             bool saved, int pitch, int lane) {
  constexpr int PL = D / 32;                       // elements of a row per lane
  constexpr int kBatch = 4;
  const int bh = grow / p.N, i = grow - bh * p.N, b = bh / p.H, h = bh - b * p.H;
  const float g = scale[(size_t)b * p.scale_sb + (size_t)h * p.N + i] * p.sm_scale;
  const float a = (p.alpha - 1.0f) * g;
  const float tau = tau_in[grow];
  const size_t hbase = (size_t)b * p.sb + (size_t)h * p.sh;
  PackedShare<PL> qs, gs;
  load_packed<PL, 32>(q + hbase + (size_t)i * p.sn, lane, qs);
  load_packed<PL, 32>(d_o + hbase + (size_t)i * p.sn, lane, gs);
  const Entry* list = entries + (size_t)grow * pitch;
  float yv[S], zz[S], dpv[S];
  int jj[S];
  unsigned in[S];
#pragma unroll
  for (int s = 0; s < S; ++s) {
    yv[s] = -1.0f;
    zz[s] = 0.f;
    dpv[s] = 0.f;
    jj[s] = 0;
    if (lane + 32 * s < n) {
      const Entry en = list[lane + 32 * s];
      // a list saved by the forward pass holds y = (alpha-1) s in Eq. 1's units, a fresh one raw <q_i, k_j>
      yv[s] = saved ? en.y - tau : fmaf(a, en.y, -tau);
      jj[s] = en.j;
      zz[s] = saved ? en.y / a : en.y;               // raw <q_i, k_j>
    }
    in[s] = __ballot_sync(0xffffffffu, yv[s] > 0.f);
  }
  auto load_batch = [&](const __nv_bfloat16* rows, int j, unsigned rest, int t0, PackedShare<PL> (&x)[kBatch]) {
#pragma unroll
    for (int z = 0; z < kBatch; ++z) {
      const int kj = __shfl_sync(0xffffffffu, j, t0 + z);
#pragma unroll
      for (int w = 0; w < PL / 2; ++w) x[z].w[w] = 0u;
      if ((rest >> z) & 1u) load_packed<PL, 32>(rows + hbase + (size_t)kj * p.sn, lane, x[z]);
    }
  };
  // dP_ij = <dO_i, v_j> on the support
#pragma unroll
  for (int s = 0; s < S; ++s) {
#pragma unroll 1
    for (int t0 = 0; t0 < 32; t0 += kBatch) {
      const unsigned rest = in[s] >> t0;
      if (rest == 0u) break;
      PackedShare<PL> vs[kBatch];
      load_batch(v, jj[s], rest, t0, vs);
      float dp[kBatch];
#pragma unroll
      for (int z = 0; z < kBatch; ++z) {
        dp[z] = 0.f;
#pragma unroll
        for (int e = 0; e < PL; ++e) dp[z] = fmaf(packed_at(gs, e), packed_at(vs[z], e), dp[z]);
      }
      // the batch's sums over the warp in one butterfly: lane l ends up with the one of slot t0 + l mod kBatch
#pragma unroll
      for (int o = 1; o < kBatch; o <<= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int z = 0; z < kBatch; z += 2 * o)
          dp[z] = (up ? dp[z + o] : dp[z]) + __shfl_xor_sync(0xffffffffu, up ? dp[z] : dp[z + o], o);
      }
      float r = dp[0];
#pragma unroll
      for (int o = kBatch; o < 32; o <<= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
      if ((lane & ~(kBatch - 1)) == t0) dpv[s] = r;
    }
  }
  float pe[S], u[S];
  float su = 0.f, sud = 0.f;
#pragma unroll
  for (int s = 0; s < S; ++s) {
    pe[s] = 0.f;
    u[s] = 0.f;
    if (yv[s] > 0.f) pow_pair(yv[s], p.expo_class, p.expo, pe[s], u[s]);
    su += u[s];
    sud += u[s] * dpv[s];
  }
  su = warp_sum(su);
  sud = warp_sum(sud);
  const float rho = su > 0.f ? sud / su : 0.f;
  if (dc_rows) {
    // dL/dc_i = sum_j dS_ij z_ij with z_ij = <q_i,k_j> sm_scale (chain rule through s = c z)
    float dc = 0.f;
#pragma unroll
    for (int s = 0; s < S; ++s) dc = fmaf(u[s] * (dpv[s] - rho), zz[s], dc);
    dc = warp_sum(dc);
    if (lane == 0) dc_rows[grow] = dc * p.sm_scale;
  }
  float acc[PL];
#pragma unroll
  for (int t = 0; t < PL; ++t) acc[t] = 0.f;
  const size_t arow = (size_t)bh * p.N;
#pragma unroll
  for (int s = 0; s < S; ++s) {
    const float gds_own = g * u[s] * (dpv[s] - rho);
#pragma unroll 1
    for (int t0 = 0; t0 < 32; t0 += kBatch) {
      const unsigned rest = in[s] >> t0;
      if (rest == 0u) break;
      PackedShare<PL> ks[kBatch];
      load_batch(k, jj[s], rest, t0, ks);
#pragma unroll
      for (int z = 0; z < kBatch; ++z) {
        const int kj = __shfl_sync(0xffffffffu, jj[s], t0 + z);
        const float gds = __shfl_sync(0xffffffffu, gds_own, t0 + z);
        const float pj = __shfl_sync(0xffffffffu, pe[s], t0 + z);
        if ((rest >> z) & 1u) {
          float x[PL];
#pragma unroll
          for (int e = 0; e < PL; ++e) {
            acc[e] = fmaf(gds, packed_at(ks[z], e), acc[e]);
            x[e] = gds * packed_at(qs, e);
          }
          add_share<PL, 32>(acc_dk + (arow + kj) * D, lane, x);
#pragma unroll
          for (int e = 0; e < PL; ++e) x[e] = pj * packed_at(gs, e);
          add_share<PL, 32>(acc_dv + (arow + kj) * D, lane, x);
        }
      }
    }
  }
  store_share<PL, 32>(dq + hbase + (size_t)i * p.sn, lane, acc);
}

// Backward of 32 / W rows at once, W lanes per row (W = 8 or 16), for rows with at most W list entries.  Bound by the
// latency of the gathers: four V rows, then four (head_dim 64) or two K rows are in flight at a time, and q_i, dO_i and
// the gathered rows stay packed until they are used (as floats batches of four spill).  One row at a time before ->
// now: 8 x 12 x 1024 x 64 74 -> 57 us, 4 x 16 x 8192 x 64 281 -> 217, 16 x 32768 x 128 632 -> 570.
template <int D, int W>
__device__ __forceinline__ void bwd_rows_sub(const Problem& p, const __nv_bfloat16* __restrict__ q,
                                             const __nv_bfloat16* __restrict__ k, const __nv_bfloat16* __restrict__ v,
                                             const __nv_bfloat16* __restrict__ d_o, const float* __restrict__ scale,
                                             const float* __restrict__ tau_in, const Entry* __restrict__ entries,
                                             __nv_bfloat16* __restrict__ dq, float* __restrict__ acc_dk,
                                             float* __restrict__ acc_dv, float* __restrict__ dc_rows, int grow,
                                             bool active, int n_list, bool saved, int pitch, int lane) {
  constexpr int PL = D / W;                        // elements of a row per lane
  constexpr int kBatch = PL <= 8 ? 4 : 2;          // rows in flight
  constexpr unsigned kWMask = (1u << W) - 1u;
  const int sl = lane & (W - 1);
  const int base = lane & (32 - W);
  const int n = active ? n_list : 0;
  const int bh = grow / p.N, i = grow - bh * p.N, b = bh / p.H, h = bh - b * p.H;
  const float g = active ? scale[(size_t)b * p.scale_sb + (size_t)h * p.N + i] * p.sm_scale : 0.f;
  const float a = (p.alpha - 1.0f) * g;
  const float tau = active ? tau_in[grow] : 0.f;
  const size_t hbase = (size_t)b * p.sb + (size_t)h * p.sh;
  PackedShare<PL> qs, gs;
  load_packed<PL, W>(q + hbase + (size_t)i * p.sn, sl, qs);
  load_packed<PL, W>(d_o + hbase + (size_t)i * p.sn, sl, gs);
  const Entry* list = entries + (size_t)grow * pitch;
  float yv = -1.0f, zz = 0.f;
  int j = 0;
  if (sl < n) {
    const Entry en = list[sl];
    // a list saved by the forward pass holds y = (alpha-1) s in Eq. 1's units, a fresh one raw <q_i, k_j>
    yv = saved ? en.y - tau : fmaf(a, en.y, -tau);
    j = en.j;
    zz = saved ? en.y / a : en.y;                  // raw <q_i, k_j>
  }
  const bool in = yv > 0.f;
  const unsigned msub = (__ballot_sync(0xffffffffu, in) >> base) & kWMask;
  // slots of the fullest row of the warp
  const int last = 32 - __clz(__reduce_or_sync(0xffffffffu, msub));
  // dP_ij = <dO_i, v_j> on the support.  (A slot without an entry names key 0: its row is loaded and the product dropped.)
  float dpv = 0.f;
#pragma unroll 1
  for (int t0 = 0; t0 < last; t0 += kBatch) {
    PackedShare<PL> vs[kBatch];
#pragma unroll
    for (int z = 0; z < kBatch; ++z)
      load_packed<PL, W>(v + hbase + (size_t)__shfl_sync(0xffffffffu, j, base + t0 + z) * p.sn, sl, vs[z]);
    float dp[kBatch];
#pragma unroll
    for (int z = 0; z < kBatch; ++z) {
      dp[z] = 0.f;
#pragma unroll
      for (int e = 0; e < PL; ++e) dp[z] = fmaf(packed_at(gs, e), packed_at(vs[z], e), dp[z]);
    }
    // the batch's sums over the row's lanes in one butterfly: lane sl ends up with the one of slot t0 + sl mod kBatch
    const bool odd = sl & 1;
    float r = (odd ? dp[1] : dp[0]) + __shfl_xor_sync(0xffffffffu, odd ? dp[0] : dp[1], 1);
    if constexpr (kBatch == 4) {
      const float s23 = (odd ? dp[3] : dp[2]) + __shfl_xor_sync(0xffffffffu, odd ? dp[2] : dp[3], 1);
      const bool upper = sl & 2;
      r = (upper ? s23 : r) + __shfl_xor_sync(0xffffffffu, upper ? r : s23, 2);
    }
#pragma unroll
    for (int o = kBatch; o < W; o <<= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    if ((sl & ~(kBatch - 1)) == t0) dpv = r;
  }
  float pe = 0.f, u = 0.f;
  if (in) pow_pair(yv, p.expo_class, p.expo, pe, u);
  else dpv = 0.f;
  const float su = sub_sum<W>(u), sud = sub_sum<W>(u * dpv);
  const float rho = su > 0.f ? sud / su : 0.f;
  const float gds_own = g * u * (dpv - rho);
  if (dc_rows) {
    // dL/dc_i = sum_j dS_ij z_ij with z_ij = <q_i,k_j> sm_scale (chain rule through s = c z)
    const float dc = sub_sum<W>(u * (dpv - rho) * zz);
    if (active && sl == 0) dc_rows[grow] = dc * p.sm_scale;
  }
  float acc[PL];
#pragma unroll
  for (int t = 0; t < PL; ++t) acc[t] = 0.f;
  const size_t arow = (size_t)bh * p.N;
#pragma unroll 1
  for (int t0 = 0; t0 < last; t0 += kBatch) {
    PackedShare<PL> ks[kBatch];
#pragma unroll
    for (int z = 0; z < kBatch; ++z)
      load_packed<PL, W>(k + hbase + (size_t)__shfl_sync(0xffffffffu, j, base + t0 + z) * p.sn, sl, ks[z]);
#pragma unroll
    for (int z = 0; z < kBatch; ++z) {
      const int kj = __shfl_sync(0xffffffffu, j, base + t0 + z);
      const float gds = __shfl_sync(0xffffffffu, gds_own, base + t0 + z);
      const float pj = __shfl_sync(0xffffffffu, pe, base + t0 + z);
      if ((msub >> (t0 + z)) & 1u) {
        float* dk_row = acc_dk + (arow + kj) * D + 4 * sl;
        float* dv_row = acc_dv + (arow + kj) * D + 4 * sl;
#pragma unroll
        for (int c = 0; c < PL / 4; ++c) {
#pragma unroll
          for (int e = 4 * c; e < 4 * c + 4; ++e) acc[e] = fmaf(gds, packed_at(ks[z], e), acc[e]);
          red_add_v4(dk_row + 4 * W * c, gds * packed_at(qs, 4 * c), gds * packed_at(qs, 4 * c + 1),
                     gds * packed_at(qs, 4 * c + 2), gds * packed_at(qs, 4 * c + 3));
          red_add_v4(dv_row + 4 * W * c, pj * packed_at(gs, 4 * c), pj * packed_at(gs, 4 * c + 1),
                     pj * packed_at(gs, 4 * c + 2), pj * packed_at(gs, 4 * c + 3));
        }
      }
    }
  }
  if (active) store_share<PL, W>(dq + hbase + (size_t)i * p.sn, sl, acc);
}

// (register cap: this kernel waits on gathers and reductions, warps are what hides them.  Four CTAs per SM at head_dim 64,
// where three take 60 us instead of 57 on 8 x 12 x 1024; three at 128, where the cap of four spills: 640 us against 570 on
// 16 x 32768)
template <int D>
__global__ void __launch_bounds__(kWarpsPerCta * 32, D == 64 ? 4 : 3) row_bwd_kernel(
    Problem p, const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ k,
    const __nv_bfloat16* __restrict__ v, const __nv_bfloat16* __restrict__ d_o, const float* __restrict__ scale,
    const float* __restrict__ tau_in, const int32_t* __restrict__ list_cnt, const Entry* __restrict__ entries,
    __nv_bfloat16* __restrict__ dq, float* __restrict__ acc_dk, float* __restrict__ acc_dv,
    float* __restrict__ dc_rows, int32_t* fb_count, int32_t* fb_list, uint32_t* tile_mask, int32_t* tile_flag,
    int32_t* tile_list, int32_t* tile_count, int32_t* status, int saved, int pitch, int rpw) {
  pdl_begin();
  // saved != 0: `list_cnt` is the forward pass's final support size per row (one int per row, -2 = dense
  // row) and `entries` its compacted support lists; `pitch` = list slots per row in `entries`
  const int lane = threadIdx.x & 31;
  const int total = p.B * p.H * p.N;
  const int blocks = (total + rpw - 1) / rpw;
  for (int blk = blockIdx.x * kWarpsPerCta + (threadIdx.x >> 5); blk < blocks; blk += gridDim.x * kWarpsPerCta) {
    // A warp takes rpw (16 or 8) consecutive rows; lane l (and l + 16) looks at row rpw*blk + l.  Rows are served by list
    // length: four at a time (<= 8 entries), two at a time (<= 16), one at a time (<= 32, or the long form).
    const int my_row = (lane & 15) < rpw ? rpw * blk + (lane & 15) : total;
    int mc = 0;
    int cls = 4;                                     // 0: <= 8 entries, 1: <= 16, 2: <= 32, 3: more / dense, 4: no row
    if (my_row < total) {
      mc = list_cnt[saved ? (size_t)my_row : 2 * (size_t)my_row];
      cls = (mc < 0 || mc > 32) ? 3 : mc <= 8 ? 0 : mc <= 16 ? 1 : 2;
    }
    unsigned m8 = __ballot_sync(0xffffffffu, lane < 16 && cls == 0);
    unsigned m16 = __ballot_sync(0xffffffffu, lane < 16 && cls == 1);
    unsigned m32 = __ballot_sync(0xffffffffu, lane < 16 && cls == 2);
    unsigned mlong = __ballot_sync(0xffffffffu, lane < 16 && cls == 3);
    {
      // rows without a usable list go to the dense path, all of the warp's at once
      const unsigned mdense = __ballot_sync(0xffffffffu, lane < 16 && my_row < total && mc < 0);
      push_dense_tiles(p, mdense, my_row, tile_mask, tile_flag, tile_list, tile_count, status, lane);
      mlong &= ~mdense;
      // ... and the ones with long lists to a launch of their own (see push_long_rows)
      push_long_rows(mlong | m32, my_row, total, fb_count, fb_list, lane);
    }
    while (m8) {
      const unsigned src = __fns(m8, 0, (lane >> 3) + 1);          // the row of this group of eight lanes
      const bool active = src < 32u;
      const int n_list = __shfl_sync(0xffffffffu, mc, active ? src : 0);
      bwd_rows_sub<D, 8>(p, q, k, v, d_o, scale, tau_in, entries, dq, acc_dk, acc_dv, dc_rows,
                         active ? rpw * blk + (int)src : 0, active, n_list, saved != 0, pitch, lane);
#pragma unroll
      for (int t = 0; t < 4; ++t) m8 &= m8 - 1;
    }
    while (m16) {
      const unsigned src = __fns(m16, 0, (lane >> 4) + 1);
      const bool active = src < 32u;
      const int n_list = __shfl_sync(0xffffffffu, mc, active ? src : 0);
      bwd_rows_sub<D, 16>(p, q, k, v, d_o, scale, tau_in, entries, dq, acc_dk, acc_dv, dc_rows,
                          active ? rpw * blk + (int)src : 0, active, n_list, saved != 0, pitch, lane);
      m16 &= m16 - 1;
      m16 &= m16 - 1;
    }
  }
}

// The rows row_bwd_kernel listed as long (push_long_rows): one warp per row.
template <int D>
__global__ void __launch_bounds__(kWarpsPerCta * 32, 4) row_bwd_long_kernel(
    Problem p, const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ k,
    const __nv_bfloat16* __restrict__ v, const __nv_bfloat16* __restrict__ d_o, const float* __restrict__ scale,
    const float* __restrict__ tau_in, const int32_t* __restrict__ list_cnt, const Entry* __restrict__ entries,
    __nv_bfloat16* __restrict__ dq, float* __restrict__ acc_dk, float* __restrict__ acc_dv,
    float* __restrict__ dc_rows, const int32_t* __restrict__ fb_count, const int32_t* __restrict__ fb_list, int saved,
    int pitch) {
  pdl_begin();
  const int lane = threadIdx.x & 31;
  const int total = p.B * p.H * p.N;
  const int n_long = fb_count[kLongCounter];
  for (int t = blockIdx.x * kWarpsPerCta + (threadIdx.x >> 5); t < n_long; t += gridDim.x * kWarpsPerCta) {
    const int grow = fb_list[total - 1 - t];
    const int n_list = list_cnt[saved ? (size_t)grow : 2 * (size_t)grow];
#define ENTMAX_ROW_BWD_WIDE(S)                                                                                              \
  bwd_row_wide<D, S>(p, q, k, v, d_o, scale, tau_in, entries, dq, acc_dk, acc_dv, dc_rows, grow, n_list, saved != 0, pitch, \
                     lane)
    if (n_list <= 32) ENTMAX_ROW_BWD_WIDE(1);
    else if (n_list <= 64) ENTMAX_ROW_BWD_WIDE(2);
    else if (n_list <= 128) ENTMAX_ROW_BWD_WIDE(4);
    else ENTMAX_ROW_BWD_WIDE(kSlots);
#undef ENTMAX_ROW_BWD_WIDE
  }
}

// Copies every row's final support (at most `slots` entries) from the forward call's lists into a compact
// table; rows without a list, or with a longer one, get the count -2 and are recomputed by the backward pass.
// Eight lanes per row: most supports are one pass of them, and nothing is divided (a thread per slot of the table, with a
// 64-bit division each, took 65 us on 4 x 16 x 8192 rows; now 29).
__global__ void __launch_bounds__(256) save_supports_kernel(int rows, int slots, const int32_t* __restrict__ row_cnt,
                                                            const Entry* __restrict__ entries,
                                                            int32_t* __restrict__ out_cnt, Entry* __restrict__ out_entries) {
  pdl_begin();
  const int sub = threadIdx.x & 7;
  const int step = gridDim.x * 32;
  for (int row = blockIdx.x * 32 + (threadIdx.x >> 3); row < rows; row += step) {
    const int cnt = row_cnt[row];
    const bool fits = cnt >= 0 && cnt <= slots;
    if (sub == 0) out_cnt[row] = fits ? cnt : -2;
    if (fits)
      for (int slot = sub; slot < cnt; slot += 8)
        out_entries[(size_t)row * slots + slot] = entries[(size_t)row * kListCap + slot];
  }
}

// Rows per warp (forward up to 32, backward up to 16).  A warp works its rows off in rounds of dependent loads, so while the
// grid fits the machine at once its time is that of one warp: 8 rows per warp there (with 16: 8 x 12 x 1024 x 64 forward 50 ->
// 54 us, backward 74 -> 80).  More rows pack better into rounds and win where the grid is several waves long; 4 lose more in
// packing than they save (2 x 12 x 3001 x 64: 37 -> 47 and 93 -> 112 us).  (Compared before the gathers were packed, which
// shortened both sides.)
inline int rows_per_warp(const Problem& p, int most) {
  const long rows = (long)p.B * p.H * p.N;
  return rows >= 148L * 64 * most ? most : rows >= 148L * 64 * 16 ? 16 : 8;
}
inline int row_grid(const Problem& p, int rpw) {
  const long warps = ((long)p.B * p.H * p.N + rpw - 1) / rpw;
  const long ctas = (warps + kWarpsPerCta - 1) / kWarpsPerCta;
  const long cap = 148L * 8 * 8;
  return (int)(ctas < cap ? ctas : cap);
}

}  // namespace

cudaError_t launch_row_fwd(const Problem& p, const void* v, const float* scale, int32_t* row_cnt,
                           const int32_t* list_cnt, const float* list_thr, Entry* entries, void* o, float* tau,
                           int32_t* fb_count, int32_t* fb_list, int32_t* tile_flag, int32_t* tile_list,
                           int32_t* tile_count, int32_t* status, cudaStream_t stream) {
  const int rpw = rows_per_warp(p, 32);
  const int grid = row_grid(p, rpw);
#define ENTMAX_ROW_FWD(D, EC)                                                                                         \
  launch_kernel(row_fwd_kernel<D, EC>, grid, kWarpsPerCta * 32, 0, stream, p, (const __nv_bfloat16*)v, scale, row_cnt, list_cnt, \
                                                                list_thr, entries, (__nv_bfloat16*)o, tau, fb_count,  \
                                                                fb_list,                                              \
                                                                tile_flag, tile_list, tile_count, status, rpw)
  if (p.D == 64) {
    if (p.expo_class == kExpo2) ENTMAX_ROW_FWD(64, kExpo2);
    else if (p.expo_class == kExpo1) ENTMAX_ROW_FWD(64, kExpo1);
    else if (p.expo_class == kExpo4) ENTMAX_ROW_FWD(64, kExpo4);
    else ENTMAX_ROW_FWD(64, kExpoGeneral);
  } else {
    if (p.expo_class == kExpo2) ENTMAX_ROW_FWD(128, kExpo2);
    else if (p.expo_class == kExpo1) ENTMAX_ROW_FWD(128, kExpo1);
    else if (p.expo_class == kExpo4) ENTMAX_ROW_FWD(128, kExpo4);
    else ENTMAX_ROW_FWD(128, kExpoGeneral);
  }
#undef ENTMAX_ROW_FWD
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) return err;
  // the rows it listed as long, one warp each (normally none or a few: the launch then ends at once)
  const int lgrid = grid < 148 * 4 ? grid : 148 * 4;
#define ENTMAX_ROW_FWD_LONG(D, EC)                                                                                     \
  launch_kernel(row_fwd_long_kernel<D, EC>, lgrid, kWarpsPerCta * 32, 0, stream, p, (const __nv_bfloat16*)v, scale, row_cnt,       \
                                                                      list_cnt, list_thr, entries, (__nv_bfloat16*)o,  \
                                                                      tau, fb_count, fb_list)
  if (p.D == 64) {
    if (p.expo_class == kExpo2) ENTMAX_ROW_FWD_LONG(64, kExpo2);
    else if (p.expo_class == kExpo1) ENTMAX_ROW_FWD_LONG(64, kExpo1);
    else if (p.expo_class == kExpo4) ENTMAX_ROW_FWD_LONG(64, kExpo4);
    else ENTMAX_ROW_FWD_LONG(64, kExpoGeneral);
  } else {
    if (p.expo_class == kExpo2) ENTMAX_ROW_FWD_LONG(128, kExpo2);
    else if (p.expo_class == kExpo1) ENTMAX_ROW_FWD_LONG(128, kExpo1);
    else if (p.expo_class == kExpo4) ENTMAX_ROW_FWD_LONG(128, kExpo4);
    else ENTMAX_ROW_FWD_LONG(128, kExpoGeneral);
  }
#undef ENTMAX_ROW_FWD_LONG
  return cudaGetLastError();
}

cudaError_t launch_save_supports(const Problem& p, int slots, const int32_t* row_cnt, const Entry* entries,
                                 int32_t* out_cnt, Entry* out_entries, cudaStream_t stream) {
  const int rows = p.B * p.H * p.N;
  const int blocks = (rows + 31) / 32 < 148 * 32 ? (rows + 31) / 32 : 148 * 32;
  launch_kernel(save_supports_kernel, blocks, 256, 0, stream, rows, slots, row_cnt, entries, out_cnt, out_entries);
  return cudaGetLastError();
}

cudaError_t launch_row_bwd(const Problem& p, const void* q, const void* k, const void* v, const void* d_o,
                           const float* scale, const float* tau, const int32_t* list_cnt, Entry* entries, void* dq,
                           float* acc_dk, float* acc_dv, float* dc_rows, int32_t* fb_count, int32_t* fb_list,
                           uint32_t* tile_mask, int32_t* tile_flag, int32_t* tile_list, int32_t* tile_count, int32_t* status,
                           int saved, int pitch, cudaStream_t stream) {
  const int rpw = rows_per_warp(p, 16);
  const int grid = row_grid(p, rpw);
  if (p.D == 64)
    launch_kernel(row_bwd_kernel<64>, grid, kWarpsPerCta * 32, 0, stream, p, (const __nv_bfloat16*)q, (const __nv_bfloat16*)k, (const __nv_bfloat16*)v, (const __nv_bfloat16*)d_o, scale,
        tau, list_cnt, entries, (__nv_bfloat16*)dq, acc_dk, acc_dv, dc_rows, fb_count,
        fb_list, tile_mask, tile_flag, tile_list, tile_count, status, saved, pitch, rpw);
  else
    launch_kernel(row_bwd_kernel<128>, grid, kWarpsPerCta * 32, 0, stream, p, (const __nv_bfloat16*)q, (const __nv_bfloat16*)k, (const __nv_bfloat16*)v, (const __nv_bfloat16*)d_o, scale,
        tau, list_cnt, entries, (__nv_bfloat16*)dq, acc_dk, acc_dv, dc_rows, fb_count,
        fb_list, tile_mask, tile_flag, tile_list, tile_count, status, saved, pitch, rpw);
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) return err;
  // the rows it listed as long, one warp each (normally none or a few: the launch then ends at once)
  const int lgrid = grid < 148 * 4 ? grid : 148 * 4;
  if (p.D == 64)
    launch_kernel(row_bwd_long_kernel<64>, lgrid, kWarpsPerCta * 32, 0, stream, p, (const __nv_bfloat16*)q, (const __nv_bfloat16*)k, (const __nv_bfloat16*)v, (const __nv_bfloat16*)d_o, scale,
        tau, list_cnt, entries, (__nv_bfloat16*)dq, acc_dk, acc_dv, dc_rows, fb_count, fb_list, saved, pitch);
  else
    launch_kernel(row_bwd_long_kernel<128>, lgrid, kWarpsPerCta * 32, 0, stream, p, (const __nv_bfloat16*)q, (const __nv_bfloat16*)k, (const __nv_bfloat16*)v, (const __nv_bfloat16*)d_o, scale,
        tau, list_cnt, entries, (__nv_bfloat16*)dq, acc_dk, acc_dv, dc_rows, fb_count, fb_list, saved, pitch);
  return cudaGetLastError();
}

}  // namespace entmax
