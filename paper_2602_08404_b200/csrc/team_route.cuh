// Eq. 4's classification of a row, and the selection of a call of few rows inside the kernel that consumes it.
#pragma once

#include "team_common.cuh"
#include "team_topk.cuh"

namespace team {

__device__ __forceinline__ bool is_decoded(int s) { return s == TEAM_TOK_NEW || s == TEAM_TOK_CACHED; }

// What the walk over a run of rows reads of a row: ((group * 256 + branch) * 2 + decoded, position).  An index out of range is
// reported and clamped.
__device__ __forceinline__ int2 walk_entry(const StepPtrs& st, int t, int state, int G, int32_t* status) {
  int g = st.group[t], b = st.branch[t];
  if (g < 0 || g >= G || b < 0 || b > 255) {
    set_status(status, TEAM_ERR_STATE, 1);
    g = min(max(g, 0), G - 1);
    b = min(max(b, 0), 255);
  }
  return make_int2((g * 256 + b) * 2 + (is_decoded(state) ? 1 : 0), st.pos[t]);
}
__device__ __forceinline__ int walk_group(const int2& w) { return w.x >> 9; }

// Eq. 4 for row t, without the rule for groups that have no first-round row.
__device__ __forceinline__ int classify_row(const int2* walk, int t, int T, int state, float conf, const Policy& p, int32_t* status) {
  if (state == TEAM_TOK_CACHED) return (p.flags & TEAM_F_DCD) ? TEAM_CLS_SKIP : TEAM_CLS_FIRST;
  if (state == TEAM_TOK_NEW || !(p.flags & TEAM_F_LAC)) return TEAM_CLS_FIRST;
  const int key = walk[t].x >> 1, mypos = walk[t].y;
  const int lim = p.inclusive ? p.L_hot : p.L_hot - 1;   // |pos - j| <= lim
  bool hot = conf > p.tau_hot;
  if (p.prefix_decoded && mypos + 1 <= lim) hot = true;
  // the row's own run, first downwards, then upwards, four rows per step (their loads overlap: one by one a block
  // of 32 took 9600 clock cycles)
#pragma unroll 1
  for (int dir = -1; dir <= 1 && !hot; dir += 2) {
    bool inside = true;
#pragma unroll 1
    for (int o = 1; inside && !hot; o += 4) {           // offsets 1-4, ..., 61-64, then the check
      int2 w[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int u = t + dir * (o + q);
        w[q] = walk[min(max(u, 0), T - 1)];
        if (u < 0 || u >= T) w[q].x = -1;
      }
      if (o > TEAM_MAX_BLOCK) {                         // further away than a block is long
        if ((w[0].x >> 1) == key) set_status(status, TEAM_ERR_STATE, 2);
        break;
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        inside = inside && (w[q].x >> 1) == key;
        if (inside && (w[q].x & 1) && abs(mypos - w[q].y) <= lim) hot = true;
      }
    }
  }
  return hot ? TEAM_CLS_FIRST : TEAM_CLS_COLD;
}

// Position of the n-th (0-based) set bit of m; popcount(m) > n.  Five halvings instead of a bit-by-bit walk.
__device__ __forceinline__ int nth_set_bit(uint32_t m, int n) {
  int pos = 0;
#pragma unroll
  for (int width = 16; width >= 1; width >>= 1) {
    const int c = __popc(m & (((1u << width) - 1u) << pos));
    if (n >= c) {
      n -= c;
      pos += width;
    }
  }
  return pos;
}

// ---------------------------------------------------------------------------------------------------------
// Selection inside the consumer: every CTA of the kernel behind the router classifies and routes all rows of the call by
// itself, into shared memory, and goes on from there.  That saves the selection kernel, its launch and the tables that it
// hands over in global memory, for the issue slots of one warp routing a row, times the rows, on every SM.
// ---------------------------------------------------------------------------------------------------------
struct InlineRoute {     // shared memory
  uint32_t* mask;        // [G][8] E_A bits
  int2* walk;            // [T]
  float* w;              // [T * k] routing weight of each choice
  int16_t* idx;          // [T * k] expert of each choice (-1: row skipped)
  uint8_t* cls;          // [T]
  uint8_t* has_first;    // [G]
};

__host__ __device__ inline size_t inline_route_layout(const Dims& d, InlineRoute* s, unsigned char* base) {
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t at = o;
    o += (bytes + 15) & ~size_t(15);
    return at;
  };
  const size_t a_mask = take((size_t)d.G * 32), a_walk = take((size_t)d.T * 8), a_w = take((size_t)d.T * d.k * 4);
  const size_t a_idx = take((size_t)d.T * d.k * 2), a_cls = take((size_t)d.T), a_hf = take((size_t)d.G);
  if (s != nullptr) {
    s->mask = reinterpret_cast<uint32_t*>(base + a_mask);
    s->walk = reinterpret_cast<int2*>(base + a_walk);
    s->w = reinterpret_cast<float*>(base + a_w);
    s->idx = reinterpret_cast<int16_t*>(base + a_idx);
    s->cls = base + a_cls;
    s->has_first = base + a_hf;
  }
  return o;
}

// The routing rounds over the rows of one class: the i-th row of the class belongs to warp i mod warps; the logits of a
// warp's next row are requested before it routes the current one.
template <int WARPS, int NE, typename Logit>
__device__ __forceinline__ void route_class(int want, Logit logit, const Dims& d, const Policy& p, const InlineRoute& s, uint32_t* bits,
                                            int W1, int32_t* status) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, T = d.T, E = d.E, k = d.k;
  int word = -1, left = warp;            // word of rows under way, rows of the class to pass over from here on
  uint32_t m = 0u;
  auto next_row = [&]() {
    while (left >= __popc(m)) {
      left -= __popc(m);
      if (++word * 32 >= T) return -1;
      const int t = word * 32 + lane;
      m = __ballot_sync(0xffffffffu, t < T && s.cls[t] == want);
    }
    const int t = word * 32 + nth_set_bit(m, left);
    left += WARPS;
    return t;
  };
  float v[kMaxPerLane], nv[NE];
  auto fetch = [&](int t) {
#pragma unroll
    for (int i = 0; i < NE; ++i) nv[i] = t >= 0 && i * 32 + lane < E ? logit(t, i * 32 + lane) : kNegInf;
  };
  int t = next_row();
  fetch(t);
#pragma unroll 1
  while (t >= 0) {
#pragma unroll
    for (int i = 0; i < NE; ++i) v[i] = nv[i];
    const int cur = t, g = walk_group(s.walk[t]);
    t = next_row();
    fetch(t);
    TopkResult r;
    float row_max, denom;
    const float w = route_logits<NE>(v, want == TEAM_CLS_COLD ? s.mask + g * 8 : nullptr, k, lane, E, p.norm_topk, !p.norm_topk, false, false, r,
                                     row_max, denom);
    if (lane < k) {
      s.idx[cur * k + lane] = (int16_t)r.idx;
      s.w[cur * k + lane] = w;
      if (r.idx < 0) {
        if (blockIdx.x == 0) set_status(status, TEAM_ERR_STATE, 3);
      } else {
        if (want == TEAM_CLS_FIRST) atomicOr(&s.mask[g * 8 + (r.idx >> 5)], 1u << (r.idx & 31));
        if (r.idx >= d.elo && r.idx < d.ehi) atomicOr(&bits[r.idx * W1 + (cur >> 5)], 1u << (cur & 31));
      }
    }
  }
}

// Classes, choices and weights of all rows (T <= THREADS), and the bit matrix [expert][row] of who chose whom (W1 words per
// expert; of this rank's own experts, shared ones behind the routed ones).  What the step state holds is read ahead of the
// wait for the preceding kernel (the router, which itself waited for whatever wrote the state), the logits behind it.  Ends
// with a barrier.  CTA 0 leaves the classes in cls_out.  logit(t, e): the logit of row t and expert e.
template <int THREADS, typename Logit>
__device__ __forceinline__ void block_select(Logit logit, const StepPtrs& st, const Dims& d, const Policy& p, const InlineRoute& s,
                                             uint32_t* bits, int W1, uint8_t* cls_out, int32_t* status) {
  constexpr int WARPS = THREADS / 32;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, T = d.T, EN = d.E + d.ns;
  int state = TEAM_TOK_CACHED, cls = TEAM_CLS_SKIP;
  float conf = 0.f;
  if (tid < T) {
    state = st.tok_state[tid];
    conf = st.conf[tid];
    s.walk[tid] = walk_entry(st, tid, state, d.G, status);
  }
  for (int i = tid; i < d.G * 8; i += THREADS) s.mask[i] = 0u;
  for (int i = tid; i < d.G; i += THREADS) s.has_first[i] = 0;
  for (int i = tid; i < EN * W1; i += THREADS) bits[i] = 0u;
  __syncthreads();
  int g = 0;
  if (tid < T) {
    g = walk_group(s.walk[tid]);
    cls = classify_row(s.walk, tid, T, state, conf, p, status);
    if (cls == TEAM_CLS_FIRST) s.has_first[g] = 1;
  }
  __syncthreads();
  if (tid < T) {
    if (cls == TEAM_CLS_COLD && !s.has_first[g]) cls = TEAM_CLS_FIRST;      // nothing to confine its rows to
    s.cls[tid] = (uint8_t)cls;
    if (cls == TEAM_CLS_SKIP)
      for (int j = 0; j < d.k; ++j) s.idx[tid * d.k + j] = -1;
  }
  if (d.ns > 0 && warp * 32 < T) {                                          // shared experts take every computed row
    const uint32_t m = __ballot_sync(0xffffffffu, tid < T && cls != TEAM_CLS_SKIP);
    if (lane < d.ns) bits[(d.E + lane) * W1 + warp] = m;
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");                        // the logits are complete
  if (blockIdx.x == 0 && tid < T) cls_out[tid] = (uint8_t)cls;
  __syncthreads();
#pragma unroll 1
  for (int want = TEAM_CLS_FIRST; want <= TEAM_CLS_COLD; ++want) {
    if (d.E <= 128) route_class<WARPS, 4>(want, logit, d, p, s, bits, W1, status);
    else route_class<WARPS, kMaxPerLane>(want, logit, d, p, s, bits, W1, status);
    __syncthreads();
  }
}

}  // namespace team
