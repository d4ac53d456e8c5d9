// Router kernels (Algorithm 1 "Router"; Sec. 4.1 for which rows are computed).
//
//  k_router_logits_small : up to 8 rows: logits[t,e] = sum_h x[t,h] * W_r[e,h] in fp32, spread as widely as possible.
//  k_router_logits_mma   : more rows, bf16 activations: the same sums on the tensor cores, weights as three bf16 parts.
//  k_router_logits : more rows, fp32 activations (and hidden sizes the small kernel does not hold).  The work is split
//                    over experts (one warp per expert, 128-bit loads of the expert's row) and over tiles of 8 rows
//                    whose activations sit in shared memory.
//  The first two also zero the output rows that the streaming expert kernel accumulates into, or the bit matrix of the choices
//  for the tensor-memory kernels.
//  k_router_topk   : one warp per row: softmax over all experts, plain top-k by warp shuffles,
//                    renormalised weights, decision margin (team_route's outputs).
#include <mutex>

#include "team_common.cuh"
#include "team_topk.cuh"

namespace team {

constexpr int kRowTile = 8;       // rows per CTA in the logits kernel
constexpr int kExpertsPerCta = 8; // one warp each

// Which of the first 32 of n rows from t0 on are computed, as a bit string: one load per lane, in place of one after the other
// (0.6 us of a step of 128 rows when the tensor-memory path's rows were zeroed here, too).
__device__ __forceinline__ uint32_t rows_to_zero(const uint8_t* __restrict__ tok_state, int t0, int n, int lane, int flags) {
  return __ballot_sync(0xffffffffu, lane < n && !((flags & TEAM_F_DCD) && tok_state[t0 + lane] == TEAM_TOK_CACHED));
}

__global__ void __launch_bounds__(kExpertsPerCta * 32)
k_router_logits(const float* __restrict__ x, const float* __restrict__ w_router, float* __restrict__ logits, Dims d) {
  extern __shared__ __align__(16) float s_x[];   // [kRowTile][H]
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the selection kernel may stage its inputs meanwhile
  const int t0 = blockIdx.y * kRowTile;
  const int nt = min(kRowTile, d.T - t0);
  const int tid = threadIdx.x;
  const int H = d.H;
  // this warp's expert: the first batch of its weight row is requested before anything else
  const int warp = tid >> 5, lane = tid & 31;
  const int e = blockIdx.x * kExpertsPerCta + warp;
  const float4* wrow = reinterpret_cast<const float4*>(w_router + (size_t)min(e, d.E - 1) * H);
  const int n4 = H >> 2;
  constexpr int kBatch = 8;             // float4 per lane and batch: 4 KB of the row per warp in flight
  float4 wv[kBatch];
#pragma unroll
  for (int i = 0; i < kBatch; ++i)
    wv[i] = lane + 32 * i < n4 ? __ldg(wrow + lane + 32 * i) : make_float4(0.f, 0.f, 0.f, 0.f);

  const float4* src = reinterpret_cast<const float4*>(x + (size_t)t0 * H);
  for (int i = tid; i < nt * H / 4; i += blockDim.x) reinterpret_cast<float4*>(s_x)[i] = __ldg(src + i);
  for (int i = nt * H + tid; i < kRowTile * H; i += blockDim.x) s_x[i] = 0.f;

  __syncthreads();

  if (e >= d.E) return;
  float acc[kRowTile];
#pragma unroll
  for (int r = 0; r < kRowTile; ++r) acc[r] = 0.f;
  // batches of kBatch float4 per lane; the next batch is requested before the current one is used
  // (the summation order over c is unchanged: ascending c within a lane)
  for (int base = 0; base < n4; base += 32 * kBatch) {
    float4 wn[kBatch];
    const int nbase = base + 32 * kBatch;
#pragma unroll
    for (int i = 0; i < kBatch; ++i)
      wn[i] = nbase + lane + 32 * i < n4 ? __ldg(wrow + nbase + lane + 32 * i) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int i = 0; i < kBatch; ++i) {
      const int c = base + lane + 32 * i;
      if (c < n4) {
        const float4 w = wv[i];
#pragma unroll
        for (int r = 0; r < kRowTile; ++r) {
          const float4 xv = *reinterpret_cast<const float4*>(s_x + r * H + c * 4);
          acc[r] = fmaf(w.x, xv.x, acc[r]);
          acc[r] = fmaf(w.y, xv.y, acc[r]);
          acc[r] = fmaf(w.z, xv.z, acc[r]);
          acc[r] = fmaf(w.w, xv.w, acc[r]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < kBatch; ++i) wv[i] = wn[i];
  }
#pragma unroll
  for (int r = 0; r < kRowTile; ++r) {
    const float s = warp_sum(acc[r]);
    if (lane == 0 && r < nt) logits[(size_t)(t0 + r) * d.E + e] = s;
  }
}


// More than eight rows of bf16 activations: x W_r^T on the tensor cores, with the accuracy of fp32.
//
// An fp32 weight is exactly the sum of three bf16 numbers (8 + 8 + 8 mantissa bits, split by truncation) and a product
// of two bf16 numbers is exact in fp32.  The tensor core truncates while it accumulates (chains over the whole hidden
// dimension were off by 1.05e-6 against 64 bits), so a chain is the three parts of one fragment of 16 elements, the
// smallest first, and the fragments are added with rounded fp32 additions: 1.08e-7, against 1.57e-7 of the fp32 FMA
// kernels that this one replaced (2-norm, 16 to 2048 rows, hidden 2048).  team_route at hidden 2048 x 128 experts, replayed, with its top-k:
// 2048 rows 46.0 -> 17.4 us, 1024 rows 25.9 -> 12.5, 128 rows 12.9 -> 7.1; the mma.sync rate and the reads of x and W from
// L2 are what is left.  mma.sync and not tcgen05: a tcgen05 chain cannot be cut every 16 elements.
//
// A warp owns MT x 16 rows by NT x 8 experts and every eighth block of 32 hidden elements.  Lane (g, c) of a fragment
// takes elements 8c .. 8c+7 of its row's block -- 16 contiguous bytes of x, 32 of W -- which is a permutation of the
// k index common to both operands, so fragments come straight from global memory: no staging, no barrier before the
// first mma, the next blocks are in flight while the current ones are multiplied.  The eight warps' partial tiles meet
// in shared memory and are summed in warp order.
constexpr int kMmaWarps = 8;

// The two truncated bf16 halves of a pair (low half = a), and the pair's exact remainders.
__device__ __forceinline__ uint32_t split_pair(float& a, float& b) {
  const uint32_t ua = __float_as_uint(a), ub = __float_as_uint(b);
  a -= __uint_as_float(ua & 0xffff0000u);
  b -= __uint_as_float(ub & 0xffff0000u);
  return __byte_perm(ua, ub, 0x7632);
}

__device__ __forceinline__ void router_mma(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// The logits of expert e and rows t + j * step (bit j of `again`) as plain fp32 sums: with an infinity or NaN among the
// operands (or an overflow) the sum of the split weights is not finite, because the remainders of an infinity are NaN.
// A thread's logits are formed together and share their expert's weights.  2048 rows x 128 experts, hidden 2048, 21 us for
// the call and its top-k: with all rows NaN 143 us, with one 83 (each logit by itself and element by element: 2270, 85).
template <int PER>
__device__ __forceinline__ void logits_again(const __nv_bfloat16* __restrict__ x, const float* __restrict__ w_router,
                                             float* __restrict__ logits, int H, int E, int T, int e, int t, int step, uint32_t again) {
  const int n4 = H >> 2;
  const float4* wp = reinterpret_cast<const float4*>(w_router + (size_t)e * H);
  auto add = [](float sum, const float4& w, const uint2& v) {
    sum = fmaf(w.x, __uint_as_float(v.x << 16), sum);
    sum = fmaf(w.y, __uint_as_float(v.x & 0xffff0000u), sum);
    sum = fmaf(w.z, __uint_as_float(v.y << 16), sum);
    return fmaf(w.w, __uint_as_float(v.y & 0xffff0000u), sum);
  };
  const uint2* xp[PER];
  float sum[PER];
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    xp[j] = reinterpret_cast<const uint2*>(x + (size_t)min(t + j * step, T - 1) * H);
    sum[j] = 0.f;
  }
#pragma unroll 4
  for (int k = 0; k < n4; ++k) {
    const float4 w = __ldg(wp + k);
#pragma unroll
    for (int j = 0; j < PER; ++j) sum[j] = add(sum[j], w, __ldg(xp[j] + k));
  }
#pragma unroll
  for (int j = 0; j < PER; ++j)
    if ((again >> j) & 1u) logits[(size_t)(t + j * step) * E + e] = sum[j];
}

// kX8: x is only 8-byte aligned (team_route takes such rows), loaded in two pieces
// kHalf: with half the registers of an SM, so that a selection of 512 threads starts beside it
template <int MT, int NT, bool kX8 = false, bool kHalf = false>
__global__ void __launch_bounds__(kMmaWarps * 32, kHalf ? 2 : 1)
k_router_logits_mma(const __nv_bfloat16* __restrict__ x, const float* __restrict__ w_router,
                    const uint8_t* __restrict__ tok_state, float* __restrict__ logits, float* __restrict__ y_zero,
                    uint32_t* __restrict__ bits_zero, Dims d, int flags) {
  constexpr int R = MT * 16, N = NT * 8;
  constexpr int U = MT * NT == 1 ? (kHalf ? 2 : 4) : (MT * NT == 2 ? 2 : 1);      // blocks of 32 in flight beside the current ones
  extern __shared__ __align__(16) float s_part[];                   // [warps][R][N]
  // in this order: the selection kernel stages the step state ahead of its own wait, and that state may come from the
  // kernel in front of this one
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, c = lane & 3;
  const int H = d.H, T = d.T, E = d.E, nb = H >> 5;
  const int t0 = blockIdx.x * R, e0 = blockIdx.y * N;
  const uint4* xr[MT][2];                                           // rows and experts past the end repeat the last one
  const float4* wr[NT];
#pragma unroll
  for (int m = 0; m < MT; ++m)
#pragma unroll
    for (int h = 0; h < 2; ++h) xr[m][h] = reinterpret_cast<const uint4*>(x + (size_t)min(t0 + m * 16 + h * 8 + g, T - 1) * H) + c;
#pragma unroll
  for (int n = 0; n < NT; ++n) wr[n] = reinterpret_cast<const float4*>(w_router + (size_t)min(e0 + n * 8 + g, E - 1) * H) + 2 * c;
  uint4 xc[U][MT][2], xn[U][MT][2];
  float4 wc[U][NT][2], wn[U][NT][2];
  auto load = [&](int b0, uint4 (&xv)[U][MT][2], float4 (&wv)[U][NT][2]) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int b = b0 + u * kMmaWarps;
#pragma unroll
      for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int h = 0; h < 2; ++h) wv[u][n][h] = b < nb ? __ldg(wr[n] + b * 8 + h) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if constexpr (kX8) {
            const uint2* p = reinterpret_cast<const uint2*>(xr[m][h]) + b * 8;
            const uint2 lo = b < nb ? __ldg(p) : make_uint2(0u, 0u), hi = b < nb ? __ldg(p + 1) : make_uint2(0u, 0u);
            xv[u][m][h] = make_uint4(lo.x, lo.y, hi.x, hi.y);
          } else {
            xv[u][m][h] = b < nb ? __ldg(xr[m][h] + b * 4) : make_uint4(0u, 0u, 0u, 0u);
          }
        }
    }
  };
  load(warp, xc, wc);
  if (bits_zero != nullptr)
    for (int i = (blockIdx.y * gridDim.x + blockIdx.x) * blockDim.x + tid; i < (E + d.ns) * (bit_words(T) + 1); i += gridDim.x * gridDim.y * blockDim.x)
      bits_zero[i] = 0u;
  // output rows of computed tokens start from zero (the expert kernel adds partial sums into them); the CTAs of one
  // row tile share the job
  if (y_zero != nullptr) {
#pragma unroll
    for (int w = 0; w < R; w += 32)
      for (uint32_t m = rows_to_zero(tok_state, t0 + w, min(R - w, T - t0 - w), lane, flags); m != 0u; m &= m - 1u) {
        float4* row = reinterpret_cast<float4*>(y_zero + (size_t)(t0 + w + __ffs(m) - 1) * H);
        for (int i = blockIdx.y * blockDim.x + tid; i < H / 4; i += gridDim.y * blockDim.x) row[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
  }
  float acc[MT][NT][4];
#pragma unroll
  for (int m = 0; m < MT; ++m)
#pragma unroll
    for (int n = 0; n < NT; ++n) acc[m][n][0] = acc[m][n][1] = acc[m][n][2] = acc[m][n][3] = 0.f;
#pragma unroll 1
  for (int b = warp; b < nb; b += kMmaWarps * U) {
    load(b + kMmaWarps * U, xn, wn);
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int h = 0; h < 2; ++h)                                   // elements 0-3, then 4-7 of the lane's eight
#pragma unroll
        for (int n = 0; n < NT; ++n) {
          float4 w = wc[u][n][h];
          uint32_t b0[3], b1[3];
#pragma unroll
          for (int part = 0; part < 3; ++part) {
            b0[part] = split_pair(w.x, w.y);
            b1[part] = split_pair(w.z, w.w);
          }
#pragma unroll
          for (int m = 0; m < MT; ++m) {
            const uint4 lo = xc[u][m][0], hi = xc[u][m][1];
            const uint32_t a0 = h ? lo.z : lo.x, a1 = h ? hi.z : hi.x, a2 = h ? lo.w : lo.y, a3 = h ? hi.w : hi.y;
            float t[4] = {0.f, 0.f, 0.f, 0.f};
            router_mma(t, a0, a1, a2, a3, b0[2], b1[2]);
            router_mma(t, a0, a1, a2, a3, b0[1], b1[1]);
            router_mma(t, a0, a1, a2, a3, b0[0], b1[0]);
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[m][n][q] += t[q];
          }
        }
#pragma unroll
    for (int u = 0; u < U; ++u) {
#pragma unroll
      for (int m = 0; m < MT; ++m) { xc[u][m][0] = xn[u][m][0]; xc[u][m][1] = xn[u][m][1]; }
#pragma unroll
      for (int n = 0; n < NT; ++n) { wc[u][n][0] = wn[u][n][0]; wc[u][n][1] = wn[u][n][1]; }
    }
  }
  float* mine = s_part + warp * R * N;
#pragma unroll
  for (int m = 0; m < MT; ++m)
#pragma unroll
    for (int n = 0; n < NT; ++n) {
      *reinterpret_cast<float2*>(mine + (m * 16 + g) * N + n * 8 + 2 * c) = make_float2(acc[m][n][0], acc[m][n][1]);
      *reinterpret_cast<float2*>(mine + (m * 16 + g + 8) * N + n * 8 + 2 * c) = make_float2(acc[m][n][2], acc[m][n][3]);
    }
  __syncthreads();
  constexpr int kThreads = kMmaWarps * 32, PER = (R * N + kThreads - 1) / kThreads;
  static_assert(kThreads % N == 0, "a thread's logits belong to one expert");
  const int e = e0 + tid % N;
  uint32_t again = 0;                                               // logits to be formed again
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const int i = tid + j * kThreads, t = t0 + i / N;
    if (i >= R * N || t >= T || e >= E) continue;
    float sum = 0.f;
#pragma unroll
    for (int w = 0; w < kMmaWarps; ++w) sum += s_part[w * R * N + i];
    logits[(size_t)t * E + e] = sum;
    // not for rows that nobody computes: what their x holds must cost nothing
    if (!isfinite(sum) && !((flags & TEAM_F_DCD) && tok_state[t] == TEAM_TOK_CACHED)) again |= 1u << j;
  }
  if (again != 0) logits_again<PER>(x, w_router, logits, H, E, T, e, t0 + tid / N, kThreads / N, again);
}

// Few rows (T <= kRowTile): the whole job is one pass over the 4*E*H bytes of router weights, so it
// is spread as widely as possible -- two experts per CTA, four warps per expert, each lane issuing all
// of its 128-bit weight loads before anything else -- and the activations are staged once per CTA.
constexpr int kSmallExperts = 2;   // experts per CTA
constexpr int kSmallSplit = 4;     // warps per expert (each takes H/4 of the dot product)
constexpr int kSmallMaxVec = 8;    // float4 per lane: supports H <= 4096

template <typename XT>
__global__ void __launch_bounds__(kSmallExperts * kSmallSplit * 32)
k_router_logits_small(const XT* __restrict__ x, const float* __restrict__ w_router,
                      const uint8_t* __restrict__ tok_state, float* __restrict__ logits, float* __restrict__ y_zero,
                      uint32_t* __restrict__ bits_zero, Dims d, int flags) {
  extern __shared__ __align__(16) float s_x[];   // [T][H] then partial sums
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the selection kernel may stage its inputs meanwhile
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int H = d.H, T = d.T;
  const int e = blockIdx.x * kSmallExperts + warp / kSmallSplit;
  const int part = warp % kSmallSplit;
  const int n4 = H >> 2, per_part = n4 / kSmallSplit;   // float4 per warp

  // 1. weights first: every load in flight at once
  float4 w[kSmallMaxVec];
  const float4* wrow = reinterpret_cast<const float4*>(w_router + (size_t)min(e, d.E - 1) * H) + part * per_part;
#pragma unroll
  for (int i = 0; i < kSmallMaxVec; ++i)
    w[i] = (lane + 32 * i < per_part) ? __ldg(wrow + lane + 32 * i) : make_float4(0.f, 0.f, 0.f, 0.f);

  // 2. stage the rows (16-byte loads), zero this CTA's share of the output rows
  if constexpr (sizeof(XT) == 2) {
    const uint4* src = reinterpret_cast<const uint4*>(x);
    for (int i = tid; i < T * H / 8; i += blockDim.x) {
      const uint4 v = __ldg(src + i);
      const __nv_bfloat162* p = reinterpret_cast<const __nv_bfloat162*>(&v);
      float4 lo, hi;
      float2 f;
      f = __bfloat1622float2(p[0]); lo.x = f.x; lo.y = f.y;
      f = __bfloat1622float2(p[1]); lo.z = f.x; lo.w = f.y;
      f = __bfloat1622float2(p[2]); hi.x = f.x; hi.y = f.y;
      f = __bfloat1622float2(p[3]); hi.z = f.x; hi.w = f.y;
      reinterpret_cast<float4*>(s_x)[2 * i] = lo;
      reinterpret_cast<float4*>(s_x)[2 * i + 1] = hi;
    }
  } else {
    const float4* src = reinterpret_cast<const float4*>(x);
    for (int i = tid; i < T * H / 4; i += blockDim.x) reinterpret_cast<float4*>(s_x)[i] = __ldg(src + i);
  }
  if (bits_zero != nullptr)
    for (int i = blockIdx.x * blockDim.x + tid; i < (d.E + d.ns) * (bit_words(T) + 1); i += gridDim.x * blockDim.x) bits_zero[i] = 0u;
  if (y_zero != nullptr) {
    const int total4 = T * H / 4;
    for (int i = blockIdx.x * blockDim.x + tid; i < total4; i += gridDim.x * blockDim.x) {
      const int t = (i * 4) / H;
      const bool skip = (flags & TEAM_F_DCD) && tok_state[t] == TEAM_TOK_CACHED;
      if (!skip) reinterpret_cast<float4*>(y_zero)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  __syncthreads();

  // 3. partial dot products, warp reduction, then the four parts of each expert are added in a fixed order
  float acc[kRowTile];
#pragma unroll
  for (int r = 0; r < kRowTile; ++r) acc[r] = 0.f;
#pragma unroll
  for (int i = 0; i < kSmallMaxVec; ++i) {
    if (lane + 32 * i < per_part) {
      const int c = part * per_part + lane + 32 * i;
#pragma unroll
      for (int r = 0; r < kRowTile; ++r) {
        if (r < T) {
          const float4 xv = *reinterpret_cast<const float4*>(s_x + r * H + c * 4);
          acc[r] = fmaf(w[i].x, xv.x, acc[r]);
          acc[r] = fmaf(w[i].y, xv.y, acc[r]);
          acc[r] = fmaf(w[i].z, xv.z, acc[r]);
          acc[r] = fmaf(w[i].w, xv.w, acc[r]);
        }
      }
    }
  }
  float* s_part = s_x + T * H;   // [warps][kRowTile]
#pragma unroll
  for (int r = 0; r < kRowTile; ++r) {
    const float sum = warp_sum(acc[r]);
    if (lane == 0) s_part[warp * kRowTile + r] = sum;
  }
  __syncthreads();
  if (tid < kSmallExperts * kRowTile) {
    const int le = tid / kRowTile, r = tid % kRowTile;
    const int ee = blockIdx.x * kSmallExperts + le;
    if (ee < d.E && r < T) {
      float sum = 0.f;
#pragma unroll
      for (int q = 0; q < kSmallSplit; ++q) sum += s_part[(le * kSmallSplit + q) * kRowTile + r];
      logits[(size_t)r * d.E + ee] = sum;
    }
  }
}

__global__ void __launch_bounds__(256)
k_router_topk(const float* __restrict__ logits, const uint8_t* __restrict__ tok_state, RoutePtrs out, Dims d,
              Policy p) {
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (warp >= d.T) return;
  const int t = warp;
  const bool skip = (p.flags & TEAM_F_DCD) && tok_state[t] == TEAM_TOK_CACHED;
  if (skip) {
    if (out.probs)
      for (int e = lane; e < d.E; e += 32) out.probs[(size_t)t * d.E + e] = 0.f;
    if (lane < d.k) {
      if (out.topk_idx) out.topk_idx[t * d.k + lane] = -1;
      if (out.topk_w) out.topk_w[t * d.k + lane] = 0.f;
    }
    if (lane == 0 && out.margin) out.margin[t] = __builtin_huge_valf();
    return;
  }
  float v[kMaxPerLane];
  float row_max, denom;
  load_row(logits + (size_t)t * d.E, d.E, lane, v, row_max, denom);
  if (out.probs) {
#pragma unroll
    for (int i = 0; i < kMaxPerLane; ++i) {
      const int e = i * 32 + lane;
      if (e < d.E) out.probs[(size_t)t * d.E + e] = expf(v[i] - row_max) / denom;
    }
  }
  TopkResult r = warp_topk(v, d.k, lane, d.E);
  const float w = routing_weight(r, d.k, lane, row_max, denom, p.norm_topk);
  if (lane < d.k) {
    if (out.topk_idx) out.topk_idx[t * d.k + lane] = r.idx;
    if (out.topk_w) out.topk_w[t * d.k + lane] = w;
  }
  if (lane == 0 && out.margin) out.margin[t] = r.margin;
}

// Tiles of the tensor-core router, largest first.  A call takes the largest one that still gives about two thirds of the
// SMs a CTA: larger tiles split every weight fewer times and read x and W fewer times from L2, smaller ones keep more
// SMs loading.
struct MmaTile {
  int rows, experts;
  void (*kernel)(const __nv_bfloat16*, const float*, const uint8_t*, float*, float*, uint32_t*, Dims, int);
};
static const MmaTile kMmaTiles[] = {{64, 32, k_router_logits_mma<4, 4>}, {32, 32, k_router_logits_mma<2, 4>},
                                    {32, 16, k_router_logits_mma<2, 2>}, {16, 16, k_router_logits_mma<1, 2>},
                                    {16, 8, k_router_logits_mma<1, 1>}, {32, 16, k_router_logits_mma<2, 2, true>},
                                    {16, 8, k_router_logits_mma<1, 1, false, true>}};
// One takes rows that are only 8-byte aligned, at every size: 64 rows x 128 experts, hidden 2048, 9.1 us with the
// top-k behind it, against 10.3 of the fp32 FMA kernel that read 8 bytes at a time.
constexpr int kMmaTileX8 = 5;
// The smallest tile once more, with half the blocks in flight and half the registers: in front of the selection kernel that starts
// beside it (128 rows 131.3 -> 128.5 us, 8 passes of a block of 32 x 4 849 -> 830); in front of an expert kernel that routes the
// rows itself, which finds no room beside either, it is the slower one (32 rows 76.2 and 77.9 us).
constexpr int kMmaTileHalf = 6;
static MmaTile mma_tile(const Dims& d, bool x8, bool beside) {
  if (x8) return kMmaTiles[kMmaTileX8];
  for (int i = 0; i < kMmaTileX8 - 1; ++i) {
    const MmaTile& t = kMmaTiles[i];
    if (((d.T + t.rows - 1) / t.rows) * ((d.E + t.experts - 1) / t.experts) >= 96) return t;
  }
  return kMmaTiles[beside ? kMmaTileHalf : kMmaTileX8 - 1];
}

// Opt in to the dynamic shared memory the kernels need (done once per context, outside any stream capture).
static bool small_router_ok(const Dims& d) {
  return d.T <= kRowTile && d.H % (4 * kSmallSplit) == 0 && d.H / (4 * kSmallSplit) <= 32 * kSmallMaxVec;
}

// All kernels of the layer ask for the largest shared-memory carve-out, as the expert kernel must:
// an SM whose carve-out differs from what the next kernel prefers is drained and reconfigured first.
template <typename K>
static cudaError_t prepare_kernel(K kernel, int smem) {
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  return e;
}

// The opt-in is a per-device property of the kernel, shared by every context (and by the context-free
// entry point): it is only ever raised, so that preparing for a small hidden size cannot take away
// what a larger one needs.
int router_smem_bytes(int hidden) { return kRowTile * hidden * (int)sizeof(float) + 1024; }

cudaError_t configure_router(int dtype, int hidden) {
  static std::mutex mu;
  static int prepared[64][2] = {};   // [device][dtype]: shared-memory bytes opted in so far
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const int smem = router_smem_bytes(hidden);
  const int di = dtype == TEAM_DTYPE_F32 ? 0 : 1;
  std::lock_guard<std::mutex> lock(mu);
  if (dev >= 0 && dev < 64 && prepared[dev][di] >= smem) return cudaSuccess;
  if (dtype == TEAM_DTYPE_F32) {
    e = prepare_kernel(k_router_logits, smem);
    if (e == cudaSuccess) e = prepare_kernel(k_router_logits_small<float>, smem);
  } else {
    e = prepare_kernel(k_router_logits_small<__nv_bfloat16>, smem);
    for (const MmaTile& t : kMmaTiles)
      if (e == cudaSuccess) e = prepare_kernel(t.kernel, kMmaWarps * t.rows * t.experts * (int)sizeof(float));
  }
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_router_topk, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  if (e == cudaSuccess && dev >= 0 && dev < 64) prepared[dev][di] = smem;
  return e;
}

cudaError_t launch_router_logits(const void* x, int dtype, const float* w_router, const uint8_t* tok_state,
                                 float* logits, float* y_zero, uint32_t* bits_zero, Dims d, int flags, cudaStream_t s) {
  const bool x8 = ((uintptr_t)x & 15) != 0;                          // bf16 only: the tensor-core kernel reads 8 bytes at a time
  if (small_router_ok(d) && !x8) {
    dim3 grid((d.E + kSmallExperts - 1) / kSmallExperts), block(kSmallExperts * kSmallSplit * 32);
    const size_t smem = (size_t)d.T * d.H * sizeof(float) + kSmallExperts * kSmallSplit * kRowTile * sizeof(float);
    if (dtype == TEAM_DTYPE_F32)
      k_router_logits_small<float><<<grid, block, smem, s>>>(static_cast<const float*>(x), w_router, tok_state,
                                                             logits, y_zero, bits_zero, d, flags);
    else
      k_router_logits_small<__nv_bfloat16><<<grid, block, smem, s>>>(static_cast<const __nv_bfloat16*>(x), w_router,
                                                                     tok_state, logits, y_zero, bits_zero, d, flags);
    return cudaGetLastError();
  }
  if (dtype == TEAM_DTYPE_BF16) {
    const MmaTile t = mma_tile(d, x8, bits_zero != nullptr);      // the bit matrix: a selection kernel and the tensor-memory kernels follow
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((d.T + t.rows - 1) / t.rows, (d.E + t.experts - 1) / t.experts);
    cfg.blockDim = dim3(kMmaWarps * 32);
    cfg.dynamicSmemBytes = (size_t)kMmaWarps * t.rows * t.experts * sizeof(float);
    cfg.stream = s;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;      // the launch latency hides behind the preceding kernel
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, t.kernel, static_cast<const __nv_bfloat16*>(x), w_router, tok_state, logits, y_zero, bits_zero, d, flags);
  }
  dim3 grid((d.E + kExpertsPerCta - 1) / kExpertsPerCta, (d.T + kRowTile - 1) / kRowTile);
  dim3 block(kExpertsPerCta * 32);
  const size_t smem = (size_t)kRowTile * d.H * sizeof(float);
  k_router_logits<<<grid, block, smem, s>>>(static_cast<const float*>(x), w_router, logits, d);
  return cudaGetLastError();
}

cudaError_t launch_router_topk(const float* logits, const uint8_t* tok_state, RoutePtrs out, Dims d, Policy p,
                               cudaStream_t s) {
  const int warps_per_block = 8;
  dim3 grid((d.T + warps_per_block - 1) / warps_per_block);
  k_router_topk<<<grid, warps_per_block * 32, 0, s>>>(logits, tok_state, out, d, p);
  return cudaGetLastError();
}

}  // namespace team
