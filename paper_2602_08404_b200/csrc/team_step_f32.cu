// The whole fp32 step of few rows and few weights as one kernel on one thread-block cluster.
//
// The four kernels of the general path (router, selection, gate / up, down) take 20.5 us for a step of 4 rows (hidden 256, 16
// experts of 128 columns) whose weights L2 delivers in two: what counts is launches and the hops between them.  Here the CTAs
// of one cluster meet at its hardware barrier instead: the router's dot products are spread over all warps and every CTA
// receives all logits through distributed shared memory, routes the rows by itself (team_route.cuh), and the (expert, column)
// pairs of the gate / up products and the (row, column) pairs of the down product are spread over all warps again, the
// activations passing through global memory.  An expert's gate and up rows are read once for all of its rows.  13.6 us.  One
// cluster is 16 SMs, so calls with many weights stay on the general path.
#include <cooperative_groups.h>

#include <mutex>

#include "team_route.cuh"

namespace team {

namespace cg = cooperative_groups;

constexpr int kF32Threads = 1024, kF32Warps = kF32Threads / 32;
constexpr int kF32Rows = 8;
constexpr int kF32IdleThreads = kF32Threads - kF32Rows * 32;      // of the warps without a row
static_assert(kF32Rows * TEAM_MAX_EXPERTS <= 8 * kF32IdleThreads, "logit = thread of the smallest cluster");
static_assert(kF32Threads >= TEAM_MAX_EXPERTS + TEAM_MAX_SHARED, "expert = thread");
constexpr int kF32Cluster = 16;                       // needs the opt-in beyond the portable 8
// What one cluster reads at L2's rate to 16 SMs, where the general path has all of them: the weights of a call (its experts' and
// the router's) at most, and the router's weights times rows (every CTA multiplies its share with all rows out of shared memory).
// Replayed, general path and here, us: 3.0 MB (4 rows x 2 choices, hidden 256, 16 experts of 128 columns) 14.2, 14.1; 3.8 MB (4 x 2,
// hidden 512, 80 columns) 14.8, 13.4; 4.0 MB, 1 of them the router's (2 rows x 2, hidden 1024, 256 of 64) 16.5, 15.3.  Above
// the limit 4.5 MB (4 x 2, hidden 256, 16 of 192) 15.1, 15.9; 6.0 MB (same, 256 columns) 15.3, 17.8; 7.0 MB, 4 of them the
// router's (4 x 1, hidden 4096, 256 of 16) 25.8, 30.0.  Rows x router of 4 MB and 8 MB: 8 x 1024 x 128 (2 choices) 18.0, 16.9, x
// 256 experts 18.0, 19.1; 8 x 2048 x 64 (1 choice) 20.6, 20.3, x 128 21.0, 21.2.  (Launched one by one the general path takes 3
// to 5 us more, the host's time for four launches.)
constexpr size_t kF32MaxBytes = 4 << 20, kF32MaxRouterRows = 4 << 20;
constexpr size_t kF32MaxSmem = 200 << 10;

struct F32Args {
  const float* x;                // [T, H]
  const float* w_router;         // [E, H]
  const float* w_gate;           // [E + ns, I, H]
  const float* w_up;
  const float* w_down;           // [E + ns, I/16, H, 16]
  float* logits;                 // [T, E] left for team_select_experts
  float* act;                    // [T * (k + ns), I]
  float* y;                      // [T, H]
  StepPtrs st;
  Policy p;
  Dims d;
  uint8_t* cls_out;
  int32_t* status;
};

struct F32Smem {
  float* x;                      // [T][H]
  float* logits;                 // [T][E]
  uint32_t* bits;                // [EN] rows that chose the expert
  int32_t* list;                 // [EN] experts with rows
  int32_t* cnt;                  // [warps] of them per warp of experts
  InlineRoute rt;
};
__host__ __device__ inline size_t f32_smem_layout(const Dims& d, F32Smem* s, unsigned char* base) {
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t at = o;
    o += (bytes + 15) & ~size_t(15);
    return at;
  };
  const size_t EN = d.E + d.ns;
  const size_t a_x = take((size_t)d.T * d.H * 4), a_l = take((size_t)d.T * d.E * 4), a_b = take(EN * 4), a_i = take(EN * 4), a_c = take(kF32Warps * 4);
  if (s != nullptr) {
    s->x = reinterpret_cast<float*>(base + a_x);
    s->logits = reinterpret_cast<float*>(base + a_l);
    s->bits = reinterpret_cast<uint32_t*>(base + a_b);
    s->list = reinterpret_cast<int32_t*>(base + a_i);
    s->cnt = reinterpret_cast<int32_t*>(base + a_c);
  }
  return o + inline_route_layout(d, s != nullptr ? &s->rt : nullptr, base + o);
}

__device__ __forceinline__ void f32_fma4(float& acc, const float4& w, const float4& v) {
  acc = fmaf(w.x, v.x, acc);
  acc = fmaf(w.y, v.y, acc);
  acc = fmaf(w.z, v.z, acc);
  acc = fmaf(w.w, v.w, acc);
}

__global__ void __launch_bounds__(kF32Threads, 1) k_step_f32(F32Args a) {
  extern __shared__ __align__(16) unsigned char f32_smem[];
  F32Smem s;
  f32_smem_layout(a.d, &s, f32_smem);
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, rank = blockIdx.x, n = gridDim.x;
  const int T = a.d.T, H = a.d.H, E = a.d.E, k = a.d.k, I = a.d.I, EN = E + a.d.ns, n4 = H >> 2;
  const int me = warp * n + rank, all = kF32Warps * n;          // this warp among the cluster's
  cluster.barrier_arrive();                                     // waited for before another CTA's shared memory is written
  asm volatile("griddepcontrol.wait;" ::: "memory");            // x, the step state and y may belong to the preceding kernel
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  for (int i = tid; i < T * n4; i += kF32Threads) reinterpret_cast<float4*>(s.x)[i] = __ldg(reinterpret_cast<const float4*>(a.x) + i);
  __syncthreads();
  cluster.barrier_wait();                                       // all CTAs of the cluster have started
  const float4* xs = reinterpret_cast<const float4*>(s.x);
  // ---- router: warp = expert ----
  for (int e = me; e < E; e += all) {
    const float4* wr = reinterpret_cast<const float4*>(a.w_router + (size_t)e * H);
    float acc[kF32Rows] = {};
#pragma unroll 4
    for (int c = lane; c < n4; c += 32) {
      const float4 w = __ldg(wr + c);
#pragma unroll
      for (int r = 0; r < kF32Rows; ++r)
        if (r < T) f32_fma4(acc[r], w, xs[r * n4 + c]);
    }
#pragma unroll
    for (int r = 0; r < kF32Rows; ++r)
      if (r < T) {
        const float sum = warp_sum(acc[r]);
        if (lane < n) *cluster.map_shared_rank(s.logits + r * E + e, lane) = sum;      // every CTA gets a copy
      }
  }
  cluster.sync();
  // The logits are left for team_select_experts, by threads that route no row: 0.05 us of the step (in front of the meeting the
  // stores cost 0.4, behind the activations 0.05 as well).
  if (const int i = rank * kF32IdleThreads + tid - kF32Rows * 32; tid >= kF32Rows * 32 && i < T * E) a.logits[i] = s.logits[i];
  // ---- selection, by every CTA; the experts with rows, in ascending order ----
  block_select<kF32Threads>([&](int t, int e) { return s.logits[t * E + e]; }, a.st, a.d, a.p, s.rt, s.bits, 1, a.cls_out, a.status);
  const unsigned act_b = __ballot_sync(0xffffffffu, tid < EN && s.bits[min(tid, EN - 1)] != 0u);
  if (lane == 0) s.cnt[warp] = __popc(act_b);
  __syncthreads();
  int n_act = 0, at = __popc(act_b & ((1u << lane) - 1u));
#pragma unroll
  for (int w = 0; w < (TEAM_MAX_EXPERTS + TEAM_MAX_SHARED + 31) / 32; ++w) {
    if (w < warp) at += s.cnt[w];
    n_act += s.cnt[w];
  }
  if ((act_b >> lane) & 1u) s.list[at] = tid;
  __syncthreads();
  // ---- gate / up: warp = (expert, intermediate column), all of the expert's rows ----
  for (int it = me; it < n_act * I; it += all) {
    const int e = s.list[it / I], i = it % I;
    const uint32_t m = s.bits[e];
    const float4* wg = reinterpret_cast<const float4*>(a.w_gate + ((size_t)e * I + i) * H);
    const float4* wu = reinterpret_cast<const float4*>(a.w_up + ((size_t)e * I + i) * H);
    float ag[kF32Rows] = {}, au[kF32Rows] = {};
#pragma unroll 4
    for (int c = lane; c < n4; c += 32) {
      const float4 g = __ldg(wg + c), u = __ldg(wu + c);
#pragma unroll
      for (int r = 0; r < kF32Rows; ++r)
        if ((m >> r) & 1u) {
          const float4 v = xs[r * n4 + c];
          f32_fma4(ag[r], g, v);
          f32_fma4(au[r], u, v);
        }
    }
#pragma unroll
    for (int r = 0; r < kF32Rows; ++r)
      if ((m >> r) & 1u) {
        const float g = warp_sum(ag[r]), u = warp_sum(au[r]);
        const unsigned which = __ballot_sync(0xffffffffu, lane < k && s.rt.idx[r * k + min(lane, k - 1)] == e);
        const int slot = e < E ? r * k + __ffs(which) - 1 : T * k + (e - E) * T + r;
        if (lane == 0) a.act[(size_t)slot * I + i] = g / (1.f + expf(-g)) * u;
      }
  }
  cluster.sync();                                               // the activations of all CTAs are in global memory
  // ---- down: warp = (row, 2, 4 or 8 output columns), the row's slots in order ----
  // Lane = (16-row block of the intermediate columns, output column, four of the 16): a load is 64 bytes per output column, and
  // the only hop from lane to lane comes behind all slots.  As many columns as leave every warp at most one piece, so that a
  // row's loads are in flight together.  One column per warp and a sum over the lanes per slot, against this, us: 8 rows x 3
  // choices of 20 experts (hidden 384, 32 columns) 25.5, 15.5 (general path 21.6); 4 rows x 2 of 16 (hidden 256, 128) 14.6, 13.6.
  const int lc = T * H <= 2 * all ? 1 : T * H <= 4 * all ? 2 : 3, per_t = (H + (1 << lc) - 1) >> lc;
  const int q = lane & 3, col = (lane >> 2) & ((1 << lc) - 1), ib0 = lane >> (2 + lc), ibs = 8 >> lc;
  for (int it = me; it < T * per_t; it += all) {
    const int t = it / per_t, h = ((it - t * per_t) << lc) + col;
    if (s.rt.cls[t] == TEAM_CLS_SKIP) continue;
    float out = 0.f;
    for (int j = 0; j < k + a.d.ns; ++j) {
      const int slot = j < k ? t * k + j : T * k + (j - k) * T + t, e = j < k ? s.rt.idx[slot] : E + j - k;
      const float w = j < k ? s.rt.w[slot] : 1.f;
      if (h >= H || e < 0 || (e < E && (e < a.d.elo || e >= a.d.ehi))) continue;
      const float4* wr = reinterpret_cast<const float4*>(a.w_down + ((size_t)e * (I / 16) * H + h) * 16) + q;
      const float4* ar = reinterpret_cast<const float4*>(a.act + (size_t)slot * I) + q;
      float acc = 0.f;
#pragma unroll 4
      for (int ib = ib0; ib < I / 16; ib += ibs) f32_fma4(acc, __ldg(wr + (size_t)ib * H * 4), __ldcg(ar + ib * 4));
      out = fmaf(w, acc, out);
    }
    out += __shfl_xor_sync(0xffffffffu, out, 1);
    out += __shfl_xor_sync(0xffffffffu, out, 2);
    for (int o = 4 << lc; o < 32; o <<= 1) out += __shfl_xor_sync(0xffffffffu, out, o);
    if (h < H && (lane & ~(((1 << lc) - 1) << 2)) == 0) a.y[(size_t)t * H + h] = out;
  }
}

static cudaLaunchConfig_t f32_launch(int ctas, size_t smem, cudaStream_t s, cudaLaunchAttribute (&at)[2]) {
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(ctas);
  lc.blockDim = dim3(kF32Threads);
  lc.dynamicSmemBytes = smem;
  lc.stream = s;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = ctas; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at;
  lc.numAttrs = 2;
  return lc;
}

// CTAs of the cluster that the device can hold (0: none), asked once per device.
cudaError_t configure_step_f32(int* ctas) {
  static std::mutex mu;
  static int known[64] = {};                                    // 1 + CTAs
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mu);
  if (dev < 64 && known[dev] > 0) {
    *ctas = known[dev] - 1;
    return cudaSuccess;
  }
  e = cudaFuncSetAttribute(k_step_f32, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kF32MaxSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_step_f32, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_step_f32, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  *ctas = 0;
  for (int n = kF32Cluster; n >= 8 && *ctas == 0; n /= 2) {
    cudaLaunchAttribute at[2];
    cudaLaunchConfig_t lc = f32_launch(n, kF32MaxSmem, nullptr, at);
    lc.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, k_step_f32, &lc) != cudaSuccess) cudaGetLastError();
    else if (clusters > 0) *ctas = n;
  }
  if (dev < 64) known[dev] = 1 + *ctas;
  return cudaSuccess;
}

bool step_f32_supported(const Dims& d) {
  const size_t slots = (size_t)d.T * (d.k + d.ns), experts = slots < (size_t)(d.E + d.ns) ? slots : d.E + d.ns;
  const size_t router = (size_t)d.E * d.H * 4;
  return d.T <= kF32Rows && experts * d.H * d.I * 12 + router <= kF32MaxBytes && router * d.T <= kF32MaxRouterRows && f32_smem_layout(d, nullptr, nullptr) <= kF32MaxSmem;
}

cudaError_t launch_step_f32(const void* x, const float* w_router, const void* w_gate, const void* w_up, const void* w_down, Workspace ws,
                            const InlineSelect& sel, float* y, Dims d, int ctas, cudaStream_t s) {
  F32Args a = {};
  a.x = static_cast<const float*>(x);
  a.w_router = w_router;
  a.w_gate = static_cast<const float*>(w_gate);
  a.w_up = static_cast<const float*>(w_up);
  a.w_down = static_cast<const float*>(w_down);
  a.logits = ws.logits;
  a.act = ws.act;
  a.y = y;
  a.st = sel.st;
  a.p = sel.p;
  a.d = d;
  a.cls_out = ws.r.tok_class;
  a.status = ws.status;
  cudaLaunchAttribute at[2];
  const cudaLaunchConfig_t lc = f32_launch(ctas, f32_smem_layout(d, nullptr, nullptr), s, at);
  return cudaLaunchKernelEx(&lc, k_step_f32, a);
}

}  // namespace team
