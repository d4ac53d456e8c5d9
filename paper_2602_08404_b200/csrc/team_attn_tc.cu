// The attention half of delayed caching (Sec. 4.1; block diffusion, Sec. 2) on the fifth-generation tensor cores:
// S = Q K^T and O += P V are tcgen05.mma instructions with their accumulators, and P, in tensor memory.
//
// The (computed row, query head) pairs of a sequence that share one key / value head are packed over its branches (they
// attend to the same prefix) and cut into M tiles of 128.  One CTA owns one or two M tiles and a share of the keys (the
// CTAs of a thread-block cluster split the keys and merge their partial results through distributed shared memory).  The
// keys of a CTA are the prefix and then the block once per branch that its pairs belong to; a pair sees its own branch's.
// Two M tiles use the same key / value tile: the tensor core works for one while the softmax of the other runs, and a
// tile is fetched once for 256 pairs.  Thirteen warps, three roles:
//   warps 0-7  softmax, four per M tile: thread i owns pair i = lane i of tensor memory.  Per tile of 64 keys it reads its
//              row of S, keeps a running maximum (one that only moves when the new maximum exceeds it by 2^8, except for
//              few tiles of head size 64; then the output accumulator in tensor memory is rescaled), and writes
//              P = 2^(s - m) as a bf16 pair hi + lo over the columns of S (the A operand of the second product).
//   warp 8     issues the MMAs: S(t+1) of both M tiles ahead of P V(t).
//   warps 9-12 loaders.  A tile that lies in the prefix is fetched by one thread with TMA boxes of [64 keys][64
//              elements], swizzled on the way; tiles that reach into the block (prefix, fresh rows and in-block cache mixed)
//              are stored by all four warps.  Keys are the K-major and values, stored the same way, the MN-major operand.
// What bounds it (clock stamps at 1850 MHz, head size 128): a tile of 64 keys and two M tiles takes 2450 clock cycles (one M tile:
// 1530), of which the counters show the tensor pipe busy for 1300 (S at N = 64 reads its A operand as long as it computes, and P
// counts twice) and the softmax needs 1300 (16 exponentials per clock and SM); the rest is hand-offs between the two.  Around
// the tiles of a split call with two M tiles: 8200 cycles until the first scores, 1900 to leave the partial result, 13000 for
// the cluster's barriers and the merge, whose reads of distributed shared memory run at about 12 bytes per clock and SM.  Kernel
// at 4096 cached tokens, 32 query and 4 key / value heads of 128, block of 32 x 4 branches: 43 us with one M tile per CTA,
// loads through registers and P in shared memory, 25 now.
// Every wait is an mbarrier wait with a limit; when one runs out the CTA stops working, reports TEAM_ERR_TIMEOUT and
// still takes part in the cluster's barriers and frees its tensor memory.
#include <cooperative_groups.h>
#include <cuda.h>

#include <mutex>

#include "team_attn.cuh"
#include "team_tc_ptx.cuh"
#include "team_topk.cuh"

namespace cg = cooperative_groups;

namespace team {

constexpr int kAtKeys = 64;                 // keys per tile
constexpr int kAtPairs = 256;               // pairs per CTA at most: two M tiles
constexpr int kAtSoftmaxWarps = 8, kAtLoadWarps = 4;
constexpr int kAtLoadThreads = kAtLoadWarps * 32;
constexpr int kAtThreads = (kAtSoftmaxWarps + 1 + kAtLoadWarps) * 32;
constexpr int kAtTmemCols = 512;            // per M tile: S / P twice 64 columns, O 128 (64 with head size 64)

template <int D>
struct AtShape {
  static constexpr int NH = D / 64;                        // 64-element halves of a head: one swizzle atom wide each
  static constexpr int kStages = D == 128 ? 4 : 6;         // of the key and of the value ring
  static constexpr int kQTile = 128 * 128;                 // one half of an M tile's queries: [128 rows][128 B]
  static constexpr int kHalf = kAtKeys * 128;              // one half of a key or value tile: [64 keys][128 B]
  static constexpr int kOffK = 2 * NH * kQTile, kOffV = kOffK + kStages * NH * kHalf, kOffBars = kOffV + kStages * NH * kHalf;
  static constexpr int kSmem = kOffBars + 512 + 1024;      // + barriers + slack for the 1024-byte alignment
  // head size 64 has room for a second output accumulator, which takes the products of P lo: half as many truncated
  // additions to the large sum
  static constexpr int kOLo = D == 64 ? 64 : 0;
  // The maximum in use may stay behind the running one by 2^kMoveBy, which saves most of the rescaling of the output
  // accumulator.  But P then no longer ends at 1: the largest weights lie anywhere in their binade, and the rounding of lo is
  // up to twice as large relative to them.  With head size 64 nothing else is as large while a CTA has few tiles, so up to
  // kExactTiles of them the maximum always moves: at 1, 4, 8, 12, 16, 32 tiles the error against 64 bits is 1.9, 2.1, 2.2,
  // 2.3, 2.2, 2.4e-6 that way, 1.9, 2.4, 2.4, 2.6, 2.5, 2.7e-6 with a maximum left behind, and 1.9, 2.1, 2.4, 2.8, 3.2,
  // 5.2e-6 with mma.sync fragments.  It costs 15 % of a tile.  With head size 128 the maximum is left behind: 2.8e-6 at 4096 keys, as
  // it was or smaller at every shape measured; always moving it gives 2.5e-6 but takes 16 layers from 448 to 467 us.
  static constexpr float kMoveBy = 8.f;
  static constexpr int kExactTiles = D == 64 ? 11 : 0;
  static constexpr int kOStride = D + 4;                   // floats per row of the partial output (aliases the operands)
  static_assert(kAtPairs * kOStride * 4 <= kOffBars, "partial output must fit");
};

__device__ __forceinline__ float at_ex2(float x) {          // 2^x, relative error 2^-22; -inf -> 0
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// two fp32 operations in one instruction
__device__ __forceinline__ float2 at_fma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("{\n\t.reg .b64 a, b, c, d;\n\t"
      "mov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tmov.b64 c, {%6, %7};\n\t"
      "fma.rn.f32x2 d, a, b, c;\n\tmov.b64 {%0, %1}, d;\n\t}"
      : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}
__device__ __forceinline__ float2 at_add2(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 a, b, d;\n\t"
      "mov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
      "add.rn.f32x2 d, a, b;\n\tmov.b64 {%0, %1}, d;\n\t}"
      : "=f"(d.x), "=f"(d.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
// thirty-two columns of this warp's lanes of tensor memory; the load is complete only after tmem_wait_ld
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "
               "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
               "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
                 "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
                 "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
                 "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
               : "r"(taddr));
}
// the operands tie the loaded registers to the wait
__device__ __forceinline__ void tmem_wait_ld(uint32_t* r) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]),
                 "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]),
                 "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]),
                 "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
               :
               : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
               "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
               "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
               ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
                 "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]),
                 "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]),
                 "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
               : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// D[tmem] (+)= (A hi + A lo)[tmem] * B[smem desc] over 64 keys: eight instructions of 16 keys (8 columns of A, 2048 B of
// B), first the 32 columns of hi, then the 32 of lo; bf16 inputs, fp32 accumulate, M = 128; issued by a converged warp.
// The products of lo go to d_lo, which may be d_tmem.
__device__ __forceinline__ void tc_mma_ts_hilo(uint32_t d_tmem, uint32_t d_lo, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, q, t, u;\n\t.reg .b64 b1, b2, b3;\n\t.reg .b32 a1, a2, a3, a4, a5, a6, a7;\n\t"
      "elect.sync _|q, 0xffffffff;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "setp.eq.b32 t, 0, 0;\n\t"
      "setp.ne.b32 u, %6, 0;\n\t"
      "add.s64 b1, %2, 128;\n\tadd.s64 b2, %2, 256;\n\tadd.s64 b3, %2, 384;\n\t"
      "add.u32 a1, %1, 8;\n\tadd.u32 a2, %1, 16;\n\tadd.u32 a3, %1, 24;\n\tadd.u32 a4, %1, 32;\n\tadd.u32 a5, %1, 40;\n\t"
      "add.u32 a6, %1, 48;\n\tadd.u32 a7, %1, 56;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [a1], b1, %3, t;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [a2], b2, %3, t;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [a3], b3, %3, t;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%5], [a4], %2, %3, u;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%5], [a5], b1, %3, t;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%5], [a6], b2, %3, t;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%5], [a7], b3, %3, t;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(d_lo), "r"(accumulate | (uint32_t)(d_lo == d_tmem))
      : "memory");
}
// MN-major operand, 128-byte swizzle: atoms of [8 k][64 mn], 1024 B apart along k, half_bytes apart along mn
__device__ __forceinline__ uint64_t make_mnmajor_sw128_desc(uint32_t smem_addr, int half_bytes) {
  return (make_kmajor_sw128_desc(smem_addr) & ~((uint64_t)0x3fff << 16)) | (uint64_t)(half_bytes >> 4) << 16;
}
// one [64 keys][64 elements] box of a [rows][heads][D] tensor
__device__ __forceinline__ void tma_box(uint32_t dst, const void* map, int x, int head, int row, uint32_t bar) {
  asm volatile("cp.async.bulk.tensor.3d.shared::cta.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
               ::"r"(dst), "l"(map), "r"(x), "r"(head), "r"(row), "r"(bar)
               : "memory");
}
// sets the bf16 values of v that are infinite or not a number to 0; whether there was one
__device__ __forceinline__ bool at_drop_nonfinite(uint4& v) {
  uint32_t* w = &v.x;
  bool any = false;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if ((w[i] & 0x7f80u) == 0x7f80u) { w[i] &= 0xffff0000u; any = true; }
    if ((w[i] & 0x7f800000u) == 0x7f800000u) { w[i] &= 0xffffu; any = true; }
  }
  return any;
}
// Where S (and P over it) of tile i, M tile m lives: two buffers per M tile, or four if there is one M tile only.
__device__ __forceinline__ int s_buf(int i, int m, int n_m) { return n_m == 1 ? i & 3 : 2 * m + (i & 1); }
__device__ __forceinline__ uint32_t s_phase(int i, int n_m) { return (i >> (n_m == 1 ? 2 : 1)) & 1; }
__device__ __forceinline__ uint32_t s_cols(int i, int m, int n_m) {
  const int b = s_buf(i, m, n_m);
  return (b >> 1) * 256 + (b & 1) * kAtKeys;
}
__device__ __forceinline__ void bar_loaders() { asm volatile("bar.sync 1, %0;" ::"n"(kAtLoadThreads) : "memory"); }

template <int D>
__global__ void __launch_bounds__(kAtThreads, 1)
k_block_attention_tc(AttnArgs a, int cta_pairs, int n_splits, const __grid_constant__ CUtensorMap kmap, const __grid_constant__ CUtensorMap vmap) {
  using P = AtShape<D>;
  constexpr int NH = P::NH, ST = P::kStages;
  extern __shared__ unsigned char at_smem_raw[];
  unsigned char* smem = at_smem_raw + ((1024u - (smem_u32(at_smem_raw) & 1023u)) & 1023u);      // swizzled tiles: 1024-byte aligned
  const uint32_t sm0 = smem_u32(smem);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + P::kOffBars);
  uint64_t* k_full = bars;                        // [ST] the key tile has landed
  uint64_t* k_empty = k_full + ST;                // [ST] MMA commit: S of that tile is done
  uint64_t* v_full = k_empty + ST;                // [ST] the value tile has landed
  uint64_t* v_empty = v_full + ST;                // [ST] MMA commit: P V of that tile is done
  uint64_t* s_full = v_empty + ST;                // [4] MMA commit: the scores are in tensor memory
  uint64_t* p_full = s_full + 4;                  // [4] softmax warps (4): P is in tensor memory, O is rescaled
  uint64_t* pv_done = p_full + 4;                 // [M tile] MMA commit: O holds the tiles so far
  uint64_t* q_full = pv_done + 2;                 // [1] softmax warps (8): the queries are in shared memory
  uint64_t* all_done = q_full + 1;                // [1] MMA commit: every MMA of the CTA is complete
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(all_done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int32_t* status_sink = reinterpret_cast<int32_t*>(tmem_slot + 2);      // [2] stands in for a null status pointer
  static_assert((4 * ST + 12) * 8 + 16 <= 512, "barriers must fit");
  __shared__ int s_row[kAtPairs + 1], s_off[kAtPairs], s_cnt[kAtThreads / 32], s_nonfinite;
  __shared__ float s_m[kAtPairs], s_l[kAtPairs], s_f[kAttnMaxSplits][kAtPairs];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int sg = blockIdx.x % (a.S * a.Hkv), s = sg / a.Hkv, g = sg - s * a.Hkv, z = blockIdx.z;
  const int L = a.L, rep = a.Hq / a.Hkv, n_rows = a.B * L, row0 = s * n_rows;
  const int pair0 = (int)(blockIdx.x / (a.S * a.Hkv)) * cta_pairs, first_row = pair0 / rep;      // first of the sequence's computed rows
  int32_t* status = a.status != nullptr ? a.status : status_sink;
  if (tid == 0) {
    for (int i = 0; i < ST; ++i) {
      mbar_init(smem_u32(k_full + i), 1);
      mbar_init(smem_u32(k_empty + i), 1);
      mbar_init(smem_u32(v_full + i), 1);
      mbar_init(smem_u32(v_empty + i), 1);
    }
    for (int i = 0; i < 4; ++i) {
      mbar_init(smem_u32(s_full + i), 1);
      mbar_init(smem_u32(p_full + i), 4);
    }
    mbar_init(smem_u32(pv_done), 1);
    mbar_init(smem_u32(pv_done + 1), 1);
    mbar_init(smem_u32(q_full), kAtSoftmaxWarps);
    mbar_init(smem_u32(all_done), 1);
    *abort_flag = 0;
    s_nonfinite = 0;
    status_sink[0] = status_sink[1] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kAtSoftmaxWarps) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"((uint32_t)kAtTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // everything from here on reads what preceding kernels may have written; the kernel behind this one may be scheduled
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // ---- the sequence's rows: layout contract, which of them are computed, this CTA's ----
  const int plen = min(max(a.prefix_len[s], 0), a.P);
  int n_comp = 0;
  for (int base = 0; base < n_rows; base += kAtThreads) {
    const int r = base + tid, t = row0 + r;
    bool comp = false;
    if (r < n_rows) {
      const int b = r / L;
      const bool ok = a.pos[t] == r - b * L && a.group[t] == s && a.branch[t] == b;
      if (!ok && a.status != nullptr) set_status(a.status, TEAM_ERR_STATE, 40);
      comp = attn_computed(a.tok_state[t], a.flags);
    }
    const unsigned bal = __ballot_sync(0xffffffffu, comp);
    if (base > 0) __syncthreads();                          // the counts of the pass before have been read
    if (lane == 0) s_cnt[warp] = __popc(bal);
    __syncthreads();
    int at = n_comp + __popc(bal & ((1u << lane) - 1u)) - first_row;
#pragma unroll
    for (int w = 0; w < kAtThreads / 32; ++w) {
      const int c = s_cnt[w];
      if (w < warp) at += c;
      n_comp += c;
    }
    if (comp && at >= 0 && at <= kAtPairs) s_row[at] = r;
  }
  const int my_pairs = min(cta_pairs, n_comp * rep - pair0);
  if (my_pairs <= 0) {                                      // the whole cluster has the same pairs: it leaves together
    if (warp == kAtSoftmaxWarps)
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(*tmem_slot), "r"((uint32_t)kAtTmemCols) : "memory");
    return;
  }
  const int n_m = my_pairs > 128 ? 2 : 1;                   // M tiles in use
  __syncthreads();                                          // s_row is complete
  const int b0 = s_row[0] / L, b1 = s_row[(pair0 + my_pairs - 1) / rep - first_row] / L;      // branches of the pairs
  int my_branch = b0;
  if (tid < kAtPairs) {
    int off = -1;
    if (tid < my_pairs) {
      const int cr = (pair0 + tid) / rep, r = s_row[cr - first_row];
      off = (row0 + r) * a.Hq + g * rep + (pair0 + tid - cr * rep);
      my_branch = r / L;
    }
    s_off[tid] = off;
  }
  const int n_keys = plen + (b1 - b0 + 1) * L;
  const int tiles_total = (n_keys + kAtKeys - 1) / kAtKeys;
  const int tps = (tiles_total + n_splits - 1) / n_splits;
  const int t_begin = min(z * tps, tiles_total), t_end = min(t_begin + tps, tiles_total);
  const int n_tiles = t_end - t_begin;
  tc_fence_before();
  __syncthreads();                                          // s_off and the tensor memory's address
  tc_fence_after();
  const uint32_t tmem_base = warp_uniform(*tmem_slot);

  if (warp > kAtSoftmaxWarps) {
    // ------------------------------ loaders ------------------------------
    const int ltid = tid - (kAtSoftmaxWarps + 1) * 32;
    bool ok = true;
    for (int i = 0; i < n_tiles; ++i) {
      const int st = i % ST, key0 = (t_begin + i) * kAtKeys;
      const uint32_t free_parity = ((i / ST) & 1) ^ 1;
      const uint32_t kst = sm0 + P::kOffK + st * NH * P::kHalf, vst = sm0 + P::kOffV + st * NH * P::kHalf;
      if (key0 + kAtKeys <= plen) {
        if (warp == kAtSoftmaxWarps + 1 && ok) {            // inside the prefix: one thread, boxes of one half each
          ok = mbar_wait_warp<32>(smem_u32(k_empty + st), free_parity, abort_flag, status, 51);
          if (ok && lane == 0) {
            mbar_expect_tx(smem_u32(k_full + st), NH * P::kHalf);
            for (int h = 0; h < NH; ++h) tma_box(kst + h * P::kHalf, &kmap, h * 64, g, s * a.P + key0, smem_u32(k_full + st));
          }
          if (ok) ok = mbar_wait_warp<32>(smem_u32(v_empty + st), free_parity, abort_flag, status, 52);
          if (ok && lane == 0) {
            mbar_expect_tx(smem_u32(v_full + st), NH * P::kHalf);
            for (int h = 0; h < NH; ++h) tma_box(vst + h * P::kHalf, &vmap, h * 64, g, s * a.P + key0, smem_u32(v_full + st));
          }
          __syncwarp();
        }
        continue;
      }
      // only the warp that has followed every phase of the ring may wait for the stage; the others wait for it
      if (warp == kAtSoftmaxWarps + 1 && ok) {
        ok = mbar_wait_warp<32>(smem_u32(k_empty + st), free_parity, abort_flag, status, 51);
        if (ok) ok = mbar_wait_warp<32>(smem_u32(v_empty + st), free_parity, abort_flag, status, 52);
      }
      bar_loaders();
      ok = ok && !*abort_flag;
      if (ok) {
        constexpr int PIECES = D / 8, PER = kAtKeys * PIECES / kAtLoadThreads;      // 16-byte pieces per row, per thread
        uint4 kk[PER], vv[PER];
#pragma unroll
        for (int q = 0; q < PER; ++q) {
          const int idx = ltid + q * kAtLoadThreads, j = idx / PIECES, c = idx % PIECES, key = key0 + j;
          kk[q] = vv[q] = make_uint4(0u, 0u, 0u, 0u);       // keys past the end: zero rows
          if (key < n_keys) {
            const __nv_bfloat16 *ks = a.k_prefix, *vs = a.v_prefix;
            size_t o;
            if (key < plen) {
              o = (((size_t)s * a.P + key) * a.Hkv + g) * D;
            } else {
              const int r = b0 * L + key - plen;             // row of the sequence
              if (attn_computed(a.tok_state[row0 + r], a.flags)) {
                o = ((size_t)(row0 + r) * a.Hkv + g) * D;
                ks = a.k_new; vs = a.v_new;
              } else {
                o = (((size_t)s * L + r % L) * a.Hkv + g) * D;
                ks = a.k_block; vs = a.v_block;
              }
            }
            kk[q] = *reinterpret_cast<const uint4*>(ks + o + c * 8);
            vv[q] = *reinterpret_cast<const uint4*>(vs + o + c * 8);
          }
        }
        // the tile is multiplied with P = 0 for the pairs of other branches: a value of the block that is not finite must
        // not reach them.  It counts as 0 here and is added to its own branch's outputs at the end.  (A loop of its own:
        // looked at where it is loaded, every value would be waited for before the next one is requested: a call of 4
        // branches x 16 rows, 2 query heads per key / value head of 128, no prefix, 15.8 us, 14.9 this way.)
        if (b1 > b0) {
#pragma unroll
          for (int q = 0; q < PER; ++q)
            if (key0 + (ltid + q * kAtLoadThreads) / PIECES >= plen && at_drop_nonfinite(vv[q])) s_nonfinite = 1;
        }
#pragma unroll
        for (int q = 0; q < PER; ++q) {
          const int idx = ltid + q * kAtLoadThreads, j = idx / PIECES, c = idx % PIECES;
          const uint32_t off = (c >> 3) * P::kHalf + sw128(j, c & 7);
          *reinterpret_cast<uint4*>(smem + P::kOffK + st * NH * P::kHalf + off) = kk[q];
          *reinterpret_cast<uint4*>(smem + P::kOffV + st * NH * P::kHalf + off) = vv[q];
        }
      }
      fence_async_smem();                                   // generic-proxy writes, read by the tensor core
      bar_loaders();
      if (ok && ltid == 0) {
        mbar_arrive(smem_u32(k_full + st));
        mbar_arrive(smem_u32(v_full + st));
      }
    }
    if (!ok) {
      // gave up: the copies already issued still land in this CTA's shared memory; give them time before the CTA exits
      for (int i = 0; i < 64; ++i) __nanosleep(1000);
    }
  } else if (warp == kAtSoftmaxWarps) {
    // ------------------------------ MMA issuer ------------------------------
    const uint32_t idesc_s = make_idesc_bf16(kAtKeys), idesc_o = make_idesc_bf16(D) | (1u << 16);      // V: MN-major
    const int tiles = (int)warp_uniform(n_tiles), n_mt = (int)warp_uniform(n_m);
    bool ok = mbar_wait_warp(smem_u32(q_full), 0, abort_flag, status, 50);
    // S of tile i, M tile m: the columns were P of an earlier tile whose product has been issued before
    auto issue_s = [&](int i, int m) {
      const int st = i % ST;
      if (m == 0) {
        if (!(ok = mbar_wait_warp(smem_u32(k_full + st), (i / ST) & 1, abort_flag, status, 53))) return;
        tc_fence_after();
      }
      const uint32_t kst = sm0 + P::kOffK + st * NH * P::kHalf;
#pragma unroll
      for (int h = 0; h < NH; ++h)
        tc_mma_k64(tmem_base + s_cols(i, m, n_mt), make_kmajor_sw128_desc(sm0 + (m * NH + h) * P::kQTile),
                   make_kmajor_sw128_desc(kst + h * P::kHalf), idesc_s, h != 0);
      tc_commit(smem_u32(s_full + s_buf(i, m, n_mt)));
      if (m == n_mt - 1) tc_commit(smem_u32(k_empty + st));
    };
    // one M tile: scores three tiles ahead; two: one tile ahead, and the M tiles interleaved, so that the tensor core has
    // work queued while this warp waits for P
    const int ahead = n_mt == 1 ? 3 : 1;
    for (int i = 0; i < ahead && i < tiles && ok; ++i)
      for (int m = 0; m < n_mt && ok; ++m) issue_s(i, m);
    for (int i = 0; i < tiles && ok; ++i) {
      const int st = i % ST;
      const uint64_t db = make_mnmajor_sw128_desc(sm0 + P::kOffV + st * NH * P::kHalf, P::kHalf);
      for (int m = 0; m < n_mt && ok; ++m) {
        if (i + ahead < tiles) {
          issue_s(i + ahead, m);
          if (!ok) break;
        }
        if (m == 0 && !(ok = mbar_wait_warp(smem_u32(v_full + st), (i / ST) & 1, abort_flag, status, 56))) break;
        if (!(ok = mbar_wait_warp(smem_u32(p_full + s_buf(i, m, n_mt)), s_phase(i, n_mt), abort_flag, status, 55))) break;
        tc_fence_after();
        tc_mma_ts_hilo(tmem_base + m * 256 + 128, tmem_base + m * 256 + 128 + P::kOLo, tmem_base + s_cols(i, m, n_mt), db, idesc_o, i != 0);
        tc_commit(smem_u32(pv_done + m));
      }
      if (ok) tc_commit(smem_u32(v_empty + st));
    }
    if (ok && tiles > 0) tc_commit(smem_u32(all_done));
  } else {
    // ---- the queries of this CTA's pairs: A operand of S = Q K^T, per M tile NH halves of [128 rows][128 B], swizzled ----
    // A split without a key tile has no product to wait for (all_done) before its partial result goes over these bytes,
    // so it must not store queries: a slower warp's would end up in the partial result.
    if (n_tiles > 0) {
      constexpr int PIECES = D / 8, PER = 128 * PIECES / (kAtSoftmaxWarps * 32);      // 16-byte pieces per row, per thread and M tile
      const int c = tid % PIECES;
      uint4 v[2 * PER];
#pragma unroll
      for (int q = 0; q < 2 * PER; ++q) {
        const int off = s_off[tid / PIECES + q * (kAtSoftmaxWarps * 32 / PIECES)];      // -1 past the CTA's pairs
        v[q] = off >= 0 ? *reinterpret_cast<const uint4*>(a.q + (size_t)off * D + c * 8) : make_uint4(0u, 0u, 0u, 0u);
      }
#pragma unroll
      for (int q = 0; q < 2 * PER; ++q) {
        const int r = tid / PIECES + q * (kAtSoftmaxWarps * 32 / PIECES);
        *reinterpret_cast<uint4*>(smem + ((r >> 7) * NH + (c >> 3)) * P::kQTile + sw128(r & 127, c & 7)) = v[q];
      }
      fence_async_smem();                                   // generic-proxy writes, read by the tensor core
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(q_full));
    // ------------------------------ softmax ------------------------------
    const int m = warp >> 2;                                 // M tile
    const uint32_t tm_lane = tmem_base + ((uint32_t)((warp & 3) * 32) << 16), tm = tm_lane + m * 256;      // this warp's quarter of the lanes
    const int own_lo = plen + (my_branch - b0) * L;          // first key of the pair's own block
    const int pr = tid;                                      // pair of the CTA = lane of tensor memory + 128 * M tile
    const float sl2 = rsqrtf((float)D) * 1.4426950408889634f;      // scores in base 2
    const float move_by = n_tiles > P::kExactTiles ? P::kMoveBy : 0.f;
    float m_used = kNegInf, l_run = 0.f;                     // running maximum in use (base 2) and row sum
    bool ok = true;
    for (int i = 0; i < n_tiles && ok && m < n_m; ++i) {
      const int b = s_buf(i, m, n_m);
      if (!(ok = mbar_wait_warp(smem_u32(s_full + b), s_phase(i, n_m), abort_flag, status, 57))) break;
      tc_fence_after();
      const uint32_t tm_s = tm_lane + s_cols(i, m, n_m);
      uint32_t sc[kAtKeys];
      tmem_ld32(tm_s, sc);
      tmem_ld32(tm_s + 32, sc + 32);
      tmem_wait_ld(sc);
      tmem_wait_ld(sc + 32);
      // mask the other branches' keys (tiles that reach into the block only), the tile's maximum
      const int key0 = (t_begin + i) * kAtKeys;
      if (key0 + kAtKeys > plen) {
#pragma unroll
        for (int e = 0; e < kAtKeys; ++e)
          if (key0 + e >= plen && (unsigned)(key0 + e - own_lo) >= (unsigned)L) sc[e] = __float_as_uint(kNegInf);
      }
      float mx4[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) mx4[e] = __uint_as_float(sc[e]);
#pragma unroll
      for (int e = 4; e < kAtKeys; ++e) mx4[e & 3] = fmaxf(mx4[e & 3], __uint_as_float(sc[e]));
      const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3])) * sl2;      // sl2 > 0: the maximum of the scaled scores
      // the maximum in use moves only when it has to: P stays below 2^kMoveBy, far inside fp32 and the bf16 pair
      const bool move = mx > m_used + move_by;               // always on the first tile with a key of the pair (m_used = -inf)
      float corr = 1.f;
      if (move) {
        corr = at_ex2(m_used - mx);                          // 0 on the first tile
        m_used = mx;
        l_run *= corr;
      }
      // scale and shift in one operation, 2^x, the row sum, and P as bf16 pairs hi = rn(p), lo = rn(p - hi): two keys
      // per column, the 32 columns of hi in front of the 32 of lo
      const float sh = m_used == kNegInf ? 0.f : -m_used;    // no key of the pair so far: every score is -inf
      const float2 scale = make_float2(sl2, sl2), shift = make_float2(sh, sh), minus = make_float2(-1.f, -1.f);
      float2 sum[4] = {};
      uint32_t lo[kAtKeys / 2];
#pragma unroll
      for (int e = 0; e < kAtKeys / 2; ++e) {
        float2 p = at_fma2(make_float2(__uint_as_float(sc[2 * e]), __uint_as_float(sc[2 * e + 1])), scale, shift);
        p.x = at_ex2(p.x);
        p.y = at_ex2(p.y);
        sum[e & 3] = at_add2(sum[e & 3], p);
        const __nv_bfloat162 h2 = __floats2bfloat162_rn(p.x, p.y);
        const uint32_t h = *reinterpret_cast<const uint32_t*>(&h2);
        const float2 rest = at_fma2(make_float2(__uint_as_float(h << 16), __uint_as_float(h & 0xffff0000u)), minus, p);
        const __nv_bfloat162 l2 = __floats2bfloat162_rn(rest.x, rest.y);
        sc[e] = h;
        lo[e] = *reinterpret_cast<const uint32_t*>(&l2);
      }
      sum[0] = at_add2(at_add2(sum[0], sum[1]), at_add2(sum[2], sum[3]));
      l_run += sum[0].x + sum[0].y;
      tmem_st32(tm_s, sc);
      tmem_st32(tm_s + 32, lo);
      // O belongs to the tensor core until P V of the previous tile is complete
      if (i > 0) {
        if (!(ok = mbar_wait_warp(smem_u32(pv_done + m), (i - 1) & 1, abort_flag, status, 58))) break;
        if (__any_sync(0xffffffffu, move)) {
          tc_fence_after();
          constexpr int W = P::kExactTiles > 0 ? 64 : 32;     // where it is in every tile's way: two loads in flight
#pragma unroll 1
          for (int c0 = 0; c0 < 128; c0 += W) {             // both accumulators with head size 64
            uint32_t r[W];
#pragma unroll
            for (int c = 0; c < W; c += 32) tmem_ld32(tm + 128 + c0 + c, r + c);
#pragma unroll
            for (int c = 0; c < W; c += 32) tmem_wait_ld(r + c);
#pragma unroll
            for (int e = 0; e < W; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) * corr);
#pragma unroll
            for (int c = 0; c < W; c += 32) tmem_st32(tm + 128 + c0 + c, r + c);
          }
        }
      }
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(p_full + b));
    }
    // ---- the CTA's partial result: (maximum, sum, unnormalised output) of its pairs into shared memory, over the
    //      operands: every MMA of both M tiles has to be complete ----
    if (ok && n_tiles > 0) ok = mbar_wait_warp<32>(smem_u32(all_done), 0, abort_flag, status, 59);
    tc_fence_after();
    if (m < n_m) {
      float* s_o = reinterpret_cast<float*>(smem);
      const bool have = ok && n_tiles > 0;
      s_m[pr] = have ? m_used : kNegInf;
      s_l[pr] = have ? l_run : 0.f;
#pragma unroll 1
      for (int c0 = 0; c0 < D; c0 += 32) {
        uint32_t r[32];
        if (have) {                                          // warp-uniform
          tmem_ld32(tm + 128 + c0, r);
          tmem_wait_ld(r);
          if (P::kOLo > 0) {
            uint32_t lo[32];
            tmem_ld32(tm + 128 + P::kOLo + c0, lo);
            tmem_wait_ld(lo);
#pragma unroll
            for (int e = 0; e < 32; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) + __uint_as_float(lo[e]));
          }
        } else {
#pragma unroll
          for (int e = 0; e < 32; ++e) r[e] = 0u;
        }
        uint4* dst = reinterpret_cast<uint4*>(s_o + (size_t)pr * P::kOStride + c0);
#pragma unroll
        for (int e = 0; e < 8; ++e) dst[e] = make_uint4(r[4 * e], r[4 * e + 1], r[4 * e + 2], r[4 * e + 3]);
      }
    }
  }

  // ------------------------------ merge over the cluster, teardown ------------------------------
  tc_fence_before();
  __syncthreads();
  cg::cluster_group cluster = cg::this_cluster();
  if (n_splits > 1) cluster.sync();
  if (!*abort_flag) {
    // rank z writes its share of the pairs
    float* s_o = reinterpret_cast<float*>(smem);
    constexpr int TPR = D / 4;                              // threads per pair (one float4 each)
    const int R = (my_pairs + n_splits - 1) / n_splits, r0 = z * R, r1 = min(my_pairs, r0 + R);
    bool nonfinite;
    if (n_splits == 1) {
      // nothing to merge: read from this CTA's own shared memory, not at the 12 bytes per clock of the cluster's, and without
      // the cluster's barriers (4 branches x 16 rows, 2 query heads per key / value head of 128, no prefix: 14.9 us for the
      // call through the merge below, 10.7 here; 256 sequences of one row, 100 cached tokens: 77.1, 64.6)
      nonfinite = s_nonfinite != 0;
      for (int i = tid; i < my_pairs * TPR; i += kAtThreads) {
        const int pr = i / TPR, c4 = i % TPR;
        const float f = 1.f / s_l[pr];
        const float4 v = *reinterpret_cast<const float4*>(s_o + (size_t)pr * P::kOStride + c4 * 4);
        *reinterpret_cast<float4*>(a.out + (size_t)s_off[pr] * D + c4 * 4) = make_float4(f * v.x, f * v.y, f * v.z, f * v.w);
      }
    } else {
      // merge of all partials (distributed shared memory): first each split's weight per pair, then the outputs
      for (int pr = r0 + tid; pr < r1; pr += kAtThreads) {
        float mk[kAttnMaxSplits], lk[kAttnMaxSplits], mx = kNegInf, den = 0.f;
#pragma unroll
        for (int k = 0; k < kAttnMaxSplits; ++k) {
          mk[k] = k < n_splits ? *cluster.map_shared_rank(&s_m[pr], k) : kNegInf;
          lk[k] = k < n_splits ? *cluster.map_shared_rank(&s_l[pr], k) : 0.f;
          mx = fmaxf(mx, mk[k]);
        }
#pragma unroll
        for (int k = 0; k < kAttnMaxSplits; ++k) {
          mk[k] = at_ex2(mk[k] - mx);                        // 0 for a split without a key of the pair (its maximum is -inf)
          den = fmaf(mk[k], lk[k], den);
        }
        const float inv = 1.f / den;
#pragma unroll
        for (int k = 0; k < kAttnMaxSplits; ++k) s_f[k][pr] = mk[k] * inv;
      }
      nonfinite = __any_sync(0xffffffffu, lane < n_splits && *cluster.map_shared_rank(&s_nonfinite, min(lane, n_splits - 1)) != 0);
      __syncthreads();
      for (int i = r0 * TPR + tid; i < r1 * TPR; i += kAtThreads) {
        const int pr = i / TPR, c4 = i % TPR;
        float4 v[kAttnMaxSplits];
#pragma unroll
        for (int k = 0; k < kAttnMaxSplits; ++k) {
          v[k] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (k < n_splits) v[k] = *reinterpret_cast<const float4*>(cluster.map_shared_rank(s_o + (size_t)pr * P::kOStride + c4 * 4, k));
        }
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int k = 0; k < kAttnMaxSplits; ++k) {
          const float f = s_f[k][pr];
          acc.x = fmaf(f, v[k].x, acc.x); acc.y = fmaf(f, v[k].y, acc.y); acc.z = fmaf(f, v[k].z, acc.z); acc.w = fmaf(f, v[k].w, acc.w);
        }
        *reinterpret_cast<float4*>(a.out + (size_t)s_off[pr] * D + c4 * 4) = acc;
      }
    }
    if (nonfinite) {
      // values of the block that were not finite counted as 0: they are added to their own branch's outputs
      for (int i = r0 * TPR + tid; i < r1 * TPR; i += kAtThreads) {
        const int pr = i / TPR, c4 = i % TPR;
        float4* dst = reinterpret_cast<float4*>(a.out + (size_t)s_off[pr] * D + c4 * 4);
        float4 acc = *dst;                                  // this thread's own store
        const int t = s_off[pr] / a.Hq;                     // the pair's row; its block begins at t - pos
        const int t_block = t - (t - row0) % L;
        for (int p = 0; p < L; ++p) {
          const bool fresh = attn_computed(a.tok_state[t_block + p], a.flags);
          const __nv_bfloat16* v4 = (fresh ? a.v_new + ((size_t)(t_block + p) * a.Hkv + g) * D : a.v_block + (((size_t)s * L + p) * a.Hkv + g) * D) + c4 * 4;
          const float x0 = __bfloat162float(v4[0]), x1 = __bfloat162float(v4[1]), x2 = __bfloat162float(v4[2]), x3 = __bfloat162float(v4[3]);
          if (!isfinite(x0)) acc.x += x0;
          if (!isfinite(x1)) acc.y += x1;
          if (!isfinite(x2)) acc.z += x2;
          if (!isfinite(x3)) acc.w += x3;
        }
        *dst = acc;
      }
    }
  }
  if (n_splits > 1) cluster.sync();                        // peers may still be reading this CTA's partial
  else __syncthreads();
  if (a.insert) {
    // this cluster holds all pairs of (sequence, key / value head), so nobody reads the in-block cache any more: the
    // delayed insertion (see k_attn_insert), positions spread over the cluster
    for (int i = tid; i < L * (D / 8); i += kAtThreads) {
      const int p = i / (D / 8), c = i % (D / 8), st = a.tok_state[row0 + p];
      if (p % n_splits != z || !attn_computed(st, a.flags) || st == TEAM_TOK_MASKED) continue;
      const size_t src = ((size_t)(row0 + p) * a.Hkv + g) * D + c * 8, dst = (((size_t)s * L + p) * a.Hkv + g) * D + c * 8;
      *reinterpret_cast<uint4*>(a.k_block + dst) = *reinterpret_cast<const uint4*>(a.k_new + src);
      *reinterpret_cast<uint4*>(a.v_block + dst) = *reinterpret_cast<const uint4*>(a.v_new + src);
    }
  }
  if (warp == kAtSoftmaxWarps) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)kAtTmemCols) : "memory");
  }
}

// Per device: the shared-memory opt-in, the tensor-map encoder, and how many clusters of each size run at once (a cluster
// stays inside one GPC, so clusters of 7 or 8 leave SMs unused that clusters of 6 would take).
struct AttnSetup {
  decltype(&cuTensorMapEncodeTiled) encode;
  int clusters[2][kAttnMaxSplits + 1];                      // [head size 64, 128][cluster size]
};

template <int D>
static cudaLaunchConfig_t attn_launch(cudaLaunchAttribute (&at)[2], dim3 grid, cudaStream_t s) {
  cudaLaunchConfig_t lc = {};
  lc.gridDim = grid;
  lc.blockDim = dim3(kAtThreads);
  lc.dynamicSmemBytes = AtShape<D>::kSmem;
  lc.stream = s;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 1; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = grid.z;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;      // the launch latency hides behind the preceding kernel
  at[1].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at;
  lc.numAttrs = 2;
  return lc;
}

template <int D>
static cudaError_t setup_kernel(int n_sms, int (&clusters)[kAttnMaxSplits + 1]) {
  cudaError_t e = cudaFuncSetAttribute(k_block_attention_tc<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, AtShape<D>::kSmem);
  clusters[1] = n_sms;
  for (int n = 2; n <= kAttnMaxSplits && e == cudaSuccess; ++n) {
    cudaLaunchAttribute at[2];
    cudaLaunchConfig_t lc = attn_launch<D>(at, dim3(1, 1, n), nullptr);
    lc.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&clusters[n], k_block_attention_tc<D>, &lc) != cudaSuccess) {
      cudaGetLastError();
      clusters[n] = 0;                                      // not used
    }
  }
  return e;
}

static cudaError_t attn_setup(const AttnSetup** out) {
  static std::mutex mu;
  static AttnSetup setups[64] = {};
  int dev = 0, n_sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(mu);
  AttnSetup& st = setups[dev];
  *out = &st;
  if (st.encode != nullptr) return cudaSuccess;
  e = cudaDeviceGetAttribute(&n_sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = setup_kernel<64>(n_sms, st.clusters[0]);
  if (e == cudaSuccess) e = setup_kernel<128>(n_sms, st.clusters[1]);
  if (e == cudaSuccess) e = configure_attention_frag();
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult found;
  if (e == cudaSuccess) e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &found);
  if (e == cudaSuccess && found != cudaDriverEntryPointSuccess) e = cudaErrorNotSupported;
  if (e == cudaSuccess) st.encode = reinterpret_cast<decltype(&cuTensorMapEncodeTiled)>(fn);
  return e;
}

// Waves of clusters of which `at_once` run at once.
static long long at_waves(long long clusters, int at_once) { return clusters <= at_once ? 1 : (clusters + at_once - 1) / at_once; }

// Head size 64: whether a call runs the fragment kernel (then how) instead of the tensor-memory kernel, planned as given.
//
// With few pairs over few key tiles it takes fewer steps: 4 sequences x 4 key / value heads, 4 pairs, no prefix 5.9 us against
// 7.9; 64 pairs, 3000 cached tokens 13.0 against 13.2; 256 pairs 17.3 against 15.8.  Both are estimated in ns: every wave of
// clusters takes its tiles of keys and what is around them, which grows with a CTA's pairs (fitted to 1400 and 2800 replayed calls
// of 1 to 1024 sequences x heads, 4 to 1024 pairs, prefixes of 0 to 6000, within 5 and 6 % rms).  How many rows are
// computed is not known here: with delayed caching the estimates are means over 4, 3, 2 and 1 quarters of them.
static bool use_fragments(const AttnArgs& a, const AttnSetup& st, int tiles_max, int tc_m, int tc_splits, int* m_tiles, int* n_splits) {
  const int run_pairs = a.L * (a.Hq / a.Hkv);              // of a sequence and branch
  const long long heads = (long long)a.S * a.Hkv, runs = heads * a.B;
  // M tiles by the largest number of pairs; splits until the grid fills the SMs, each keeping at least two tiles
  *m_tiles = (run_pairs + 127) / 128;
  int n = 1;
  while (n < kAttnMaxSplits && *m_tiles * runs * n * 2 <= st.clusters[0][1] && tiles_max >= 4 * n) n *= 2;
  *n_splits = n;
  if (st.clusters[0][n] < 1) return false;
  // The insertion (0.9 us) is part of either kernel where one cluster holds all pairs of a (sequence, key / value head), else a
  // launch of its own, which takes 2 us of the host's time: calls that are not replayed are bound by that (4 branches x 4
  // rows, 16 pairs, 100 cached tokens: 12.7 us a call on the tensor-memory kernel, 15.4 with two launches; replayed 8.2 and 7.2).
  const bool insert_launch = a.B > 1 || *m_tiles > 1, tc_launch = (long long)run_pairs * a.B > 128 * tc_m;
  const int split = tc_splits > 1;
  const long long tc_tiles = (tiles_max + tc_splits - 1) / tc_splits, tiles = (tiles_max + n - 1) / n;
  const int tile = tc_tiles > AtShape<64>::kExactTiles ? (tc_m == 1 ? 870 : 1130) : (tc_m == 1 ? 970 : 1290);
  long long tc = 0, frag = 0;
  for (int q = (a.flags & TEAM_F_DCD) ? 1 : 4; q <= 4; ++q) {
    const long long run = ((long long)q * run_pairs + 3) / 4, all = ((long long)q * run_pairs * a.B + 3) / 4;
    const int warps = ((int)(run < 128 ? run : 128) + 15) / 16, of_cta = (int)(all < 128 * tc_m ? all : 128 * tc_m);
    tc += at_waves((all + 128 * tc_m - 1) / (128 * tc_m) * heads, st.clusters[0][tc_splits]) *
          (tc_tiles * tile + (split ? 6550 : 6050) + of_cta * (split ? 2330 : 1600) / 128);
    frag += at_waves((run + 127) / 128 * runs, st.clusters[0][n]) * (tiles * (857 + 88 * warps) + 4000 + 376 * warps) +
            (insert_launch && !tc_launch ? 2900 : 900);
  }
  return frag * 105 < tc * 100;        // clearly less: the estimates scatter by more than that
}

template <int D>
static cudaError_t launch(AttnArgs a, const AttnSetup& st, cudaStream_t s, bool* inserted) {
  // One or two M tiles per CTA and how many CTAs split the keys: whatever should end first, at 1500 clock cycles for a key
  // tile of one M tile, 2100 of two and 10000 around the tiles per wave of clusters, which were fitted to whole calls.  (Clock
  // stamps inside one CTA give 1530, 2450 and 19000 to 25000, which overlap with the next wave's; with those the choice is
  // another one for 1 of 80 random calls of up to 512 rows and 8192 cached tokens.)  A decoded block has a quarter of its rows cached on average when delayed caching is on.  Where the clusters of
  // three quarters of the rows just run at once, the first passes of a block take two waves (32 x 4 rows, 32 query and 4 key /
  // value heads of 128, 1500 cached tokens: 35 us in the first pass, 20 to 21 from the third on; 4096 tokens: 51, 27).
  const long long pairs = (long long)a.B * a.L * (a.Hq / a.Hkv), expected = (a.flags & TEAM_F_DCD) ? (3 * pairs + 3) / 4 : pairs;
  const int tiles_max = (a.P + a.L + kAtKeys - 1) / kAtKeys;
  int cta_pairs = 128, n_splits = 1;
  long long best = -1;
  for (int m = 1; m <= 2; ++m) {
    const long long units = (expected + 128 * m - 1) / (128 * m) * a.S * a.Hkv;
    for (int n = 1; n <= kAttnMaxSplits && (n == 1 || tiles_max >= 2 * n); ++n) {
      const int at_once = st.clusters[D / 128][n];
      if (at_once < 1) continue;
      const long long cost = ((units + at_once - 1) / at_once) * ((tiles_max + n - 1) / n * (m == 1 ? 1500 : 2100) + 10000);
      if (best < 0 || cost < best) {
        best = cost;
        cta_pairs = 128 * m;
        n_splits = n;
      }
    }
  }
  if (D == 64) {
    int frag_m_tiles, frag_splits;
    if (use_fragments(a, st, tiles_max, cta_pairs / 128, n_splits, &frag_m_tiles, &frag_splits)) {
      a.insert = *inserted = a.B == 1 && frag_m_tiles == 1;
      return launch_attention_frag(a, frag_m_tiles, frag_splits, s);
    }
  }
  const int m_tiles = (int)((pairs + cta_pairs - 1) / cta_pairs);
  a.insert = *inserted = m_tiles == 1;      // the only cluster of its sequence and head also inserts: one launch fewer
  CUtensorMap kmap = {}, vmap = {};
  if (a.P >= kAtKeys) {                                     // else no tile lies in the prefix and the maps are not used
    const cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)a.Hkv, (cuuint64_t)a.S * a.P};
    const cuuint64_t strides[2] = {(cuuint64_t)D * 2, (cuuint64_t)a.Hkv * D * 2};
    const cuuint32_t box[3] = {64, 1, kAtKeys}, elem[3] = {1, 1, 1};
    for (int i = 0; i < 2; ++i) {
      const __nv_bfloat16* base = i ? a.v_prefix : a.k_prefix;
      if (st.encode(i ? &vmap : &kmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<__nv_bfloat16*>(base), dims, strides, box, elem,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    }
  }
  cudaLaunchAttribute at[2];
  const cudaLaunchConfig_t lc = attn_launch<D>(at, dim3(a.S * a.Hkv * m_tiles, 1, n_splits), s);      // clusters without a computed row come last
  return cudaLaunchKernelEx(&lc, k_block_attention_tc<D>, a, cta_pairs, n_splits, kmap, vmap);
}

cudaError_t launch_attention_tc(const AttnArgs& a, cudaStream_t s, bool* inserted) {
  const AttnSetup* st = nullptr;
  const cudaError_t e = attn_setup(&st);
  if (e != cudaSuccess) return e;
  return a.d == 128 ? launch<128>(a, *st, s, inserted) : launch<64>(a, *st, s, inserted);
}

}  // namespace team
