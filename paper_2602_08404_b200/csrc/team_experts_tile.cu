// Grouped SwiGLU experts on the tensor cores (tcgen05 / tensor memory) for calls with many rows.
//
// With tens of token-slots per activated expert the SwiGLU experts (Eq. 1) are two grouped GEMMs with the
// weights on the M side (128 rows per instruction) and an expert's token-slots on the N side (up to 128, all
// of them in one pass, so an expert's weights cross HBM once however many rows chose it):
//
//   kernel A   D[128, N] = Wgu_tile[128, H] * X[N, H]^T      128 rows = 64 intermediate columns, stored as four
//              blocks of [16 gate rows | 16 up rows]; SwiGLU straight from tensor memory (a gate row and its up
//              row sit 16 lanes apart in one warp), rounded to bf16, written as the B tiles kernel B reads.
//   kernel B   D[128, N] = Wd_tile[128 hidden rows, I] * A[N, I]^T, scaled by the slot's routing weight and
//              added into y[row, :] with fp32 reductions (a row's k experts meet there).
//
// Both are the same pipeline with a different epilogue.  A unit of work is (tile, chunk): a tile is 64 intermediate
// columns (A) or 128 hidden rows (B) of an activated expert, a chunk up to 128 of its token-slots.  The list of units
// is cut into one contiguous range per CTA (grid = number of SMs) of equal cost, no CTA ever waits for another one,
// nothing is exchanged between CTAs inside a kernel.
//
// Operands.  Weights are read from a tile-major copy made once per layer (team_pack_w_tiles): every
// [128 rows x 64 k] bf16 tile is 16 KB contiguous and already in the 128-byte-swizzled K-major layout the
// tensor core reads, so a pipeline stage is one-dimensional bulk copies (weight tiles from HBM with an evict-first hint,
// kernel B's token tiles from L2) that complete on the stage's mbarrier.  Kernel A fetches its token tiles from the rows of
// x themselves, 16 bytes per asynchronous copy; kernel B's are what kernel A wrote.  (A kernel in front that gathered the
// rows into tiles, every row written once per expert that chose it, held up the first weights by 5 us at 128 rows, 11 at
// 1024 and 20 at 2048.)
//
// Plan.  The selection leaves a bit matrix [expert][row] of who chose whom and the experts' numbers of slots.  From these every
// CTA of either kernel forms the experts' places and its own range by itself: nothing is sorted, nobody waits for a table.
//
// Warp roles: warp 0 = producer (one lane issues the bulk copies), warp 1 = MMA issuer and owner of the tensor memory
// (converged warp, one elected lane issues), warps 2-9 = epilogue (one lane quarter of one accumulator each), kernel A: warps
// 10-13 = token rows.  Two buffers of two accumulators of 128 columns: the tensor core works on the next step while the
// epilogue drains the previous one.  Every wait is bounded; on expiry the kernel records TEAM_ERR_TIMEOUT, leaves its loops,
// lets its copies land, frees its tensor memory and returns.
#include "team_common.cuh"
#include "team_tc_ptx.cuh"

namespace team {

constexpr int kLoadWarps = 4;                  // kernel A: warps that fetch token rows
constexpr int kTileThreadsA = 448, kTileThreadsB = 320;
constexpr int kTileBytes = 128 * 128;          // one [128 rows x 64 bf16] tile
constexpr int kTileElems = kTileBytes / 2;
constexpr int kTileStages = 4;                 // pipeline stages: three operand tiles each
constexpr int kStageBytes = 3 * kTileBytes;
constexpr int kTileChunk = 128;                // token-slots per chunk at most (N of the MMA)
constexpr int kTmemCols = 512;                 // two buffers of two accumulators of 128 columns
constexpr int kEpiWarps = 8;                   // two warpgroups, one per accumulator of a step
// Rows that a warp of kernel A lists once per expert, where kernel B keeps its slots' tables.  (16 KB more for all 2048 leave the
// kernel in front no room on the SM: 0.4 us of calls of 270 and 480 rows.)
constexpr int kListRows = 1024;
static_assert(kLoadWarps * kListRows * 2 <= kEpiWarps * kTileChunk * 8, "lists in the place of the tables");
constexpr int kMaxExp = TEAM_MAX_EXPERTS + TEAM_MAX_SHARED;
constexpr int kTileSmemBytes = 1024 + kTileStages * kStageBytes + kEpiWarps * kTileChunk * 8 + 256 + (3 * kMaxExp + 8) * 4 + 2 * kTileChunk * 2;

enum { kEpiSwiglu = 0, kEpiCombine = 1 };

__host__ __device__ inline int pad16(int n) { return (n + 15) & ~15; }
// Rows of an expert with n token-slots in the gathered tables: all its chunks but the last are full.
__host__ __device__ inline int padded_rows(int n) { return n / kTileChunk * kTileChunk + pad16(n % kTileChunk); }

// What an expert with n token-slots costs per weight tile, 256 a step (TileWalk): one chunk takes a step for two tiles, more
// take one for two chunks of a tile.  Where many experts have several chunks a step's time hardly depends on its rows: 6.6 us
// + 2.6 per weight tile in the gate/up pass of 2048 rows (hidden 2048, 128 experts of 768 columns), where counting bytes left
// the CTAs between 108 and 172 us of work.  A few such experts among many of one chunk (a shared expert) keep their CTAs busy
// longer: half their rows are added then.  Without and with that, us: 185 rows and a shared expert 122.5, 116.5, 486 rows 180,
// 152, 204 rows 174.5, 153; with it 2048 rows would take 330 in place of 305.
// The same holds for an expert of one chunk with more than four times the mean (a shared expert of fewer rows): half its rows
// are what its token tile adds to a step's bytes.  Without and with that, us, with a shared expert: 128 rows of one sequence
// 131.3, 117.5, of 16 sequences 210.7, 198.7 (256 experts of 512 columns, hidden 2048), of one sequence 139.9, 130.1 (128 of 768).
__device__ __forceinline__ int tile_cost(int n, bool few_large, int used, int total) {
  const int chunks = (n + kTileChunk - 1) / kTileChunk;
  const bool large = chunks <= 1 ? n > 32 && n * used > 4 * total : few_large;
  return (chunks <= 1 ? chunks * 128 : (chunks + 1) / 2 * 256) + (large ? padded_rows(n) / 2 : 0);
}

// ---------------------------------------------------------------------------------------------------------
// Weight layout: row-major -> tile-major, pre-swizzled (once per layer)
// ---------------------------------------------------------------------------------------------------------
// gu tiles: [e][u = I/64][kb = H/64][128 rows][64 k]; row r = blk*32 + m*16 + i16 holds (m ? W_up : W_gate)
//           [e][u*64 + blk*16 + i16][kb*64 ...]; 16-byte piece p of row r is stored at piece p ^ (r & 7).
// d tiles:  [e][ht = H/128][kb = I/64][128 rows][64 k]; row r holds W_down[e][ht*128 + r][kb*64 ...].
__global__ void __launch_bounds__(256)
k_pack_w_tiles(const uint4* __restrict__ w_gate, const uint4* __restrict__ w_up, const uint4* __restrict__ w_down,
               uint4* __restrict__ gu, uint4* __restrict__ dt, int n_exp, int H, int I) {
  const int U = I / 64, KB = H / 64, HT = H / 128;
  const size_t per_e = (size_t)I * H / 8;                       // 16-byte pieces per expert and matrix
  const size_t n_gu = 2 * per_e * n_exp, n_d = per_e * n_exp;
  for (size_t o = (size_t)blockIdx.x * blockDim.x + threadIdx.x; o < n_gu + n_d; o += (size_t)gridDim.x * blockDim.x) {
    if (o < n_gu) {
      const int pc = (int)(o & 7), r = (int)((o >> 3) & 127);
      const size_t tile = o >> 10;                              // 1024 pieces per tile
      const int kb = (int)(tile % KB), u = (int)((tile / KB) % U), e = (int)(tile / ((size_t)KB * U));
      const int blk = r >> 5, m = (r >> 4) & 1, i16 = r & 15, lc = pc ^ (r & 7);
      const size_t src = ((size_t)e * I + u * 64 + blk * 16 + i16) * (H / 8) + kb * 8 + lc;
      gu[o] = m ? w_up[src] : w_gate[src];
    } else {
      const size_t q = o - n_gu;
      const int pc = (int)(q & 7), r = (int)((q >> 3) & 127);
      const size_t tile = q >> 10;
      const int kb = (int)(tile % U), ht = (int)((tile / U) % HT), e = (int)(tile / ((size_t)U * HT));
      const int lc = pc ^ (r & 7);
      const size_t src = ((size_t)e * H + ht * 128 + r) * (I / 8) + kb * 8 + lc;
      dt[q] = w_down[src];
    }
  }
}

cudaError_t launch_pack_w_tiles(const void* w_gate, const void* w_up, const void* w_down, void* gu, void* dt, int n_exp,
                                int H, int I, cudaStream_t s) {
  const size_t n = 3 * (size_t)I * H / 8 * n_exp;
  const int grid = (int)((n + 255) / 256 < 148 * 16 ? (n + 255) / 256 : 148 * 16);
  k_pack_w_tiles<<<grid, 256, 0, s>>>(static_cast<const uint4*>(w_gate), static_cast<const uint4*>(w_up),
                                      static_cast<const uint4*>(w_down), static_cast<uint4*>(gu), static_cast<uint4*>(dt),
                                      n_exp, H, I);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------------------
// Who chose whom, from the rows' choices: for calls that export routing tables, whose selection kernel writes those and leaves
// the marks to this one (callers see the number of launches; calls without exports have them set where a row is routed)
// ---------------------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_mark_choices(const int32_t* topk_idx, const uint8_t* tok_class, uint32_t* bits, Dims d) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int W1 = bit_words(d.T), per_row = d.k + d.ns;
  for (int i = blockIdx.x * 256 + threadIdx.x; i < d.T * per_row; i += gridDim.x * 256) {
    const int t = i / per_row, j = i - t * per_row;
    const int e = j < d.k ? topk_idx[t * d.k + j] : (tok_class[t] != TEAM_CLS_SKIP ? d.E + j - d.k : -1);
    if ((e >= d.elo && e < d.ehi) || e >= d.E) {
      atomicOr(bits + e * W1 + (t >> 5), 1u << (t & 31));
      atomicAdd(bits + (d.E + d.ns) * W1 + e, 1u);
    }
  }
}

// ---------------------------------------------------------------------------------------------------------
// The plan: places of the experts in the activation tables, costs in front of them, where this CTA's range begins and ends
// ---------------------------------------------------------------------------------------------------------
struct PlanSmem {
  int32_t* n;              // [EN] token-slots of the expert
  int32_t* row0;           // [EN] its first row in the tables
  int32_t* cost;           // [EN + 1] cost of the experts in front of it
  int32_t* range;          // [2][3] begin and end of the range: expert, unit of pass A, of pass B
};

__device__ __forceinline__ void block_plan(const PlanSmem& s, const uint32_t* counts, int EN, int I, int H) {
  __shared__ int4 s_tot[(kMaxExp + 31) / 32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int used_warps = (EN + 31) >> 5;
  int n_slots = 0, rows_in = 0, cost_in = 0;
  if (warp < used_warps) {                                      // expert = thread
    n_slots = tid < EN ? (int)__ldcg(counts + tid) : 0;
    const int used = __popc(__ballot_sync(0xffffffffu, n_slots > 0)), large = __popc(__ballot_sync(0xffffffffu, n_slots > kTileChunk));
    const int total = __reduce_add_sync(0xffffffffu, n_slots);
    if (lane == 0) s_tot[warp] = make_int4(used, large, total, 0);
  }
  __syncthreads();
  int used = 0, large = 0, total = 0;
  for (int w = 0; w < used_warps; ++w) {
    used += s_tot[w].x;
    large += s_tot[w].y;
    total += s_tot[w].z;
  }
  const bool few_large = 4 * large < used;
  __syncthreads();
  if (warp < used_warps) {
    rows_in = padded_rows(n_slots);
    cost_in = tile_cost(n_slots, few_large, used, total);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int r1 = __shfl_up_sync(0xffffffffu, rows_in, o), c1 = __shfl_up_sync(0xffffffffu, cost_in, o);
      if (lane >= o) { rows_in += r1; cost_in += c1; }
    }
    if (lane == 31) s_tot[warp] = make_int4(rows_in, cost_in, 0, 0);
  }
  __syncthreads();
  if (tid < EN) {
    int rows = rows_in - padded_rows(n_slots), cost = cost_in - tile_cost(n_slots, few_large, used, total);
    for (int w = 0; w < warp; ++w) {
      rows += s_tot[w].x;
      cost += s_tot[w].y;
    }
    s.n[tid] = n_slots;
    s.row0[tid] = rows;
    s.cost[tid] = cost;
    if (tid == EN - 1) s.cost[EN] = cost + tile_cost(n_slots, few_large, used, total);
  }
  __syncthreads();
  if (tid < 2) {
    // where CTA b begins: the expert that holds cost total * b / CTAs, and the unit inside it (32 bits: 260 experts of 2048
    // slots cost 260 * 3072)
    const int b = blockIdx.x + tid, at = (int)((uint32_t)s.cost[EN] * b / gridDim.x);
    int lo = 0, hi = EN;                                        // the last expert with cost[e] <= at (empty ones: cost 0)
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (s.cost[mid] <= at) lo = mid; else hi = mid;
    }
    const uint32_t cost = s.cost[lo + 1] - s.cost[lo], off = at - s.cost[lo];
    const int chunks = (s.n[lo] + kTileChunk - 1) / kTileChunk;
    auto part = [&](uint32_t tiles) {
      if (cost == 0) return 0;                                  // behind the last expert
      const int per_tile = (chunks + 1) / 2;                    // steps of a tile (chunks > 1)
      // in quarters of a step (one chunk: of two tiles) or halves of one
      const uint32_t f = chunks == 1 ? 2 : 2 * per_tile;
      const int q = (int)(tiles < 16384u ? off * tiles * f / cost : (uint32_t)((unsigned long long)off * tiles * f / cost));
      if (chunks == 1) {
        // Ranges begin at whole steps where the CTAs then have hardly more steps each than there are on average, else in the
        // middle of a step, too, which costs the second CTA a step of one tile.  Allowed up to 1.07, 1.15, 1.3 times the average and
        // always, us: 128 rows 131.7, 130.5, 131.6, 131.7, block of 32 x 4 872, 851, 845, 851, 1024 rows 219.5, 219.4, 223.9, 223.9,
        // 2048 rows 301 each.  With 11 tiles (185 rows) whole steps were slower, 123.7 and 127.4: an odd tile is a step by itself.
        const float steps = (float)s.cost[EN] * tiles / (256.f * gridDim.x);
        const bool whole = (tiles & 1) == 0 && ceilf(steps) <= 1.15f * steps;
        return min((q >> 2) * 2 + (whole ? (q & 2) : (q & 3) == 3 ? 2 : (q & 3) ? 1 : 0), (int)tiles);
      }
      const int st = (q + 1) / 2;                               // the nearest step
      return min(st / per_tile * chunks + st % per_tile * 2, chunks * (int)tiles);
    };
    s.range[3 * tid] = lo;
    s.range[3 * tid + 1] = part(I / 64);
    s.range[3 * tid + 2] = part(H / 128);
  }
  __syncthreads();
}

// ---------------------------------------------------------------------------------------------------------
// The grouped GEMM
// ---------------------------------------------------------------------------------------------------------
struct TileArgs {
  const __nv_bfloat16* w_tiles;   // [e][tile][kb][16 KB]
  const __nv_bfloat16* x;         // pass A: [T, H]
  const uint32_t* bits;           // [EN][bit_words(T)] rows that chose the expert, then [EN] how many
  const int32_t* topk_idx;        // [T, k]
  const float* topk_w;
  const uint8_t* tok_class;       // [T]
  int32_t* row_of;                // [padded rows] output row of the slot: written by pass A
  float* w_of;                    // [padded rows] its routing weight
  __nv_bfloat16* act;             // activations, per chunk [u][np rows][64 columns] swizzled, from its first row * I elements
  float* y;                       // [T, H]
  int32_t* status;
  int n_k;                        // k-blocks of 64: H/64 (A) or I/64 (B)
  int tiles;                      // weight tiles per expert: I/64 (A) or H/128 (B)
  int H, I, T, E, k, EN;
};

// The walk over a CTA's range of (tile, chunk) units, tile by tile and inside a tile chunk by chunk.  A step computes up
// to two accumulators from three operand tiles: two neighbouring weight tiles for an expert of one chunk (the token
// tile is fetched once for both), or one weight tile for two chunks of a larger expert (its weights cross HBM once up to
// 256 token-slots; read again one chunk later they would come from HBM again, because the other CTAs stream more than L2
// holds in between: gate/up pass of 2048 rows of the SDAR shape 255 us that way, 168 us this way).
struct TileWalk {
  const PlanSmem p;
  int x, u, x_end, u_end, tiles;
  int row0, n, chunks, limit;
  int j, nt, c, nc, first;        // current step: tiles j .. j + nt - 1, chunks c .. c + nc - 1 of rows first, first + 128
  int slots[2];                   // token-slots of the two chunks
  __device__ __forceinline__ void load() {
    row0 = p.row0[x];
    n = p.n[x];
    chunks = (n + kTileChunk - 1) / kTileChunk;
    limit = x == x_end ? u_end : chunks * tiles;
  }
  __device__ __forceinline__ TileWalk(const PlanSmem& plan, int t, bool phase_b) : p(plan), tiles(t) {
    x = p.range[0];
    x_end = p.range[3];
    u = p.range[phase_b ? 2 : 1];
    u_end = p.range[phase_b ? 5 : 4];
    if (x < x_end || u < u_end) load();
  }
  __device__ __forceinline__ bool next() {
    if (x == x_end && u >= u_end) return false;
    while (u >= limit) {                                        // experts without slots have no units
      ++x;
      u = 0;
      if (x == x_end && u >= u_end) return false;
      load();
    }
    c = 0;
    nt = nc = 1;
    if (chunks == 1) {
      j = u;
      if ((u & 1) == 0 && u + 1 < limit) nt = 2;
    } else {
      j = u / chunks;
      c = u - j * chunks;
      if ((c & 1) == 0 && c + 1 < chunks && u + 1 < limit) nc = 2;
    }
    u += nt * nc;
    first = row0 + c * kTileChunk;
    slots[0] = min(kTileChunk, n - c * kTileChunk);
    slots[1] = min(kTileChunk, n - (c + 1) * kTileChunk);
    return true;
  }
  __device__ __forceinline__ int accs() const { return nt * nc; }
  // of accumulator i: its tile, its chunk's first gathered row and token-slots
  __device__ __forceinline__ int tile(int i) const { return nt == 2 ? j + i : j; }
  __device__ __forceinline__ int row(int i) const { return nc == 2 ? first + i * kTileChunk : first; }
  __device__ __forceinline__ int n_of(int i) const { return nc == 2 && i ? slots[1] : slots[0]; }
};

// The rows of an expert of one chunk, by one warp: a slot's number is its row's rank among the expert's.  Every lane walks the
// bits of its own words: such an expert has few of a word's rows, or there are few words.
__device__ __forceinline__ void list_chunk(uint16_t* list, const uint32_t* words, int W) {
  const int lane = threadIdx.x & 31;
  int run = 0;
  __syncwarp();
  for (int w0 = 0; w0 < W; w0 += 32) {
    const int w = w0 + lane;
    const uint32_t word = w < W ? __ldcg(words + w) : 0u;
    int incl = __popc(word);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int up = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += up;
    }
    int at = run + incl - __popc(word);
    for (uint32_t m = word; m != 0u; m &= m - 1u, ++at)
      if (at < kTileChunk) list[at] = (uint16_t)(w * 32 + __ffs(m) - 1);
    run += __shfl_sync(0xffffffffu, incl, 31);
  }
  __syncwarp();
}

// The rows of an expert's slots [begin, begin + n) where it has more than one chunk.  Two words of 32 rows per lane are fetched and
// summed up; then, unless they have few bits each, every word with a slot of the range is spread over the lanes, one row each.
// (Every lane its own words in any case: 9000 clock cycles where half of 2048 rows chose the expert; 2048 rows x 8 choices of 16
// experts, hidden 256, 1024 columns 110.2 -> 101.6 us, 24 experts x 6 choices, hidden 1536, 704 columns 139.4 -> 133.8.  This way
// in any case: 1020 rows and a shared expert 53.6 -> 54.3.  Functions of their own, and only for these experts: inlined, the
// loop over the token rows came out slower, 141.2; for experts of one chunk 11 rows of 199 experts took 32.7 us in place of 31.7.)
__device__ __noinline__ void list_rows(uint16_t* list, const uint32_t* words, int W, int begin, int n) {
  static_assert(TEAM_MAX_ROWS <= 64 * 32, "two words per lane");
  const int lane = threadIdx.x & 31;
  uint32_t word = lane < W ? __ldcg(words + lane) : 0u;
  const uint32_t word2 = lane + 32 < W ? __ldcg(words + lane + 32) : 0u;
  int before = -begin;                                         // slots in front of these words'
  __syncwarp();
#pragma unroll 1
  for (int row0 = 0; row0 < W * 32; row0 += 1024, word = word2) {
    int at = __popc(word);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int up = __shfl_up_sync(0xffffffffu, at, o);
      if (lane >= o) at += up;
    }
    const int slots = __popc(word), end = before + at;
    before = __shfl_sync(0xffffffffu, end, 31);
    at = end - slots;                                          // rank of the word's first slot
    uint32_t m = __ballot_sync(0xffffffffu, slots > 0 && at < n && end > 0);
    if ((int)__reduce_max_sync(0xffffffffu, (uint32_t)slots) <= 3 * ((__popc(m) + 3) >> 2)) {      // an exchange takes as long as 3 bits
      for (uint32_t mine = word; mine != 0u; mine &= mine - 1u, ++at)
        if (at >= 0 && at < n) list[at] = (uint16_t)(row0 + lane * 32 + __ffs(mine) - 1);
      m = 0u;
      __syncwarp();
    }
#pragma unroll 1
    while (m != 0u) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {                            // four words' exchanges in flight (the last one again where there are fewer)
        const int w = __ffs(m) - 1;
        m = (m & (m - 1u)) != 0u || u == 3 ? m & (m - 1u) : m;
        const uint32_t bits = __shfl_sync(0xffffffffu, word, w);
        const int i = __shfl_sync(0xffffffffu, at, w) + __popc(bits & ((1u << lane) - 1u));
        if (((bits >> lane) & 1u) && i >= 0 && i < n) list[i] = (uint16_t)(row0 + w * 32 + lane);
      }
    }
  }
  __syncwarp();
}

// (output row, routing weight) of n token-slots of expert x (k choices per row, 0: a shared expert), for pass B, by one warp, with
// the loads of a lane's four slots in flight together.
__device__ __noinline__ void note_slots(int32_t* row_of, float* w_of, const uint16_t* list, int n, int x, const int32_t* topk_idx,
                                        const float* topk_w, int k) {
  constexpr int kPer = kTileChunk / 32;
  const int lane = threadIdx.x & 31;
  int row[kPer], choice[kPer];                   // choice -1: a shared expert
#pragma unroll
  for (int i = 0; i < kPer; ++i) {
    row[i] = lane + 32 * i < n ? list[lane + 32 * i] : -1;
    choice[i] = -1;
  }
#pragma unroll 4
  for (int c = 0; c < k; ++c)
#pragma unroll
    for (int i = 0; i < kPer; ++i)
      if (row[i] >= 0 && __ldcg(topk_idx + row[i] * k + c) == x) choice[i] = c;
#pragma unroll
  for (int i = 0; i < kPer; ++i)
    if (row[i] >= 0) {
      row_of[lane + 32 * i] = row[i];
      w_of[lane + 32 * i] = choice[i] >= 0 ? __ldcg(topk_w + row[i] * k + choice[i]) : 1.f;
    }
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

template <int EPI>
__global__ void __launch_bounds__(EPI == kEpiSwiglu ? kTileThreadsA : kTileThreadsB, 1) k_grouped_gemm(TileArgs a) {
  extern __shared__ unsigned char tile_smem_raw[];
  // 1024-byte alignment for the swizzled tiles
  unsigned char* smem = tile_smem_raw + ((1024u - (smem_u32(tile_smem_raw) & 1023u)) & 1023u);
  unsigned char* stages = smem;
  int32_t* tab_row = reinterpret_cast<int32_t*>(smem + kTileStages * kStageBytes);      // [8 epilogue warps][128]
  float* tab_w = reinterpret_cast<float*>(tab_row + kEpiWarps * kTileChunk);            // [8][128]
  uint64_t* bars = reinterpret_cast<uint64_t*>(tab_w + kEpiWarps * kTileChunk);
  uint64_t* bar_full = bars;                       // [stages] bytes of the stage have landed
  uint64_t* bar_empty = bars + kTileStages;        // [stages] the MMAs reading the stage are done
  uint64_t* bar_dfull = bars + 2 * kTileStages;    // [2] accumulators complete
  uint64_t* bar_dempty = bar_dfull + 2;            // [2] accumulators drained by the epilogue
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar_dempty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  static_assert((2 * kTileStages + 4) * 8 + 8 <= 256, "barriers must fit");
  PlanSmem plan;
  plan.n = reinterpret_cast<int32_t*>(reinterpret_cast<unsigned char*>(bars) + 256);
  plan.row0 = plan.n + kMaxExp;
  plan.cost = plan.row0 + kMaxExp;                 // [EN + 1]
  plan.range = plan.cost + kMaxExp + 1;            // [6]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (tid == 0) {
    for (int i = 0; i < kTileStages; ++i) {
      mbar_init(smem_u32(bar_full + i), EPI == kEpiSwiglu ? 1 + kLoadWarps : 1);
      mbar_init(smem_u32(bar_empty + i), 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(smem_u32(bar_dfull + i), 1);
      mbar_init(smem_u32(bar_dempty + i), kEpiWarps);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"((uint32_t)kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = warp_uniform(*tmem_slot);
  // Everything above overlaps the preceding kernel.  Pass A: the selection's outputs are complete from here, and pass B is let go
  // only now, so it finds them complete when it starts: it forms its plan and its producer fetches its first weights ahead of
  // the wait for pass A (128 rows 140.1 -> 138.7 us, 185 rows 127.9 -> 126.1).
  if (EPI == kEpiSwiglu) asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int W1 = bit_words(a.T);
  block_plan(plan, a.bits + (size_t)a.EN * W1, a.EN, a.I, a.H);
  if (EPI == kEpiCombine && warp != 0) asm volatile("griddepcontrol.wait;" ::: "memory");

  const int NK = a.n_k;
  TileWalk wk(plan, a.tiles, EPI == kEpiCombine);

  if (warp == 0) {
    // ------------------------------ producer ------------------------------
    const uint64_t pol = stream_policy();
    uint32_t it = 0;
    const uint32_t ahead = EPI == kEpiCombine ? min(kTileStages, NK) : 0;       // stages whose weights are fetched before the wait
    bool ok = true;
    while (ok && wk.next()) {
      const __nv_bfloat16* wsrc = a.w_tiles + ((size_t)wk.x * a.tiles + wk.j) * NK * kTileElems;
      const __nv_bfloat16* bsrc = a.act + (size_t)wk.first * a.I;                // pass B
      const int np0 = pad16(wk.slots[0]), np1 = wk.nc == 2 ? pad16(wk.slots[1]) : 0;
      // stage: weight tile | second weight tile or second token tile | token tile
      auto weights = [&](uint32_t s, int kb) {
        const uint32_t full = smem_u32(bar_full + s), dst = smem_u32(stages + (size_t)s * kStageBytes);
        mbar_expect_tx(full, (uint32_t)(wk.nt * kTileBytes + (EPI == kEpiCombine ? (np0 + np1) * 128 : 0)));
        bulk_g2s_stream(dst, wsrc + (size_t)kb * kTileElems, kTileBytes, full, pol);
        if (wk.nt == 2) bulk_g2s_stream(dst + kTileBytes, wsrc + (size_t)(NK + kb) * kTileElems, kTileBytes, full, pol);
      };
      if (EPI == kEpiCombine && it == 0) {
        if (lane == 0)
          for (uint32_t s = 0; s < ahead; ++s) weights(s, (int)s);
        __syncwarp();
        asm volatile("griddepcontrol.wait;" ::: "memory");
      }
      for (int kb = 0; kb < NK; ++kb, ++it) {
        const uint32_t s = it % kTileStages;
        if (!(ok = mbar_wait_warp<32>(smem_u32(bar_empty + s), ((it / kTileStages) & 1) ^ 1, abort_flag, a.status, 31))) break;
        if (lane == 0) {
          const uint32_t full = smem_u32(bar_full + s), dst = smem_u32(stages + (size_t)s * kStageBytes);
          if (it >= ahead) weights(s, kb);
          if (EPI == kEpiCombine) bulk_g2s(dst + 2 * kTileBytes, bsrc + (size_t)kb * np0 * 64, (uint32_t)np0 * 128, full);
          if (EPI == kEpiCombine && np1 > 0) bulk_g2s(dst + kTileBytes, bsrc + (size_t)NK * (kTileChunk * 64) + (size_t)kb * np1 * 64, (uint32_t)np1 * 128, full);
        }
        __syncwarp();
      }
    }
    if (EPI == kEpiCombine && it == 0) asm volatile("griddepcontrol.wait;" ::: "memory");      // no work: still ends behind the gate/up pass
    if (!ok) {
      // gave up: the copies already issued still land in this CTA's shared memory; give them time before the CTA exits
      for (int i = 0; i < 64; ++i) __nanosleep(1000);
    }
  } else if (warp == 1) {
    // ------------------------------ MMA issuer ------------------------------
    uint32_t it = 0, un = 0;
    bool ok = true;
    for (; ok && wk.next(); ++un) {
      const uint32_t idesc0 = make_idesc_bf16(pad16(wk.n_of(0))), idesc1 = make_idesc_bf16(pad16(wk.n_of(1)));
      const int accs = wk.accs();
      const uint32_t buf = un & 1;
      if (!(ok = mbar_wait_warp(smem_u32(bar_dempty + buf), ((un >> 1) & 1) ^ 1, abort_flag, a.status, 32))) break;
      tc_fence_after();
      const uint32_t acc = tmem_base + buf * 2 * kTileChunk;
      for (int kb = 0; kb < NK; ++kb, ++it) {
        const uint32_t s = it % kTileStages;
        if (!(ok = mbar_wait_warp(smem_u32(bar_full + s), (it / kTileStages) & 1, abort_flag, a.status, 33))) break;
        tc_fence_after();
        const uint32_t base = smem_u32(stages + (size_t)s * kStageBytes);
        const uint64_t d0 = make_kmajor_sw128_desc(base), d1 = make_kmajor_sw128_desc(base + kTileBytes),
                       d2 = make_kmajor_sw128_desc(base + 2 * kTileBytes);
        tc_mma_k64(acc, d0, d2, idesc0, kb != 0);
        if (accs == 2) {
          const uint64_t da = wk.nt == 2 ? d1 : d0, db = wk.nt == 2 ? d2 : d1;
          tc_mma_k64(acc + kTileChunk, da, db, idesc1, kb != 0);
        }
        tc_commit(smem_u32(bar_empty + s));
      }
      if (ok) tc_commit(smem_u32(bar_dfull + buf));
    }
  } else if (EPI == kEpiSwiglu && warp >= 2 + kEpiWarps) {
    // ------------------------------ token rows ------------------------------
    // Eight lanes copy the 128 bytes of a row's k-block, warp lw the rows 16 i + 4 lw .. + 3 of a tile.  A stage is announced
    // kLag stages later, when this thread's copies have landed and are made visible to the tensor core.
    constexpr int kLag = 2;
    const int lw = warp - 2 - kEpiWarps, piece = lane & 7, W = (a.T + 31) >> 5;
    uint16_t* tok_list = reinterpret_cast<uint16_t*>(tab_row) + lw * kListRows;      // rows of the expert's slots
    uint32_t it = 0;
    int cur_x = -1, cur_c = -1, cur_nc = 0;
    const __nv_bfloat16* src[2][8];
    bool ok = true;
    while (ok && wk.next()) {
      if (wk.x != cur_x || wk.c != cur_c || wk.nc != cur_nc) {
        // every warp makes a list of its own, so that no warp waits for one that has given up; once per expert where it holds all
        // of its rows, although the chunks come again with every tile
        const bool all = wk.n <= kListRows;
        if (wk.n <= kTileChunk) {
          if (wk.x != cur_x) list_chunk(tok_list, a.bits + (size_t)wk.x * W1, W);
        } else if (wk.x != cur_x || !all) {
          list_rows(tok_list, a.bits + (size_t)wk.x * W1, W, all ? 0 : wk.c * kTileChunk, all ? wk.n : wk.nc * kTileChunk);
        }
        const uint16_t* chunk = tok_list + (all ? wk.c * kTileChunk : 0);
        cur_x = wk.x;
        cur_c = wk.c;
        cur_nc = wk.nc;
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int n = i * 16 + lw * 4 + (lane >> 3);
            src[q][i] = q < wk.nc && n < wk.slots[q] ? a.x + (size_t)chunk[q * kTileChunk + n] * a.H + piece * 8 : nullptr;
          }
      }
      for (int kb = 0; kb < NK; ++kb, ++it) {
        const uint32_t s = it % kTileStages;
        if (!(ok = mbar_wait_warp<32>(smem_u32(bar_empty + s), ((it / kTileStages) & 1) ^ 1, abort_flag, a.status, 35))) break;
        const uint32_t dst = smem_u32(stages + (size_t)s * kStageBytes);
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int n = i * 16 + lw * 4 + (lane >> 3);
            if (src[q][i] != nullptr) cp_async16(dst + (q == 0 ? 2 : 1) * kTileBytes + n * 128 + ((piece ^ (n & 7)) << 4), src[q][i] + kb * 64);
          }
        asm volatile("cp.async.commit_group;" ::: "memory");
        if (it >= kLag) {
          asm volatile("cp.async.wait_group %0;" ::"n"(kLag) : "memory");
          fence_async_smem();
          __syncwarp();
          if (lane == 0) mbar_arrive(smem_u32(bar_full + (it - kLag) % kTileStages));
        }
      }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    fence_async_smem();
    __syncwarp();
    if (ok && lane == 0)
      for (uint32_t i = it > kLag ? it - kLag : 0; i < it; ++i) mbar_arrive(smem_u32(bar_full + i % kTileStages));
  } else {
    // ------------------------------ epilogue: warps 2-5 accumulator 0 of a step, warps 6-9 accumulator 1 ------------------------------
    const int ew = warp - 2, half = ew >> 2;
    const int q = warp & 3;                          // this warp's lane quarter of the accumulators
    const uint32_t lane_off = (uint32_t)(q * 32) << 16;
    if (EPI == kEpiSwiglu) {
      // output rows of computed tokens start from zero (pass B adds into them).  These warps have nothing else to do before the
      // first accumulators; done by the router, the stores held up the calls with many rows (2048 rows 316.5 -> 313.5 us, 1024
      // rows 227.6 -> 225.5)
      for (int t = blockIdx.x; t < a.T; t += gridDim.x)
        if (a.tok_class[t] != TEAM_CLS_SKIP)
          for (int i = ew * 32 + lane; i < a.H / 4; i += kEpiWarps * 32)
            reinterpret_cast<float4*>(a.y + (size_t)t * a.H)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    uint32_t un = 0;
    int tab_first = -1;
    bool ok = true;
    for (; ok && wk.next(); ++un) {
      const uint32_t buf = un & 1;
      const bool mine = half < wk.accs();
      const int j = wk.tile(half), first = wk.row(half), n_c = wk.n_of(half), np = pad16(n_c);
      if (EPI == kEpiSwiglu && (ew & 3) == 0 && half < wk.nc && (wk.n <= kTileChunk ? wk.j == 0 : wk.j == (wk.c >> 1) % a.tiles)) {
        // (output row, routing weight) of the expert's slots for pass B, noted by the CTA of one of its tiles, another one for every
        // pair of chunks: one warp per chunk, while it waits for the accumulators anyway.  (All pairs at the first tile, one slot
        // after the other: 2048 rows x 8 choices of 16 experts, hidden 256, 1024 columns 128.7 us, this way 110.2.)
        uint16_t* list = reinterpret_cast<uint16_t*>(plan.n + 3 * kMaxExp + 8) + half * kTileChunk;
        const uint32_t* bits = a.bits + (size_t)wk.x * W1;
        const int n_rows = wk.n_of(half), at = wk.first + half * kTileChunk, W = (a.T + 31) >> 5;
        if (wk.n <= kTileChunk) {
          list_chunk(list, bits, W);
          for (int n = lane; n < n_rows; n += 32) {
            const int row = list[n];
            int choice = -1;                             // -1: a shared expert
            if (wk.x < a.E)
#pragma unroll 4
              for (int i = 0; i < a.k; ++i)
                if (__ldcg(a.topk_idx + row * a.k + i) == wk.x) choice = i;
            a.row_of[at + n] = row;
            a.w_of[at + n] = choice >= 0 ? __ldcg(a.topk_w + row * a.k + choice) : 1.f;
          }
        } else {
          list_rows(list, bits, W, (wk.c + half) * kTileChunk, n_rows);
          note_slots(a.row_of + at, a.w_of + at, list, n_rows, wk.x, a.topk_idx, a.topk_w, wk.x < a.E ? a.k : 0);
        }
      }
      if (EPI == kEpiCombine && mine && first != tab_first) {
        // (output row, weight) of the chunk's slots: every epilogue warp keeps a copy of its own, refilled at its own pace
        __syncwarp();
        for (int n = lane; n < n_c; n += 32) {
          tab_row[ew * kTileChunk + n] = a.row_of[first + n];
          tab_w[ew * kTileChunk + n] = a.w_of[first + n];
        }
        tab_first = first;
        __syncwarp();
      }
      if (!(ok = mbar_wait_warp<32>(smem_u32(bar_dfull + buf), (un >> 1) & 1, abort_flag, a.status, 34))) break;
      tc_fence_after();
      const uint32_t acc = tmem_base + buf * 2 * kTileChunk + half * kTileChunk + lane_off;
      if (mine) {
        if (EPI == kEpiSwiglu) {
          // lanes 0-15 hold gate rows, lanes 16-31 the up rows of the same intermediate columns j*64 + q*16 + (lane & 15):
          // the lower half finishes slots c0 .. c0+3, the upper half c0+4 .. c0+7
          const bool is_gate = lane < 16;
          const int i = q * 16 + (lane & 15), tb = is_gate ? 0 : 4;
          __nv_bfloat16* dst = a.act + (size_t)first * a.I + (size_t)j * np * 64;   // this unit's [np][64] tile
          for (int c0 = 0; c0 < np; c0 += 8) {
            float v[8];
            tmem_ld8(acc + c0, v);
#pragma unroll
            for (int t = 0; t < 4; ++t) {
              const float o = __shfl_xor_sync(0xffffffffu, is_gate ? v[t + 4] : v[t], 16);
              const float g = is_gate ? v[t] : o;
              const float u = is_gate ? o : v[t + 4];
              const int n = c0 + tb + t;
              dst[(size_t)n * 64 + (((i >> 3) ^ (n & 7)) << 3) + (i & 7)] = __float2bfloat16_rn(g / (1.f + expf(-g)) * u);
            }
          }
        } else {
          const int32_t* rows = tab_row + ew * kTileChunk;
          const float* wts = tab_w + ew * kTileChunk;
          float* ycol = a.y + (size_t)j * 128 + q * 32 + lane;
          for (int c0 = 0; c0 < n_c; c0 += 8) {
            float v[8];
            tmem_ld8(acc + c0, v);
#pragma unroll
            for (int t = 0; t < 8; ++t) {
              const int n = c0 + t;
              if (n < n_c) atomicAdd(ycol + (size_t)rows[n] * a.H, wts[n] * v[t]);
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(bar_dempty + buf));
    }
  }

  // ------------------------------ teardown ------------------------------
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)kTmemCols) : "memory");
  }
}

// ---------------------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------------------
bool experts_tile_supported(int hidden, int inter) { return hidden % 128 == 0 && inter % 64 == 0; }
int experts_tile_chunk() { return kTileChunk; }
// Rows of the gathered tables: every slot, plus the padding of each expert's last chunk.
size_t experts_tile_rows(size_t slots, size_t n_experts) { return slots + 16 * n_experts; }

// The opt-in is per device and shared by all contexts.
cudaError_t configure_experts_tile() {
  cudaError_t e = cudaSuccess;
  for (const void* fn : {reinterpret_cast<const void*>(&k_grouped_gemm<kEpiSwiglu>), reinterpret_cast<const void*>(&k_grouped_gemm<kEpiCombine>)}) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kTileSmemBytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  }
  return e;
}

static cudaError_t launch_pdl(const void* fn, dim3 grid, dim3 block, size_t smem, cudaStream_t s, void* arg) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  void* params[1] = {arg};
  return cudaLaunchKernelExC(&cfg, fn, params);
}

cudaError_t launch_mark_choices(Workspace ws, Dims d, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  const int blocks = (d.T * (d.k + d.ns) + 255) / 256;
  cfg.gridDim = dim3(blocks < 148 ? blocks : 148);
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_mark_choices, (const int32_t*)ws.r.topk_idx, (const uint8_t*)ws.r.tok_class, ws.bits, d);
}

// gate/up + SwiGLU, down + combine: two launches chained with programmatic dependent launch
cudaError_t launch_experts_tile(const void* x, const void* gu_tiles, const void* d_tiles, Workspace ws, float* y, Dims d,
                                int grid, cudaStream_t s) {
  TileArgs a = {};
  a.x = static_cast<const __nv_bfloat16*>(x);
  a.bits = ws.bits;
  a.topk_idx = ws.r.topk_idx;
  a.topk_w = ws.r.topk_w;
  a.tok_class = ws.r.tok_class;
  a.row_of = ws.tile_row;
  a.w_of = ws.tile_w;
  a.act = ws.tile_act;
  a.y = y;
  a.status = ws.status;
  a.H = d.H;
  a.I = d.I;
  a.T = d.T;
  a.E = d.E;
  a.k = d.k;
  a.EN = d.E + d.ns;
  a.w_tiles = static_cast<const __nv_bfloat16*>(gu_tiles);
  a.n_k = d.H / 64;
  a.tiles = d.I / 64;
  cudaError_t e = launch_pdl(reinterpret_cast<const void*>(&k_grouped_gemm<kEpiSwiglu>), dim3(grid), dim3(kTileThreadsA), kTileSmemBytes, s, &a);
  if (e != cudaSuccess) return e;
  a.w_tiles = static_cast<const __nv_bfloat16*>(d_tiles);
  a.n_k = d.I / 64;
  a.tiles = d.H / 128;
  return launch_pdl(reinterpret_cast<const void*>(&k_grouped_gemm<kEpiCombine>), dim3(grid), dim3(kTileThreadsB), kTileSmemBytes, s, &a);
}

}  // namespace team
