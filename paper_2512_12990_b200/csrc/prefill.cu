// Prefill of one MoE layer from bit-sliced AMAT weights: many tokens at once, so the expert FFN is a
// genuine dense contraction (Section 3 of the paper: prefill loads every expert of a layer).  Section 6.3 notes
// that prefill wants high-bit computation; the per-expert precision flag here is this library's generalisation
// (an expert can also be run from its MSB slice alone), which the mixed-precision prefill benchmark uses.
//
// Steps, all on the device, five or six launches chained by programmatic dependent launch:
//   1. plan: count the tokens of every routed expert, give every (token, expert) pair a row - the experts' rows one
//      after the other, without padding - and sort the experts by their number of tokens;
//   2. scatter x (bf16) into that order as fp16 (exact for every bf16 value in fp16's normal range);
//   3. grouped GEMM 1: per tile  H = silu(X Wg^T) * (X Wu^T)  (fp16 out);
//   4. grouped GEMM 2: per tile  Yrow = H Wd^T  (fp32 out, one row per (token, expert) pair);
//   5. combine: y[t] = sum_j w[t,j] Yrow[pos(t,j)] + shared experts, in list order (deterministic).
// In both GEMMs the weight tile is brought from the nibble planes to fp16 on the fly - the integer q - zp from both
// slices, 2^shift (q_msb - (zp >> shift)) from the MSB slice alone, both exact in fp16 - straight into tensor memory
// and multiplied on the 5th-generation tensor cores (tcgen05.mma, fp16 x fp16 -> fp32).  The scale belongs to a
// quantisation group: a group's sums are read from tensor memory and added to fp32 registers with one
// multiply-add by the scale.  No weight is rounded anywhere.
#include <cuda.h>  // CUtensorMap (types only; the encoder is fetched through the runtime)
#include <cuda_fp16.h>
#include <stddef.h>

#include "common.cuh"

namespace slicemoe {

constexpr int kPfTileN = 192, kPfNarrowN = 96;  // most token rows of a tile: the wide form, the narrow one
constexpr int kPfTileB = 128;  // weight rows per tile: 64 gate + 64 up columns of h (GEMM 1), 128 columns of y (GEMM 2)
constexpr int kPfChunkK = 128;  // contraction columns per pipeline step (two plane blocks; every width is a multiple)

// An expert with tokens, as the GEMMs see it; sorted, the longest work items first.
struct PfRun {
  int expert;             // routed: 0 .. E - 1, shared: E ..
  int count, tiles;       // tokens; tiles of equal width (up to 16) they are cut into
  int in_row, out_row;    // first row in the gathered x; first row of h and of the result rows
  int items1, items2;     // work items before this run's in GEMM 1 and GEMM 2
  int pad_;
};
struct PfHead {
  int runs;
  int items1, items2;     // work items in all
  int next1, next2;       // next work item to hand out
};

constexpr int kPfSmemExperts = 2048;
constexpr int kPfRankPairs = 4096;  // pairs that one block counts

// ---- workspace layout (host and device agree through this one function) --------------------------------
struct PfLayout {
  size_t head, counts, base, hist, runs, rank, posmap, gate, xs, h, yrow, total;
  int in_rows, out_rows, nexp_all, rank_blocks;
};
__host__ __device__ inline size_t pf_align(size_t v) { return (v + 255) & ~(size_t)255; }
__host__ __device__ inline PfLayout pf_layout(int T, int E, int k, int n_shared, int hidden, int inter, int shared_inter) {
  PfLayout L;
  L.nexp_all = E + n_shared;
  L.in_rows = T * k + (n_shared ? T : 0);  // the shared experts read the same rows
  L.out_rows = T * (k + n_shared);
  // beyond kPfSmemExperts the counters do not fit shared memory and one block counts them in the workspace
  L.rank_blocks = E > kPfSmemExperts ? 1 : (T * k + kPfRankPairs - 1) / kPfRankPairs;
  const int wide = inter > shared_inter ? inter : shared_inter;
  size_t o = 0;
  L.head = o;         o = pf_align(o + sizeof(PfHead));
  L.counts = o;       o = pf_align(o + sizeof(int) * L.nexp_all);
  L.base = o;         o = pf_align(o + sizeof(int) * L.nexp_all);
  L.hist = o;         o = pf_align(o + sizeof(int) * (size_t)L.rank_blocks * E);
  L.runs = o;         o = pf_align(o + sizeof(PfRun) * L.nexp_all);
  L.rank = o;         o = pf_align(o + sizeof(int) * (size_t)T * k);
  L.posmap = o;       o = pf_align(o + sizeof(int) * (size_t)T * (k + n_shared));
  L.gate = o;         o = pf_align(o + sizeof(float) * T);
  L.xs = o;           o = pf_align(o + sizeof(__half) * (size_t)L.in_rows * hidden);
  L.h = o;            o = pf_align(o + sizeof(__half) * (size_t)L.out_rows * wide);
  L.yrow = o;         o = pf_align(o + sizeof(float) * (size_t)L.out_rows * hidden);
  L.total = o;
  return L;
}

__device__ __forceinline__ void pf_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pf_dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ---- step 1: rows and work items ---------------------------------------------------------------------------
// A pair's row is its expert's first row, plus the pairs of the expert in the blocks of pairs before, plus its rank
// among its own block's: the rank is what the counting atomic returns.  Up to kPfRankPairs pairs the plan block counts them
// itself; above, a launch of its own does, a block per kPfRankPairs pairs.  (One block for all: 13 us for 8,192 pairs, 58 for
// 49,152, at the rate of one SM's shared-memory atomics.)  Which row a pair gets depends on the order of the atomics, the
// values computed for it do not.
constexpr int kPfPlanThreads = 1024;
struct PfPlanParams {
  const int32_t* ids;
  int T, k, E, n_shared;
  int per1_routed, per1_shared, per2;  // work items per tile: GEMM 1 of a routed / shared expert, GEMM 2
  int rank_blocks;
  int tile;             // most token rows of a tile
  PfHead* head;
  int *counts, *base;   // [experts]: counters that do not fit shared memory; first rows likewise
  int* hist;            // [block][E]: pairs of the expert in the block; the plan turns them into the block's first rows
  PfRun* runs;
  int* rank;            // [T k]
  unsigned* status;
};
// Ranks of the pairs [i0, i1) by the calling block; an id out of range gets rank -1.
__device__ __forceinline__ void pf_rank(const int32_t* ids, int i0, int i1, int E, int* counts, int* rank) {
  constexpr int kAhead = kPfRankPairs / kPfPlanThreads;
  for (int b = i0; b < i1; b += kPfRankPairs) {
    int e[kAhead];
#pragma unroll
    for (int a = 0; a < kAhead; ++a) {
      const int i = b + a * kPfPlanThreads + (int)threadIdx.x;
      e[a] = i < i1 ? ids[i] : -1;
    }
#pragma unroll
    for (int a = 0; a < kAhead; ++a) {
      const int i = b + a * kPfPlanThreads + (int)threadIdx.x;
      if (i < i1) rank[i] = e[a] >= 0 && e[a] < E ? atomicAdd(&counts[e[a]], 1) : -1;
    }
  }
}
__global__ void __launch_bounds__(kPfPlanThreads) pf_rank_kernel(const PfPlanParams p) {
  __shared__ int s_counts[kPfSmemExperts];
  pf_dep_launch();
  for (int e = threadIdx.x; e < p.E; e += kPfPlanThreads) s_counts[e] = 0;
  pf_dep_wait();  // the ids may be the work of the kernel before, which may also still read what is now the workspace
  __syncthreads();
  const int i0 = blockIdx.x * kPfRankPairs;
  pf_rank(p.ids, i0, min(i0 + kPfRankPairs, p.T * p.k), p.E, s_counts, p.rank);
  __syncthreads();
  for (int e = threadIdx.x; e < p.E; e += kPfPlanThreads) p.hist[(size_t)blockIdx.x * p.E + e] = s_counts[e];
}
// Exclusive block-wide scan of one value per thread; *total gets the sum.
__device__ int pf_block_scan(int v, int* warp_sums, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int inc = v;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int a = __shfl_up_sync(0xffffffffu, inc, off);
    if (lane >= off) inc += a;
  }
  __syncthreads();  // the previous scan's sums have been read
  if (lane == 31) warp_sums[warp] = inc;
  __syncthreads();
  int before = 0, sum = 0;
  const int w = warp_sums[lane];
  static_assert(kPfPlanThreads == 1024, "one warp sum per lane");
  before = __reduce_add_sync(0xffffffffu, lane < warp ? w : 0);
  sum = __reduce_add_sync(0xffffffffu, w);
  *total = sum;
  return before + inc - v;
}
__global__ void __launch_bounds__(kPfPlanThreads) pf_plan_kernel(const PfPlanParams p) {
  __shared__ int s_counts[kPfSmemExperts], s_base[kPfSmemExperts];
  __shared__ int s_sums[32];
  const int tid = threadIdx.x;
  const int n = p.E + p.n_shared;
  const bool fits = n <= kPfSmemExperts;
  int* counts = fits ? s_counts : p.counts;
  int* base = fits ? s_base : p.base;
  pf_dep_wait();
  pf_dep_launch();  // not before: the gather kernel reads x, which may be the work of the kernel before this one, without a wait
  const int npairs = p.T * p.k;
  const bool alone = p.rank_blocks == 1;
  for (int e = tid; e < n; e += kPfPlanThreads) {
    int c = e < p.E ? 0 : p.T;
    if (!alone && e < p.E) {
      // the blocks' counts become the pairs before each block
#pragma unroll 4
      for (int b = 0; b < p.rank_blocks; ++b) {
        const int h = p.hist[(size_t)b * p.E + e];
        p.hist[(size_t)b * p.E + e] = c;
        c += h;
      }
    }
    counts[e] = c;
  }
  if (tid == 0) {
    *p.status = 0u;
    p.head->next1 = p.head->next2 = 0;
  }
  __syncthreads();
  if (alone) {
    pf_rank(p.ids, 0, npairs, p.E, counts, p.rank);
    __syncthreads();
  }
  // rows: the routed experts' one after the other
  int rows = 0;
  for (int e0 = 0; e0 < p.E; e0 += kPfPlanThreads) {
    const int e = e0 + tid;
    int total;
    const int before = pf_block_scan(e < p.E ? counts[e] : 0, s_sums, &total);
    if (e < p.E) {
      const int first = rows + before;
      base[e] = first;
      if (alone) {
        p.hist[e] = first;
      } else {
        for (int b = 0; b < p.rank_blocks; ++b) p.hist[(size_t)b * p.E + e] += first;
      }
    }
    rows += total;
  }
  // runs: experts with tokens, shared ones first (their contraction in GEMM 2 is usually the longest), then by
  // falling number of tokens: handed out in this order, the longest items do not come last.  rank = number of
  // experts that come before.
  __syncthreads();
  for (int e = tid; e < n; e += kPfPlanThreads) {
    const int c = counts[e];
    if (c == 0) continue;
    int rank = 0;
    if (e >= p.E) {
      rank = e - p.E;
    } else {
      rank = p.n_shared;
      for (int o = 0; o < p.E; ++o) rank += counts[o] > c || (counts[o] == c && o < e);
    }
    PfRun r;
    r.expert = e;
    r.count = c;
    r.tiles = (c + p.tile - 1) / p.tile;
    r.in_row = e < p.E ? base[e] : npairs;
    r.out_row = e < p.E ? base[e] : npairs + (e - p.E) * p.T;
    r.items1 = r.items2 = r.pad_ = 0;
    p.runs[rank] = r;
  }
  __syncthreads();
  int live = 0, base1 = 0, base2 = 0;
  for (int r0 = 0; r0 < n; r0 += kPfPlanThreads) {
    // an expert's rank is below the number of experts with tokens: count them, and scan the runs' work items
    const int e = r0 + tid;
    int total;
    pf_block_scan(e < n && counts[e] > 0 ? 1 : 0, s_sums, &total);
    live += total;
  }
  for (int r0 = 0; r0 < live; r0 += kPfPlanThreads) {
    const int r = r0 + tid;
    int v1 = 0, v2 = 0, t1, t2;
    if (r < live) {
      const PfRun run = p.runs[r];
      v1 = run.tiles * (run.expert < p.E ? p.per1_routed : p.per1_shared);
      v2 = run.tiles * p.per2;
    }
    const int b1 = pf_block_scan(v1, s_sums, &t1);
    const int b2 = pf_block_scan(v2, s_sums, &t2);
    if (r < live) {
      p.runs[r].items1 = base1 + b1;
      p.runs[r].items2 = base2 + b2;
    }
    base1 += t1;
    base2 += t2;
  }
  if (tid == 0) {
    p.head->runs = live;
    p.head->items1 = base1;
    p.head->items2 = base2;
  }
}

// ---- step 2: scatter x into expert order, bf16 -> fp16 ---------------------------------------------------
// A block per token: the row is read once and written to the row of each of its pairs, and to the token's row for the shared
// experts, 16 bytes per thread and step (4 where x is not 16-byte aligned).  The pairs' rows are worked out on the way, and
// with a gated shared expert the token's gate sigmoid(gate_vec . x).  Bound: the writes.  (A warp per written row read every
// token's row k + 1 times: 17 us for 2,048 tokens x 5 rows, 53 for 8,192 x 7.)
constexpr int kPfGatherThreads = 256;
constexpr int kPfMaxSlots = SLICEMOE_MAX_TOP_K + SLICEMOE_MAX_SHARED;
struct PfGatherParams {
  const uint16_t* x;
  const int32_t* ids;
  const int *rank, *first;  // rank of a pair, [block][E] first rows
  int T, k, E, n_shared, hidden;
  int* posmap;
  __half* xs;
  const float* gate_vec;  // or null
  float* gate;
  unsigned* status;
};
template <int WORDS>
__global__ void __launch_bounds__(kPfGatherThreads) pf_gather_kernel(const PfGatherParams p) {
  __shared__ int s_row[SLICEMOE_MAX_TOP_K + 1];
  __shared__ float s_part[kPfGatherThreads / 32];
  const int t = blockIdx.x, tid = threadIdx.x, npairs = p.T * p.k;
  const uint32_t* src = reinterpret_cast<const uint32_t*>(p.x + (size_t)t * p.hidden);
  uint32_t in[WORDS];
  auto load = [&](int i) {
    if (i >= p.hidden / 2) return;
    if (WORDS == 4) {
      const uint4 v = __ldcg(reinterpret_cast<const uint4*>(src + i));
      in[0] = v.x; in[WORDS / 4] = v.y; in[WORDS / 2] = v.z; in[WORDS - 1] = v.w;
    } else {
      in[0] = __ldcg(src + i);
    }
  };
  load(tid * WORDS);
  pf_dep_wait();
  pf_dep_launch();  // not before: the GEMM kernel reads the plan without a wait
  if (tid < p.k + p.n_shared) {
    int pos;
    if (tid < p.k) {
      const int i = t * p.k + tid, e = p.ids[i], r = p.rank[i];
      pos = r >= 0 ? p.first[(size_t)(i / kPfRankPairs) * (p.E > kPfSmemExperts ? 0 : p.E) + e] + r : -1;
      if (r < 0) atomicOr(p.status, (unsigned)SLICEMOE_STATUS_BAD_EXPERT_ID);
      s_row[tid] = pos;
    } else {
      pos = npairs + (tid - p.k) * p.T + t;
    }
    p.posmap[t * (p.k + p.n_shared) + tid] = pos;
  }
  if (tid == 0 && p.n_shared > 0) s_row[p.k] = npairs + t;  // the shared experts read the same row
  const int copies = p.k + (p.n_shared > 0 ? 1 : 0);
  float dot = 0.f;
  __syncthreads();
  for (int i = tid * WORDS; i < p.hidden / 2; i += kPfGatherThreads * WORDS) {
    uint32_t out[WORDS];
#pragma unroll
    for (int j = 0; j < WORDS; ++j) {
      const float lo = __uint_as_float(in[j] << 16), hi = __uint_as_float(in[j] & 0xffff0000u);
      const __half2 h = __floats2half2_rn(lo, hi);
      out[j] = *reinterpret_cast<const uint32_t*>(&h);
      if (p.gate_vec) {
        const float2 gv = *reinterpret_cast<const float2*>(p.gate_vec + 2 * (i + j));
        dot = fmaf(gv.x, lo, dot);
        dot = fmaf(gv.y, hi, dot);
      }
    }
    load(i + kPfGatherThreads * WORDS);
    for (int c = 0; c < copies; ++c) {
      const int row = s_row[c];
      if (row < 0) continue;
      uint32_t* dst = reinterpret_cast<uint32_t*>(p.xs + (size_t)row * p.hidden) + i;
      if (WORDS == 4) *reinterpret_cast<uint4*>(dst) = make_uint4(out[0], out[WORDS / 4], out[WORDS / 2], out[WORDS - 1]);
      else *dst = out[0];
    }
  }
  if (p.gate_vec) {  // block sum in a fixed order: lanes by butterfly, then the warps one after the other
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, off);
    if ((tid & 31) == 0) s_part[tid >> 5] = dot;
    __syncthreads();
    if (tid == 0) {
      float sum = 0.f;
      for (int w = 0; w < kPfGatherThreads / 32; ++w) sum += s_part[w];
      p.gate[t] = 1.f / (1.f + expf(-sum));
    }
  }
}

// ---- steps 3 and 4: the grouped GEMM on the 5th-generation tensor cores ---------------------------------
// One persistent CTA per SM takes work items (128 weight rows x a tile of token rows) from a counter and computes the
// transposed product D[weight row, token].  Per 128-column step of the contraction:
//   - the token warp brings the token tile (rows of x or h, fp16) into shared memory with two TMA tiled copies of 64 columns,
//     128-byte swizzle: the B operand; and the raw words of the LSB planes with cp.async.  Another warp copies the MSB
//     planes' words, and scales and zero-points of 16 groups at a time;
//   - the weight warps (sets of four, taking the steps in turn) turn nibbles into fp16 integers d = q - zp (or
//     2^shift (q_msb - (zp >> shift))) and store them to tensor memory with tcgen05.st, one weight row per lane: the A
//     operand.  Weights never pass through shared memory as fp16;
//   - the MMA warp issues tcgen05.mma (M 128, K 16, N the tile's tokens) for one quantisation group at a time, into the two
//     fp32 accumulators in turn: one is read while the other is written;
//   - the sum warps read a group's sums with tcgen05.ld and add them, times the weight row's scale of that group, to fp32
//     registers: up to 96 tokens per warpgroup, one weight row per lane.
// After the last group the sum warps hold the item's result and write it: SwiGLU between gate and up rows (GEMM 1, one
// exchange between lanes), fp32 rows (GEMM 2).  A scheduler warp fetches items ahead and leaves their description in a ring in
// shared memory.
//
// Why integers and a read-out per group: the dequantised weight s (q - zp) has up to 20 significant bits.  Kept as the
// exact sum of two fp16 numbers every product is issued twice and the conversion is twice as long; the read-out costs half
// an instruction per value with packed multiply-adds.
// Two forms, by the widest tile.  192 tokens: the conversion of a weight tile is shared by all its tokens, and 96 sums per
// lane leave registers for eight weight warps.  96 tokens, where experts have few: the weights' way through the CTA bounds a
// step, not the products, and the shared and tensor memory that a narrower tile leaves take four steps of tokens and five of
// weights; one warpgroup reads the sums.  One accumulator for all of a tile's tokens: the MMA warp's serial path (a wait, eight
// products, commits) bounds a wide step, and two accumulators of half the tile's tokens run through it twice per group.
// Measured, one layer of 64 + 2 experts of 2048 x 1408 (us): 8,192 tokens 1499 -> 1425, 77 tokens 151 -> 135.5; 96 tokens
// through the wide form 155, through the narrow one 138.
// Every wait is bounded; a wait that runs out sets SLICEMOE_STATUS_WAIT_TIMEOUT and the CTA winds down (tensor memory is
// freed on every path).
constexpr int kUBoxRows = 32, kUBoxCols = 64; // a TMA copy brings a multiple of 32 token rows x 64 columns (128 bytes: the swizzle's span)
constexpr int kURawBlock = 1024;              // a row block's bytes of a step in one plane
constexpr int kURawStep = 16 * kURawBlock;    // [plane][row block]
constexpr int kUItemSlots = 8;
// Scales and zero-points of 16 quantisation groups at a time: [8 row blocks][16 groups][16 rows], 512 + 256 bytes each
constexpr int kUMetaGroups = 16, kUMetaStages = 2;
constexpr int kUMetaScale = kUMetaGroups * 32, kUMetaZp = kUMetaGroups * 16;
constexpr int kUMetaBytes = 8 * (kUMetaScale + kUMetaZp);
constexpr int kUTmemCols = 512;
constexpr int kUWCols = 64;                   // a step's weights in tensor memory: 128 fp16 per row
// What the width of the widest tile decides.  (Narrow, 77 tokens, us: four steps of tokens 135, three 140, two 156; six steps of
// raw words 138; three sets of weight warps 142, one 154; a second warpgroup for the sums 138.)
template <int TN>
struct UCfg {
  static constexpr bool wide = TN > kPfNarrowN;
  static constexpr int sum_wgs = wide ? 2 : 1;            // warpgroups that read sums, 96 tokens each
  static constexpr int half_max = 96;
  static constexpr int sets = 2;                          // sets of four weight warps; the steps go round them
  static constexpr int sum_warps = 4 * sum_wgs, warp_tok = sum_warps + 4 * sets, warp_mma = warp_tok + 1,
                       warp_sched = warp_tok + 2, warp_meta = warp_tok + 3;
  static constexpr int threads = 32 * (warp_tok + 4);
  // registers per thread: at launch, and the split, whose sum is at most the launch's
  static constexpr int regs = wide ? 96 : 128;
  static constexpr int regs_sum = 152, regs_weight = wide ? 72 : 128, regs_rest = wide ? 32 : 40;
  static_assert(32 * sum_warps * regs_sum + 128 * sets * regs_weight + 128 * regs_rest <= threads * regs, "register split");
  static constexpr int panel_bytes = TN * kUBoxCols * 2;  // half of a step's tile: 64 columns of all tokens
  static constexpr int tile_bytes = 2 * panel_bytes;
  static constexpr int accs = 2, acc_cols = TN;           // accumulators in tensor memory; the columns left take weights
  static constexpr int w_col0 = accs * acc_cols, w_stages = (kUTmemCols - w_col0) / kUWCols;
  static constexpr int tok_stages = wide ? 3 : 4;
  static constexpr int raw_stages = 4;                    // steps of raw plane words in shared memory or on their way to it
};
constexpr uint32_t kUWaitCycles = 2000000000u;
constexpr uint32_t kUCopyCycles = 2000000u;  // a millisecond: far more than any copy takes

// What a work item is.  [0] gate, [1] up in GEMM 1; both down in GEMM 2.  Pointers are at the item's first row block.
struct __align__(16) PfItem {
  const uint8_t* msb[2];
  const uint8_t* lsb[2];
  const uint16_t* scale[2];
  const uint8_t* zp[2];
  int nk;        // steps
  int n, n0;     // tokens of the tile, up to a multiple of 16; of the first warpgroup
  int count;     // tokens that are there
  int in_row, out_row;
  int col;       // first column of h or of y
  int prec;      // both slices (else the MSB slice alone)
  int stop;      // no more items
};

template <int TN>
struct USmem {
  using C = UCfg<TN>;
  static constexpr int tok = 0;
  static constexpr int raw = tok + C::tok_stages * C::tile_bytes;
  static constexpr int meta = raw + C::raw_stages * kURawStep;
  static constexpr int items = meta + kUMetaStages * kUMetaBytes;
  static constexpr int bars = items + kUItemSlots * (int)sizeof(PfItem);
  // barriers: weights of a step in, used / its tokens in, used / sums there [accumulator] / sums read [accumulator] / item
  // there, item read / scales and zero-points in, read / raw words in, read / drained
  static constexpr int w_full = 0, w_free = w_full + C::w_stages, tok_full = w_free + C::w_stages, tok_free = tok_full + C::tok_stages,
                       acc_full = tok_free + C::tok_stages, acc_free = acc_full + C::accs,
                       item_full = acc_free + C::accs, item_free = item_full + kUItemSlots, meta_full = item_free + kUItemSlots,
                       meta_free = meta_full + kUMetaStages, raw_full = meta_free + kUMetaStages, raw_free = raw_full + C::raw_stages,
                       drain = raw_free + C::raw_stages, nbars = drain + 1;
  static constexpr int tail = bars + nbars * 8;  // tensor-memory address, abort flag
  static constexpr int total = tail + 16;
};
template <int TN>
constexpr int kUSmemBytes = USmem<TN>::total + 1024 /* alignment slack */;
static_assert(USmem<192>::bars % 8 == 0 && USmem<192>::items % 16 == 0, "alignment");
static_assert(kUSmemBytes<192> <= 227 * 1024 && kUSmemBytes<kPfNarrowN> <= 227 * 1024, "shared memory budget");

constexpr int kUBoxes = kPfTileN / kUBoxRows;
struct PfMaps {
  CUtensorMap rows[kUBoxes];  // [i]: copies of 32 (i + 1) rows
};
struct PfGemmParams {
  const slicemoe_expert* experts;  // routed
  const slicemoe_expert* shared;
  const uint8_t* expert_prec;      // per routed expert: 1 = both slices, 0 = MSB slice only
  const PfRun* runs;
  PfHead* head;
  __half* h;                       // GEMM 1 output, GEMM 2 token operand [rows, ldh]
  float* yrow;                     // GEMM 2 output [rows, hidden]
  unsigned* status;
  int E, hidden, inter, shared_inter, ldh;
  int shift;  // b_high - b_low
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes) : "memory");
}
// Bounded wait for the phase of the given parity; false when the limit ran out or another role gave up.
__device__ __forceinline__ bool mbar_try(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
               : "=r"(ok)
               : "r"(smem_u32(b)), "r"(parity)
               : "memory");
  return ok != 0;
}
// The same without waiting at all.
__device__ __forceinline__ bool mbar_test(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile("{ .reg .pred p; mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
               : "=r"(ok)
               : "r"(smem_u32(b)), "r"(parity)
               : "memory");
  return ok != 0;
}
// The same, but the hardware may hold the thread for up to 10 ms while the phase is not there: a waiting warp then takes
// no issue slots from the others.
__device__ __forceinline__ bool mbar_try_long(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3; selp.u32 %0, 1, 0, p; }"
               : "=r"(ok)
               : "r"(smem_u32(b)), "r"(parity), "r"(10000000u)
               : "memory");
  return ok != 0;
}
// By a whole warp; every lane gets the same answer.  (No call: the sum warps have no registers to set aside for one.)
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, volatile int* abort_flag) {
  if (__all_sync(0xffffffffu, mbar_try(b, parity))) return true;  // the common case costs one instruction
  const uint32_t t0 = (uint32_t)clock64();
  for (;;) {
    if (__all_sync(0xffffffffu, mbar_try_long(b, parity))) return true;
    if (__any_sync(0xffffffffu, *abort_flag != 0 || (uint32_t)clock64() - t0 > kUWaitCycles)) return false;
  }
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global.L2::128B [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
// The calling thread's cp.async so far arrive at the barrier when they have landed.
__device__ __forceinline__ void cp_async_arrive(uint64_t* b) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(b)) : "memory");
}
__device__ __forceinline__ void bulk_copy(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory operand descriptor: K-major tile of 128-byte rows, 128-byte swizzle, 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFF) >> 4);  // start address / 16
  d |= (uint64_t)1 << 16;                   // leading byte offset (unused with swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;         // stride byte offset / 16
  d |= (uint64_t)1 << 46;                   // descriptor version
  d |= (uint64_t)2 << 61;                   // 128-byte swizzle
  return d;
}
// Instruction descriptor: fp16 x fp16 -> fp32, both operands K-major, M 128, N tokens (a multiple of 16).
__device__ __forceinline__ uint32_t umma_idesc(int n) { return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kPfTileB >> 4) << 24); }

// One lane of a converged warp.  The compiler knows that a branch on it is taken by one thread: what the branch computes
// stays on the uniform datapath, where the tensor instructions take their operands from.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}" : "=r"(p));
  return p != 0;
}

// D (tensor memory) (+)= A (tensor memory: lane = row, 32-bit column = two consecutive k) x B (shared memory).
__device__ __forceinline__ void umma_f16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}
// 16 rows x 32 columns: lane 4 g + c gives row g, columns 8 i + 2 c and the next, in registers 4 i and 4 i + 1, and row
// g + 8, the same columns, in registers 4 i + 2 and 4 i + 3.
__device__ __forceinline__ void tmem_st_16x32(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x256b.x4.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]),
      "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// With the wait in the same statement: nothing that uses the registers can come between.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
// Two fp32 multiply-adds in one instruction: acc += v * s, s in both halves of ss.
__device__ __forceinline__ void fma2(uint64_t& acc, uint32_t v0, uint32_t v1, uint64_t ss) {
  asm("{\n .reg .b64 v;\n mov.b64 v, {%1, %2};\n fma.rn.f32x2 %0, v, %3, %0;\n}" : "+l"(acc) : "r"(v0), "r"(v1), "l"(ss));
}
__device__ __forceinline__ float half_of(uint64_t v, int i) { return __uint_as_float((uint32_t)(v >> (32 * i))); }

__device__ __forceinline__ PfRun pf_load_run(const PfRun* at) {
  return {__ldcg(&at->expert), __ldcg(&at->count), __ldcg(&at->tiles), __ldcg(&at->in_row), __ldcg(&at->out_row), __ldcg(&at->items1), __ldcg(&at->items2), 0};
}
// The run that a work item belongs to: the last one whose first item is not above it.  Whole warp, 32 runs a step.
template <int PHASE>
__device__ __forceinline__ int u_find_run(const PfRun* runs, int n, int item, int lane) {
  int lo = 0;  // the answer is in [lo, n)
  int step = 1;
  while (step * 32 < n) step *= 32;
  for (; step >= 1; step >>= 5) {
    const int r = lo + lane * step;
    const bool below = r < n && __ldcg(PHASE == 1 ? &runs[r].items1 : &runs[r].items2) <= item;
    lo += (__popc(__ballot_sync(0xffffffffu, below)) - 1) * step;
    if (step == 1) break;
  }
  return lo;
}

// One plane of an item's eight row blocks for one step, 1024 bytes each, by one warp: `first` and `second` are the lane's place
// in the first block of gate and up (whose blocks alternate) or of down, `stride` the bytes from one block to the next.
template <int PHASE>
__device__ __forceinline__ void u_copy_raw(uint32_t dst, const uint8_t* first, const uint8_t* second, uint32_t stride) {
#pragma unroll
  for (int b = 0; b < 8; ++b) {
    const uint8_t* src = PHASE == 1 ? (b & 1 ? second : first) + (size_t)(b >> 1) * stride : first + (size_t)b * stride;
    cp_async16(dst + b * kURawBlock, src);
    cp_async16(dst + b * kURawBlock + 512, src + 512);
  }
}

template <int G, int PHASE, int TN>
__global__ void __launch_bounds__(UCfg<TN>::threads, 1) pf_umma_kernel(const PfGemmParams p, const __grid_constant__ PfMaps maps) {
  using C = UCfg<TN>;
  using S = USmem<TN>;
  constexpr int LG = G == 128 ? 7 : (G == 64 ? 6 : 5);
  extern __shared__ uint8_t u_smem_raw[];
  uint8_t* smem = u_smem_raw + ((1024 - (smem_u32(u_smem_raw) & 1023)) & 1023);
  PfItem* items = reinterpret_cast<PfItem*>(smem + S::items);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + S::bars);
  uint64_t *w_full = bars + S::w_full, *w_free = bars + S::w_free, *tok_full = bars + S::tok_full,
           *tok_free = bars + S::tok_free, *acc_full = bars + S::acc_full,
           *acc_free = bars + S::acc_free, *item_full = bars + S::item_full, *item_free = bars + S::item_free,
           *meta_full = bars + S::meta_full, *meta_free = bars + S::meta_free,
           *raw_full = bars + S::raw_full, *raw_free = bars + S::raw_free, *drain = bars + S::drain;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + S::tail);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  // the warp index by way of a shuffle: the compiler then knows that it is uniform across the warp, and keeps
  // the role branches and what they compute (addresses, descriptors, counters) on the uniform datapath
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  pf_dep_launch();
  if (tid == 0) {
    for (int s = 0; s < C::w_stages; ++s) {
      mbar_init(&w_full[s], 4);  // a set's four warps
      mbar_init(&w_free[s], 1);
    }
    for (int s = 0; s < C::tok_stages; ++s) {
      mbar_init(&tok_full[s], 1);
      mbar_init(&tok_free[s], 1);
    }
    for (int a = 0; a < C::accs; ++a) {
      mbar_init(&acc_full[a], 1);
      mbar_init(&acc_free[a], C::sum_warps);
    }
    for (int s = 0; s < kUItemSlots; ++s) {
      mbar_init(&item_full[s], 1);
      mbar_init(&item_free[s], C::sum_warps + 4 * C::sets + 3);
    }
    for (int s = 0; s < kUMetaStages; ++s) {
      mbar_init(&meta_full[s], 1);
      mbar_init(&meta_free[s], C::sum_warps + 4 * C::sets);
    }
    for (int s = 0; s < C::raw_stages; ++s) {
      mbar_init(&raw_full[s], 64);  // the lanes of the two warps that copy, one plane each
      mbar_init(&raw_free[s], 4);  // the four warps of the set that takes the step
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == C::warp_mma) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(kUTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  bool alive = true;
  // Only the token warp waits for the kernel before, whose work the token rows are (gathered x, or h).  That this kernel runs
  // says that the gather kernel's blocks have all seen the plan kernel's end: the plan, the counters and the caller's arrays
  // are there, and the weights' way through the CTA fills up meanwhile.  They are there in L2: what is read without the wait is
  // read past L1, where an SM may still hold a line of the call before (same workspace, same tables).

  if (warp >= C::warp_tok) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(C::regs_rest));
    if (warp == C::warp_tok) {
      // ---- token tiles: two TMA copies of the tile's rows x 64 columns; and the raw LSB planes ----
      uint32_t st = 0, par = 1;  // stage; parity of the use before (the first one waits for nothing)
      uint32_t rs = 0, rpar = 1;
      for (uint32_t ni = 0;; ++ni) {
        const PfItem& it = items[ni % kUItemSlots];
        if (!mbar_wait(&item_full[ni % kUItemSlots], (ni / kUItemSlots) & 1, abort_flag)) { alive = false; break; }
        if (it.stop) break;
        const int nk = it.nk, box = (it.n + kUBoxRows - 1) / kUBoxRows, row = it.in_row;
        const bool prec = it.prec != 0;
        const uint8_t *p0 = it.lsb[0] + lane * 16, *p1 = it.lsb[1] + lane * 16;
        // released at once, as by everybody: the next item's description must not depend on this one's progress (the
        // weight warps want it while they have steps of this one to deliver)
        __syncwarp();
        if (lane == 0) mbar_arrive(&item_free[ni % kUItemSlots]);
        auto copy_step = [&]() {
          if (!mbar_wait(&raw_free[rs], rpar, abort_flag)) return false;
          if (prec) {
            u_copy_raw<PHASE>(smem_u32(smem + S::raw + rs * kURawStep + 8 * kURawBlock + lane * 16), p0, p1, (uint32_t)nk * kURawBlock);
            p0 += kURawBlock;
            p1 += kURawBlock;
          }
          cp_async_arrive(&raw_full[rs]);
          if (++rs == C::raw_stages) { rs = 0; rpar ^= 1; }
          return true;
        };
        int copied = 0;
        if (ni == 0) {
          for (; copied < min(nk, C::raw_stages); ++copied)
            if (!copy_step()) break;
          pf_dep_wait();
        }
        for (int kc = 0; kc < nk; ++kc) {
          if (kc >= copied && !copy_step()) { alive = false; break; }
          if (!mbar_wait(&tok_free[st], par, abort_flag)) { alive = false; break; }
          if (elect_one()) {
            mbar_expect_tx(&tok_full[st], 2 * box * (kUBoxRows * kUBoxCols * 2));
#pragma unroll
            for (int panel = 0; panel < 2; ++panel)
              asm volatile(
                  "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(
                      smem_u32(smem + S::tok + st * C::tile_bytes + panel * C::panel_bytes)),
                  "l"(&maps.rows[box - 1]), "r"(smem_u32(&tok_full[st])), "r"(kc * kPfChunkK + panel * kUBoxCols), "r"(row)
                  : "memory");
          }
          __syncwarp();
          if (++st == C::tok_stages) { st = 0; par ^= 1; }
        }
        if (!alive) break;
      }
      pf_dep_wait();  // (without an item:) the kernel after this one counts on it
      asm volatile("cp.async.wait_all;" ::: "memory");
      // No copy may still be on its way into shared memory when the CTA ends: only after a time-out can one be, and then the
      // longest that a copy can take is waited out.
      if (!alive) {
        const uint32_t t0 = (uint32_t)clock64();
        while ((uint32_t)clock64() - t0 < kUCopyCycles) {}
      }
    } else if (warp == C::warp_mma) {
      // ---- MMA issue: D[weight row, token] += W[weight row, k] (tensor memory) x X[token, k] (shared memory) ----
      // The whole warp walks the loop, so that its state stays on the uniform datapath, where the tensor instructions take
      // their operands from; one elected lane issues.  (All of it in one lane: twice the time per step.)
      uint32_t st = 0, par = 0, ts = 0, tpar = 0;  // weight and token stage, parity of their use
      uint32_t buf = 0, bpar = 1;  // accumulator of the next group, parity of its use before
      bool issued = false;
      const uint64_t bd0 = umma_desc(smem_u32(smem + S::tok));
      constexpr int kGroups = 128 / G, kKs = G / 16;  // quantisation groups of a step, K 16 slices of a group
      for (uint32_t ni = 0; alive; ++ni) {
        const PfItem& it = items[ni % kUItemSlots];
        if (!mbar_wait(&item_full[ni % kUItemSlots], (ni / kUItemSlots) & 1, abort_flag)) { alive = false; break; }
        if (__shfl_sync(0xffffffffu, it.stop, 0)) break;
        const int nk = __shfl_sync(0xffffffffu, it.nk, 0);
        const uint32_t id = umma_idesc(__shfl_sync(0xffffffffu, it.n, 0));
        __syncwarp();
        if (elect_one()) mbar_arrive(&item_free[ni % kUItemSlots]);
        for (int kc = 0; kc < nk && alive; ++kc) {
          // The three that a step waits for are looked at together: their latencies overlap.
          {
            const bool t = mbar_test(&tok_full[ts], tpar), w = mbar_test(&w_full[st], par), a = mbar_test(&acc_free[buf], bpar);
            if (!__all_sync(0xffffffffu, t && w && a) &&
                !(mbar_wait(&tok_full[ts], tpar, abort_flag) && mbar_wait(&w_full[st], par, abort_flag) &&
                  mbar_wait(&acc_free[buf], bpar, abort_flag))) { alive = false; break; }
          }
          const uint64_t bd = bd0 + (uint64_t)((ts * C::tile_bytes) >> 4);
          const uint32_t a_step = tmem + C::w_col0 + st * kUWCols;
          const uint32_t st0 = st, ts0 = ts;
          if (++st == C::w_stages) { st = 0; par ^= 1; }
          if (++ts == C::tok_stages) { ts = 0; tpar ^= 1; }
#pragma unroll
          for (int grp = 0; grp < kGroups; ++grp) {
            if (grp > 0 && !mbar_wait(&acc_free[buf], bpar, abort_flag)) { alive = false; break; }
            tc_fence_after();
            const uint32_t d = tmem + buf * C::acc_cols;
            auto issue = [&](int ks) {
              const int k16 = grp * kKs + ks;  // within the step; four to a panel
              umma_f16_ts(d, a_step + 8 * k16, bd + (uint64_t)((k16 >> 2) * (C::panel_bytes >> 4) + 2 * (k16 & 3)), id, ks ? 1u : 0u);
            };
            if (elect_one()) {
#pragma unroll
              for (int ks = 0; ks < kKs; ++ks) issue(ks);
              if (grp == kGroups - 1) {
                umma_commit(&w_free[st0]);
                umma_commit(&tok_free[ts0]);
              }
              umma_commit(&acc_full[buf]);
            }
            issued = true;
            __syncwarp();
            if (++buf == C::accs) { buf = 0; bpar ^= 1; }
          }
        }
      }
      // the last commits must have arrived before shared and tensor memory go away
      if (issued) {
        if (elect_one()) umma_commit(drain);
        __syncwarp();
        const uint32_t t0 = (uint32_t)clock64();
        while (!mbar_try(drain, 0) && (uint32_t)clock64() - t0 < kUWaitCycles) {}
        __syncwarp();
      }
    } else if (warp == C::warp_sched) {
      // ---- scheduler: takes items from the counter and describes them ----
      int* next = PHASE == 1 ? &p.head->next1 : &p.head->next2;
      const int n_runs = __ldcg(&p.head->runs), n_items = __ldcg(PHASE == 1 ? &p.head->items1 : &p.head->items2);
      // How far ahead: one item where an item is long (its successor is fetched when the sums of the item itself have
      // begun, and no CTA sits on items that another could take) or a CTA has few, else as many as the ring holds.
      constexpr int kLongItem = 8, kAheadShort = 6;
      const int share = n_items / (int)gridDim.x, ahead_short = share < kAheadShort ? max(share, 1) : kAheadShort;
      static_assert(kAheadShort <= kUItemSlots, "items between the copies and their use");
      int ahead = ahead_short;
      for (uint32_t ni = 0;; ++ni) {
        if (ni >= (uint32_t)ahead) {
          const uint32_t j = ni - ahead;
          if (!mbar_wait(&item_free[j % kUItemSlots], (j / kUItemSlots) & 1, abort_flag)) { alive = false; break; }
        }
        int item = 0;
        if (lane == 0) item = atomicAdd(next, 1);
        item = __shfl_sync(0xffffffffu, item, 0);
        PfItem& it = items[ni % kUItemSlots];
        PfRun r{};
        bool prec = true;
        int in_run = 0;
        const slicemoe_expert* ex = nullptr;
        const void* ptr = nullptr;
        if (item < n_items) {
          const int run = u_find_run<PHASE>(p.runs, n_runs, item, lane);
          r = pf_load_run(p.runs + run);
          in_run = item - (PHASE == 1 ? r.items1 : r.items2);
          const bool is_shared = r.expert >= p.E;
          ex = is_shared ? p.shared + (r.expert - p.E) : p.experts + r.expert;
          prec = is_shared || __ldcg(p.expert_prec + r.expert) != 0;
          // lanes 0 .. 7: MSB, LSB, scales, zero-points of the first and of the second matrix
          const slicemoe_mat* m = PHASE == 1 ? ((lane & 1) ? &ex->up : &ex->gate) : &ex->down;
          const int what = (lane >> 1) & 3;
          static_assert(offsetof(slicemoe_mat, lsb) == 8 && offsetof(slicemoe_mat, scale) == 16 && offsetof(slicemoe_mat, zp) == 24, "in this order");
          ptr = reinterpret_cast<const void*>(__ldcg(reinterpret_cast<const unsigned long long*>(m) + what));
          const bool no_lsb = __any_sync(0xffffffffu, what == 1 && ptr == nullptr);
          if (prec && no_lsb) {  // both slices were asked for but the LSB planes are absent
            if (lane == 0) atomicOr(p.status, (unsigned)SLICEMOE_STATUS_MISSING_LSB);
            prec = false;
          }
        }
        if (item < n_items) {
          // items of a run: weight tile by weight tile, its token tiles next to one another (they share the weights)
          const int nt = in_run / r.tiles, tile = in_run - nt * r.tiles;
          const bool is_shared = r.expert >= p.E;
          const int K = PHASE == 1 ? p.hidden : (is_shared ? p.shared_inter : p.inter);
          ahead = K / kPfChunkK >= kLongItem ? 1 : ahead_short;
          const int width = ((r.count + r.tiles - 1) / r.tiles + 15) & ~15;  // the tiles are equally wide, the last may be shorter
          const int t0 = tile * width, count = max(0, min(width, r.count - t0)), n = (count + 15) & ~15;
          // the item's first row block: 4 of gate and of up per 64 columns of h, or 8 of down
          const size_t rb = (size_t)nt * (PHASE == 1 ? 4 : 8), blocks = rb * (K / 64), entries = rb * (K >> LG) * 16;
          const int what = (lane >> 1) & 3;
          if (lane < 8) {
            const uint8_t* b = reinterpret_cast<const uint8_t*>(ptr);
            if (what == 0) it.msb[lane & 1] = b + blocks * 512;
            else if (what == 1) it.lsb[lane & 1] = b ? b + blocks * 512 : b;
            else if (what == 2) it.scale[lane & 1] = reinterpret_cast<const uint16_t*>(b) + entries;
            else it.zp[lane & 1] = b + entries;
          }
          if (lane == 0) {
            it.nk = K / kPfChunkK;
            it.n = n;
            it.n0 = C::sum_wgs == 1 ? n : min(n, 32 * ((n + 63) / 64));  // the first warpgroup reads whole 32-column pieces
            it.count = count;
            it.in_row = (PHASE == 1 ? r.in_row : r.out_row) + t0;
            it.out_row = r.out_row + t0;
            it.col = nt * (PHASE == 1 ? 64 : 128);
            it.prec = prec ? 1 : 0;
            it.stop = 0;
          }
        } else if (lane == 0) {
          it.stop = 1;
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&item_full[ni % kUItemSlots]);
        if (item >= n_items) break;
      }
    } else {
      // ---- raw MSB planes (cp.async); scales and zero-points (bulk copies): a row block's are contiguous over the groups, so
      // for up to 16 groups at a time lanes 0 .. 7 copy a block's scales and lanes 8 .. 15 its zero-points.  (Planes by bulk
      // copies of a row block's 1024 bytes each: a warp issues those lane by lane, 60 cycles each.) ----
      uint32_t m = 0, rs = 0, rpar = 1;  // scale stages so far; raw stage, parity of its use before
      const int rbk = lane & 7, mat = PHASE == 1 ? rbk & 1 : 0, rb = PHASE == 1 ? rbk >> 1 : rbk;
      const bool second = lane >= 8;  // zero-points
      constexpr int kMetaSteps = kUMetaGroups * G / 128;  // steps of a scale and zero-point stage
      for (uint32_t ni = 0; alive; ++ni) {
        const PfItem& it = items[ni % kUItemSlots];
        if (!mbar_wait(&item_full[ni % kUItemSlots], (ni / kUItemSlots) & 1, abort_flag)) { alive = false; break; }
        if (it.stop) break;
        const int nk = it.nk, ngroups = (nk * kPfChunkK) >> LG;
        const uint8_t* src = (second ? it.zp[mat] : reinterpret_cast<const uint8_t*>(it.scale[mat])) + (size_t)rb * ngroups * (second ? 16 : 32);
        const uint8_t *p0 = it.msb[0] + lane * 16, *p1 = it.msb[1] + lane * 16;
        __syncwarp();
        if (lane == 0) mbar_arrive(&item_free[ni % kUItemSlots]);
        const bool aligned = __all_sync(0xffffffffu, lane >= 16 || (reinterpret_cast<uintptr_t>(src) & 15) == 0);
        for (int kc = 0; kc < nk; ++kc) {
          if (kc % kMetaSteps == 0) {
            const uint32_t ms = m % kUMetaStages;
            if (!mbar_wait(&meta_free[ms], ((m / kUMetaStages) & 1) ^ 1, abort_flag)) { alive = false; break; }
            const int g0 = (kc * kPfChunkK) >> LG, gs = min(kUMetaGroups, ngroups - g0), bytes = gs * (second ? 16 : 32);
            uint8_t* dst = smem + S::meta + ms * kUMetaBytes + (second ? 8 * kUMetaScale + rbk * kUMetaZp : rbk * kUMetaScale);
            const uint8_t* from = src + (size_t)g0 * (second ? 16 : 32);
            if (aligned) {
              if (lane == 0) mbar_expect_tx(&meta_full[ms], gs * 8 * 48);
              __syncwarp();
              if (lane < 16) bulk_copy(dst, from, bytes, &meta_full[ms]);
            } else {  // a caller's array that does not start on 16 bytes: byte by byte (weights: no call before has them otherwise)
              if (lane < 16)
                for (int i = 0; i < bytes; ++i) dst[i] = from[i];
              __syncwarp();
              if (lane == 0) mbar_arrive(&meta_full[ms]);
            }
            ++m;
          }
          if (!mbar_wait(&raw_free[rs], rpar, abort_flag)) { alive = false; break; }
          u_copy_raw<PHASE>(smem_u32(smem + S::raw + rs * kURawStep + lane * 16), p0, p1, (uint32_t)nk * kURawBlock);
          p0 += kURawBlock;
          p1 += kURawBlock;
          cp_async_arrive(&raw_full[rs]);
          if (++rs == C::raw_stages) { rs = 0; rpar ^= 1; }
        }
      }
      asm volatile("cp.async.wait_all;" ::: "memory");
      for (uint32_t i = m > kUMetaStages ? m - kUMetaStages : 0; i < m && !alive; ++i) {  // no copy on its way when the CTA ends
        const uint32_t t0 = (uint32_t)clock64();
        while (!mbar_try(&meta_full[i % kUMetaStages], (i / kUMetaStages) & 1) && (uint32_t)clock64() - t0 < kUWaitCycles) {}
      }
    }
  } else if (warp >= C::sum_warps) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(C::regs_weight));
    // ---- weights: sets of four warps take the steps in turn; warp q of a set owns tensor-memory lanes
    // [32 q, 32 q + 32), two row blocks, and stores their integers of the step into the stage's columns.  The planes are laid
    // out as the fragments of a 16-row store: plane lane 4 g + c holds rows g and g + 8, columns 16 w + 4 c + j, which
    // is what lane 4 g + c of tcgen05.st.16x256b gives.  So a lane reads 16 bytes of a plane block, converts and stores
    // them: both nibbles of every byte are used, and nothing is exchanged. ----
    const int q = warp & 3, set = (warp - C::sum_warps) >> 2;
    const int g = lane >> 2;
    const uint8_t* raw = smem + S::raw + 2 * q * kURawBlock + lane * 16;
    const int shift = p.shift;
    // row g's codes: MSB nibble at bit `shift`, LSB nibble below; row g + 8's the same from the high nibbles.  A slice
    // narrower than four bits leaves the top of its nibble zero, so what the second mask lets through beyond it is zero.
    const uint32_t mask = 0x0f0f0f0fu << shift;
    const int back = 4 - shift;
    // (Steps are counted over all items; every C::sets-th is the set's own.)
    int skip = set;
    uint32_t st = set, par = 1, m = 0;  // stage of the next own step, parity of its use before; scale and zero-point
                                                    // stages; steps of the item before the first own one
    uint32_t rs = set, rpar = 0;                    // raw stage of the next own step, parity of this use
    static_assert(C::sets <= C::w_stages && C::raw_stages % C::sets == 0, "a set's next stage is at most once round the rings away");
    for (uint32_t ni = 0; alive; ++ni) {
      const PfItem& it = items[ni % kUItemSlots];
      if (!mbar_wait(&item_full[ni % kUItemSlots], (ni / kUItemSlots) & 1, abort_flag)) { alive = false; break; }
      if (it.stop) break;
      const int nk = it.nk;
      const bool prec = it.prec != 0;
      const uint32_t zmask = prec ? 0xffu : 0xffu << shift;  // from the MSB slice alone: 2^shift (zp >> shift)
      __syncwarp();
      if (lane == 0) mbar_arrive(&item_free[ni % kUItemSlots]);
      int kc = skip;
      constexpr int kMetaSteps = kUMetaGroups * G / 128;  // steps of a scale and zero-point stage
      for (int k0 = 0; k0 < nk && alive; k0 += kMetaSteps, ++m) {
        const uint32_t ms = m % kUMetaStages;
        if (!mbar_wait(&meta_full[ms], (m / kUMetaStages) & 1, abort_flag)) { alive = false; break; }
        const uint8_t* zp_stage = smem + S::meta + ms * kUMetaBytes + 8 * kUMetaScale + 2 * q * kUMetaZp + g;
        const int k_end = min(nk, k0 + kMetaSteps);
        for (; kc < k_end; kc += C::sets) {
          const uint8_t* zp = zp_stage + (kc - k0) * (128 / G * 16);
          if (!mbar_wait(&raw_full[rs], rpar, abort_flag)) { alive = false; break; }
          const uint8_t* slot = raw + rs * kURawStep;
          uint4 mv[4], lv[4];  // [2 block + half]
#pragma unroll
          for (int i = 0; i < 4; ++i) mv[i] = *reinterpret_cast<const uint4*>(slot + 512 * i);
#pragma unroll
          for (int i = 0; i < 4; ++i) lv[i] = prec ? *reinterpret_cast<const uint4*>(slot + 8 * kURawBlock + 512 * i) : make_uint4(0, 0, 0, 0);
          if (!mbar_wait(&w_free[st], par, abort_flag)) { alive = false; break; }
          tc_fence_after();
          // the words are in registers: the raw stage is handed back before the conversion, not after
          __syncwarp();
          if (lane == 0) mbar_arrive(&raw_free[rs]);
          rs += C::sets;
          if (rs >= C::raw_stages) {
            rs -= C::raw_stages;
            rpar ^= 1;
          }
          const uint32_t ta = tmem + ((uint32_t)(32 * q) << 16) + C::w_col0 + st * kUWCols;
#pragma unroll
          for (int b = 0; b < 2; ++b) {
            __half2 off[128 / G][2];  // 1024 + zero-point, rows g and g + 8, twice
#pragma unroll
            for (int i = 0; i < 128 / G; ++i)
#pragma unroll
              for (int hi = 0; hi < 2; ++hi) {
                uint32_t z = zp[b * kUMetaZp + 16 * i + 8 * hi];
                z = (z & zmask) * 0x00010001u + 0x64006400u;
                off[i][hi] = *reinterpret_cast<__half2*>(&z);
              }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const uint32_t mw[4] = {mv[2 * b + h].x, mv[2 * b + h].y, mv[2 * b + h].z, mv[2 * b + h].w},
                             lw[4] = {lv[2 * b + h].x, lv[2 * b + h].y, lv[2 * b + h].z, lv[2 * b + h].w};
              uint32_t out[16];
#pragma unroll
              for (int w = 0; w < 4; ++w) {
                // four codes a row, one per byte
                const uint32_t code[2] = {((mw[w] << shift) & mask) | (lw[w] & ~mask), ((mw[w] >> back) & mask) | ((lw[w] >> 4) & ~mask)};
#pragma unroll
                for (int hi = 0; hi < 2; ++hi) {
                  // bytes -> fp16 1024 + code, minus (1024 + zero-point): exact integers
                  uint32_t h01 = __byte_perm(code[hi], 0x64646464u, 0x4140), h23 = __byte_perm(code[hi], 0x64646464u, 0x4342);
                  const __half2 o = off[(h * 64 + w * 16) / G][hi];
                  const __half2 d01 = __hsub2(*reinterpret_cast<__half2*>(&h01), o), d23 = __hsub2(*reinterpret_cast<__half2*>(&h23), o);
                  out[4 * w + 2 * hi] = *reinterpret_cast<const uint32_t*>(&d01);
                  out[4 * w + 2 * hi + 1] = *reinterpret_cast<const uint32_t*>(&d23);
                }
              }
              tmem_st_16x32(ta + ((uint32_t)(16 * b) << 16) + 32 * h, out);
            }
          }
          tmem_st_wait();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&w_full[st]);
          st += C::sets;
          if (st >= C::w_stages) {
            st -= C::w_stages;
            par ^= 1;
          }
        }
        if (alive && lane == 0) mbar_arrive(&meta_free[ms]);
      }
      skip = kc - nk;
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(C::regs_sum));
    // ---- sums: warp (q, wg) owns weight rows [32 q, 32 q + 32) x the warpgroup's tokens, in fp32 registers ----
    const int q = warp & 3, wg = warp >> 2;
    uint32_t buf = 0, bpar = 0;  // accumulator of the next unit (a group's sums for the tile or half of it), parity of its use
    uint32_t m = 0;     // scale stages so far
    for (uint32_t ni = 0; alive; ++ni) {
      const PfItem& it = items[ni % kUItemSlots];
      if (!mbar_wait(&item_full[ni % kUItemSlots], (ni / kUItemSlots) & 1, abort_flag)) { alive = false; break; }
      if (it.stop) break;
      const int n0 = it.n0;
      const int cols = wg == 0 ? n0 : it.n - n0;  // tokens of this warpgroup
      const int ngroups = (it.nk * kPfChunkK) >> LG;
      // (The first item's successor is fetched when its sums have begun, too: the CTAs do not all start at once.)
      if (ni == 0 && !mbar_wait(&acc_full[0], 0, abort_flag)) { alive = false; break; }
      const int count = wg == 0 ? min(it.count, n0) : it.count - n0, out_row = it.out_row + (wg == 0 ? 0 : n0), col = it.col;
      __syncwarp();
      if (lane == 0) mbar_arrive(&item_free[ni % kUItemSlots]);
      const uint32_t lane_base = tmem + ((uint32_t)(32 * q) << 16) + (wg ? n0 : 0);
      auto next_unit = [&]() {
        if (++buf == C::accs) { buf = 0; bpar ^= 1; }
      };
      uint64_t acc[C::half_max / 2];
#pragma unroll
      for (int i = 0; i < C::half_max / 2; ++i) acc[i] = 0ull;
      for (int g0 = 0; g0 < ngroups && alive; g0 += kUMetaGroups, ++m) {
        const uint32_t ms = m % kUMetaStages;
        if (!mbar_wait(&meta_full[ms], (m / kUMetaStages) & 1, abort_flag)) { alive = false; break; }
        const uint8_t* sc = smem + S::meta + ms * kUMetaBytes + (2 * q + (lane >> 4)) * kUMetaScale + (lane & 15) * 2;
        for (int gi = min(kUMetaGroups, ngroups - g0); gi > 0; --gi, sc += 32) {
          const float s = __half2float(*reinterpret_cast<const __half*>(sc));
          const uint64_t ss = ((uint64_t)__float_as_uint(s) << 32) | __float_as_uint(s);
          if (!mbar_wait(&acc_full[buf], bpar, abort_flag)) { alive = false; break; }
          tc_fence_after();
#pragma unroll
          for (int c = 0; c < C::half_max / 32; ++c) {
            if (32 * c < cols) {
              uint32_t v[32];
              tmem_ld32(lane_base + buf * C::acc_cols + 32 * c, v);
#pragma unroll
              for (int i = 0; i < 16; ++i) fma2(acc[16 * c + i], v[2 * i], v[2 * i + 1], ss);
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&acc_free[buf]);
          next_unit();
        }
        __syncwarp();
        if (alive && lane == 0) mbar_arrive(&meta_free[ms]);
      }
      if (!alive) break;
      if (PHASE == 1) {
        // lanes 0 .. 15 hold gate rows, lanes 16 .. 31 the up rows of the same 16 columns of h.  Of two tokens the gate lane
        // finishes the first and the up lane the second: one exchange each.
        const bool up = lane >= 16;
        __half* dst = p.h + (size_t)(out_row + (up ? 1 : 0)) * p.ldh + col + 16 * q + (lane & 15);
        const size_t two_rows = 2 * (size_t)p.ldh;
        // 16 tokens at a time, with a branch per 16: within them the chains of shuffle, exponential and reciprocal overlap
#pragma unroll
        for (int i0 = 0; i0 < C::half_max / 2; i0 += 8) {
          if (2 * i0 < count) {
#pragma unroll
            for (int i = i0; i < i0 + 8; ++i) {
              const float v0 = half_of(acc[i], 0), v1 = half_of(acc[i], 1);
              const float got = __shfl_xor_sync(0xffffffffu, up ? v0 : v1, 16);
              const float gate = up ? got : v0, upv = up ? v1 : got;
              // silu: g / (1 + e^-g), by the approximate reciprocal: its error, 2^-23, is 2^-12 of the rounding to fp16 that
              // follows.  Below -80 the result is zero in fp16 either way; the bound keeps 1 + e^-g finite.
              const float t = 1.f + __expf(fminf(-gate, 80.f));
              float r;
              asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(t));
              if (2 * i + (up ? 1 : 0) < count) *dst = __float2half_rn(gate * r * upv);
              dst += two_rows;
            }
          }
        }
      } else {
        float* dst = p.yrow + (size_t)out_row * p.hidden + col + 32 * q + lane;
#pragma unroll
        for (int i0 = 0; i0 < C::half_max / 2; i0 += 8) {
          if (2 * i0 < count) {
#pragma unroll
            for (int i = 2 * i0; i < 2 * i0 + 16; ++i) {
              if (i < count) *dst = half_of(acc[i >> 1], i & 1);
              dst += p.hidden;
            }
          }
        }
      }
    }
  }
  if (!alive) {
    *abort_flag = 1;
    if (lane == 0) atomicOr(p.status, (unsigned)SLICEMOE_STATUS_WAIT_TIMEOUT);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == C::warp_mma) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kUTmemCols) : "memory");
  }
}

// ---- step 5: weighted combine in list order ---------------------------------------------------------------
// A block per token: the token's rows and weights are read once into shared memory, then four slots' rows at a time are in
// flight.
__global__ void __launch_bounds__(256) pf_combine_kernel(const float* __restrict__ yrow, const int* __restrict__ posmap,
                                                         const float* __restrict__ weights, const float* __restrict__ gate, int k,
                                                         int n_shared, int hidden, float* __restrict__ y) {
  __shared__ int s_pos[kPfMaxSlots];
  __shared__ float s_w[kPfMaxSlots];
  const int t = blockIdx.x;
  const int slots = k + n_shared;
  pf_dep_launch();
  pf_dep_wait();
  if (threadIdx.x < slots) {
    const int j = threadIdx.x, pos = posmap[t * slots + j];
    const float w = j < k ? weights[t * k + j] : (gate ? gate[t] : 1.f);
    s_pos[j] = pos;
    s_w[j] = w;
  }
  __syncthreads();
  for (int col = threadIdx.x * 4; col < hidden; col += blockDim.x * 4) {
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int j0 = 0; j0 < slots; j0 += 4) {
      float4 v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (j0 + j < slots && s_pos[j0 + j] >= 0)
          v[j] = __ldcs(reinterpret_cast<const float4*>(yrow + (size_t)s_pos[j0 + j] * hidden + col));
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (j0 + j >= slots || s_pos[j0 + j] < 0) continue;
        const float w = s_w[j0 + j];
        a.x = fmaf(w, v[j].x, a.x);
        a.y = fmaf(w, v[j].y, a.y);
        a.z = fmaf(w, v[j].z, a.z);
        a.w = fmaf(w, v[j].w, a.w);
      }
    }
    *reinterpret_cast<float4*>(y + (size_t)t * hidden + col) = a;
  }
}

typedef CUresult (*PfEncodeTiled)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// Tensor maps of a row-major fp16 matrix [rows, cols] for tiles of 32, 64, ... rows x 64 columns with 128-byte swizzle.
static int pf_tensor_maps(PfMaps* maps, const __half* base, int rows, int cols) {
  static PfEncodeTiled encode = nullptr;
  if (!encode) {
    cudaDriverEntryPointQueryResult q;
    void* fn = nullptr;
    SM_CUDA_TRY(cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &q));
    if (!fn || q != cudaDriverEntryPointSuccess) return SLICEMOE_E_UNSUPPORTED;
    encode = reinterpret_cast<PfEncodeTiled>(fn);
  }
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)cols * sizeof(__half)};
  const cuuint32_t estr[2] = {1, 1};
  for (int i = 0; i < kUBoxes; ++i) {
    const cuuint32_t box[2] = {(cuuint32_t)kUBoxCols, (cuuint32_t)(kUBoxRows * (i + 1))};
    const CUresult r = encode(&maps->rows[i], CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<__half*>(base), dims, strides, box,
                              estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return SLICEMOE_E_INVALID_ARG;
  }
  return SLICEMOE_OK;
}

// Every kernel of a step starts while the one before it is still running and waits for it itself (pf_dep_wait), only where it
// needs that kernel's work: the gather kernel reads x and the GEMM kernels their weights before.  77 tokens through 64 + 2
// experts of 2048 x 1408: 135.5 us with every kernel waiting at its start, 129 so; 16 tokens 98 -> 92.
template <class... Args>
static int pf_launch(void (*kernel)(Args...), unsigned blocks, unsigned threads, size_t smem, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  SM_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, args...));
  return SLICEMOE_OK;
}

template <int G, int TN>
static int pf_launch_gemms(const PfGemmParams& p, const __half* xs, int in_rows, int out_rows, cudaStream_t st) {
  static bool attr_set[64];
  static int sm_count[64];
  int dev = 0;
  SM_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return SLICEMOE_E_UNSUPPORTED;
  if (!attr_set[dev]) {
    SM_CUDA_TRY(cudaFuncSetAttribute(pf_umma_kernel<G, 1, TN>, cudaFuncAttributeMaxDynamicSharedMemorySize, kUSmemBytes<TN>));
    SM_CUDA_TRY(cudaFuncSetAttribute(pf_umma_kernel<G, 2, TN>, cudaFuncAttributeMaxDynamicSharedMemorySize, kUSmemBytes<TN>));
    SM_CUDA_TRY(cudaDeviceGetAttribute(&sm_count[dev], cudaDevAttrMultiProcessorCount, dev));
    attr_set[dev] = true;
  }
  PfMaps tm_x, tm_h;
  int rc = pf_tensor_maps(&tm_x, xs, in_rows, p.hidden);
  if (rc != SLICEMOE_OK) return rc;
  rc = pf_tensor_maps(&tm_h, p.h, out_rows, p.ldh);
  if (rc != SLICEMOE_OK) return rc;
  // one persistent CTA per SM (shared memory admits one); each takes work items until there are none
  rc = pf_launch(pf_umma_kernel<G, 1, TN>, (unsigned)sm_count[dev], UCfg<TN>::threads, kUSmemBytes<TN>, st, p, tm_x);
  if (rc != SLICEMOE_OK) return rc;
  return pf_launch(pf_umma_kernel<G, 2, TN>, (unsigned)sm_count[dev], UCfg<TN>::threads, kUSmemBytes<TN>, st, p, tm_h);
}

template <int TN>
static int pf_launch_gemms(int group, const PfGemmParams& p, const __half* xs, int in_rows, int out_rows, cudaStream_t st) {
  if (group == 128) return pf_launch_gemms<128, TN>(p, xs, in_rows, out_rows, st);
  if (group == 64) return pf_launch_gemms<64, TN>(p, xs, in_rows, out_rows, st);
  return pf_launch_gemms<32, TN>(p, xs, in_rows, out_rows, st);
}

// Which form: narrow tiles where none is cut by them, or hardly any: up to 36 rows per expert on average.  (Where the two meet
// depends on how uneven the routing is and on the shared experts' part: 30 rows for 60 experts and a shared one four
// times as wide, 50 for 64 + 2, 64 and more for others; at 36 the narrow one is 3 to 13 % ahead or level.)
static int pf_tile(const slicemoe_shape* s, int T) {
  return T <= kPfNarrowN || (long long)T * (s->top_k + s->n_shared) <= 36ll * (s->n_experts + s->n_shared) ? kPfNarrowN : kPfTileN;
}

static int pf_check(const slicemoe_shape* s, int T) {
  if (!s || T <= 0) return SLICEMOE_E_INVALID_ARG;
  if (!valid_widths(s->b_high, s->b_low)) return SLICEMOE_E_UNSUPPORTED;
  if (!valid_group(s->group)) return SLICEMOE_E_UNSUPPORTED;
  if (s->hidden <= 0 || s->inter <= 0 || s->n_experts <= 0 || s->top_k < 1) return SLICEMOE_E_INVALID_ARG;
  if (s->top_k > s->n_experts || s->top_k > SLICEMOE_MAX_TOP_K) return SLICEMOE_E_INVALID_ARG;
  if (s->n_shared < 0 || s->n_shared > SLICEMOE_MAX_SHARED) return SLICEMOE_E_INVALID_ARG;
  if ((s->hidden % 128) || (s->inter % 128)) return SLICEMOE_E_INVALID_ARG;
  if (s->n_shared > 0 && (s->shared_inter <= 0 || (s->shared_inter % 128))) return SLICEMOE_E_INVALID_ARG;
  if ((long long)T * (s->top_k + s->n_shared) > (1ll << 28)) return SLICEMOE_E_UNSUPPORTED;
  return SLICEMOE_OK;
}

}  // namespace slicemoe

using namespace slicemoe;

extern "C" size_t slicemoe_prefill_workspace_bytes(const slicemoe_shape* s, int T) {
  if (pf_check(s, T) != SLICEMOE_OK) return 0;
  return pf_layout(T, s->n_experts, s->top_k, s->n_shared, s->hidden, s->inter, s->n_shared ? s->shared_inter : 0).total;
}

extern "C" int slicemoe_prefill_layer(const slicemoe_shape* s, const slicemoe_expert* experts,
                                      const slicemoe_expert* shared, const float* shared_gate_vec, const void* x, int T,
                                      const int32_t* ids, const float* weights, const uint8_t* expert_prec, float* y,
                                      void* workspace, size_t workspace_bytes, int* status_out_device, void* stream) {
  int rc = pf_check(s, T);
  if (rc != SLICEMOE_OK) return rc;
  if (!experts || !x || !ids || !weights || !expert_prec || !y || !workspace || !status_out_device)
    return SLICEMOE_E_INVALID_ARG;
  if (s->n_shared > 0 && !shared) return SLICEMOE_E_INVALID_ARG;
  if (s->n_shared > 0 && s->shared_sigmoid_gate && !shared_gate_vec) return SLICEMOE_E_INVALID_ARG;
  const int nsh = s->n_shared, E = s->n_experts, k = s->top_k;
  const int shared_inter = nsh ? s->shared_inter : 0;
  const PfLayout L = pf_layout(T, E, k, nsh, s->hidden, s->inter, shared_inter);
  if (workspace_bytes < L.total || (reinterpret_cast<uintptr_t>(workspace) & 255)) return SLICEMOE_E_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(x) & 3) || (reinterpret_cast<uintptr_t>(y) & 15)) return SLICEMOE_E_INVALID_ARG;
  if (s->n_shared > 0 && s->shared_sigmoid_gate && (reinterpret_cast<uintptr_t>(shared_gate_vec) & 7))
    return SLICEMOE_E_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  uint8_t* ws = reinterpret_cast<uint8_t*>(workspace);
  const bool gated = nsh > 0 && s->shared_sigmoid_gate;
  __half* xs = reinterpret_cast<__half*>(ws + L.xs);
  float* gate = reinterpret_cast<float*>(ws + L.gate);
  float* yrow = reinterpret_cast<float*>(ws + L.yrow);

  PfPlanParams pp;
  pp.ids = ids;
  pp.T = T;
  pp.k = k;
  pp.E = E;
  pp.n_shared = nsh;
  pp.per1_routed = s->inter / 64;
  pp.per1_shared = shared_inter / 64;
  pp.per2 = s->hidden / 128;
  pp.head = reinterpret_cast<PfHead*>(ws + L.head);
  pp.counts = reinterpret_cast<int*>(ws + L.counts);
  pp.base = reinterpret_cast<int*>(ws + L.base);
  pp.hist = reinterpret_cast<int*>(ws + L.hist);
  pp.runs = reinterpret_cast<PfRun*>(ws + L.runs);
  pp.rank = reinterpret_cast<int*>(ws + L.rank);
  pp.rank_blocks = L.rank_blocks;
  pp.tile = pf_tile(s, T);
  pp.status = reinterpret_cast<unsigned*>(status_out_device);
  int* posmap = reinterpret_cast<int*>(ws + L.posmap);
  if (L.rank_blocks > 1) {
    rc = pf_launch(pf_rank_kernel, (unsigned)L.rank_blocks, (unsigned)kPfPlanThreads, 0, st, (PfPlanParams)pp);
    if (rc != SLICEMOE_OK) return rc;
  }
  rc = pf_launch(pf_plan_kernel, 1u, (unsigned)kPfPlanThreads, 0, st, (PfPlanParams)pp);
  if (rc != SLICEMOE_OK) return rc;
  PfGatherParams pg;
  pg.x = reinterpret_cast<const uint16_t*>(x);
  pg.ids = ids;
  pg.rank = pp.rank;
  pg.first = pp.hist;
  pg.T = T;
  pg.k = k;
  pg.E = E;
  pg.n_shared = nsh;
  pg.hidden = s->hidden;
  pg.posmap = posmap;
  pg.xs = xs;
  pg.gate_vec = gated ? shared_gate_vec : nullptr;
  pg.gate = gate;
  pg.status = pp.status;
  rc = pf_launch((reinterpret_cast<uintptr_t>(x) & 15) ? pf_gather_kernel<1> : pf_gather_kernel<4>, (unsigned)T, (unsigned)kPfGatherThreads, 0, st,
                 (PfGatherParams)pg);
  if (rc != SLICEMOE_OK) return rc;
  PfGemmParams p;
  p.experts = experts;
  p.shared = shared;
  p.expert_prec = expert_prec;
  p.runs = pp.runs;
  p.head = pp.head;
  p.h = reinterpret_cast<__half*>(ws + L.h);
  p.yrow = yrow;
  p.status = pp.status;
  p.E = E;
  p.hidden = s->hidden;
  p.inter = s->inter;
  p.shared_inter = shared_inter;
  p.ldh = s->inter > shared_inter ? s->inter : shared_inter;
  p.shift = s->b_high - s->b_low;
  rc = pp.tile == kPfNarrowN ? pf_launch_gemms<kPfNarrowN>(s->group, p, xs, L.in_rows, L.out_rows, st)
                             : pf_launch_gemms<kPfTileN>(s->group, p, xs, L.in_rows, L.out_rows, st);
  if (rc != SLICEMOE_OK) return rc;
  return pf_launch(pf_combine_kernel, (unsigned)T, 256u, 0, st, (const float*)yrow, (const int*)posmap, weights,
                   gated ? (const float*)gate : (const float*)nullptr, (int)k, (int)nsh, (int)s->hidden, y);
}
