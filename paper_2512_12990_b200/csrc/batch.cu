// Decode of a small batch of tokens of one MoE layer from bit-sliced AMAT weights: every expert that any of the tokens
// names is streamed from memory once and applied to all of its tokens.  (Token after token, the batch-1 kernel streams an
// expert once for each of them: eight tokens of a layer of 64 experts, top-6, with two shared ones read 463 MB, this
// 200.)
//
// Four launches, chained by programmatic dependent launch:
//   plan     groups the (token, slot) pairs into runs - up to eight pairs of one expert - and lists, for either
//            projection, the runs' row blocks with their cost, so that every CTA finds its share in closed form;
//   gate/up  h = silu(gate x) * (up x) of every pair, fp32;
//   down     result row of every pair, fp32;
//   combine  y[t] = sum of the token's rows times their weights, slots in list order, then the shared experts.
// The two projections are one kernel.  A CTA (one per SM) takes an equal share, by measured cost, of the row blocks of all runs.
// Four groups of a producer warp and four consumer warps each take the share's row blocks in turn: the producer
// streams the planes, scales and zero-points through the group's own ring with bulk copies, never waiting for anything but
// space; the consumers split a row block's 128-column blocks.  The arithmetic is the batch-1 kernel's: activations
// as 23-bit fixed point per 128-element block in three base-256 digits (int8), integer MMAs on the codes or nibbles,
// scale and zero-point once per group.  With column n of the MMA's B operand for token n and one MMA per digit, a lane ends
// up with all digits of its two tokens, so the digits are put together in its registers and a row block's result is two
// values per lane, row half and matrix; up to two tokens take one MMA for all their digits.  A pair at MSB precision shares
// the run with pairs at both slices: its columns leave out the LSB sums and the zero-point's low bits.
//
// Bound: HBM.  Per 16 x 128 block of both planes (2 KB, 89 cycles of an SM's share of the bandwidth) a warp issues about 125
// instructions, 24 of them MMAs (53 cycles of the integer tensor pipe).
// Measured, 8 tokens, 64 x 1408 top-6 + 2 shared, hidden 2048: eight batch-1 launches 133 us, this 53.6 (where the
// tokens' experts overlap as by Zipf(1.1) popularity: 195 MB, 30 us at the copy bandwidth).
//
// Bounded waits: when one runs out the CTA's dead flag goes up and SLICEMOE_STATUS_WAIT_TIMEOUT is set; from then on nobody
// waits for data, the consumers walk through the rest of their work and the producers - their four lanes together, so that
// every copy that one of them asks for is one that its barrier counts - stop and wait for the copies on their way, for a
// millisecond at least whatever the limit.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <type_traits>

#include "batch.cuh"
#include "common.cuh"
#include "decode_common.cuh"

namespace slicemoe {

constexpr int kBGroups = 4, kBGroupWarps = 4, kBConsumers = kBGroups * kBGroupWarps;
constexpr int kBThreads = 32 * (kBConsumers + kBGroups);
constexpr int kBPlane = 8192;            // plane bytes of a stage: 4 blocks of both slices or 8 of the MSB slice
constexpr int kBPlanThreads = 256;
static_assert(kBatchTokens * SLICEMOE_MAX_TOP_K <= kBPlanThreads, "a thread per pair");
static_assert(kBMaxTasks <= kBThreads, "a thread per segment");

// The row blocks of a run - up to eight pairs of one expert - in one projection (down: for one chunk of columns).
struct __align__(16) BSeg {
  unsigned start, ucost;     // cost of the segments before, cost of a row block
  int units;                 // row blocks
  int n;                     // pairs
  const uint8_t* ptr[2][4];  // [gate, up / down][MSB, LSB, scales, zero-points]
  unsigned high;             // bit per pair: both slices
  int lsb;                   // some pair uses both slices
  int inter, hoff;           // the run's h: [n][inter] from hoff on
  int yrow;                  // down: first result row
  int kb0, nkb, row_kb;      // first 128-column block, their number, blocks of a whole row
  uint8_t tok[kBRun];
  int pad_[2];
};
static_assert(sizeof(BSeg) == 128, "a lane per word copies a segment");
struct BHead {
  int nseg[2];               // negative: see `off`
  unsigned total[2];
  int off;                   // the time-out exercise: no weights are brought, y is not written
};

struct BLayout {
  size_t head, seg1, seg2, pos, gate, xdig, xsum, xinv, h, yrow, total;
  int kc_r, kc_s;
};
static inline BLayout batch_layout(const slicemoe_shape* s, int n_shared) {
  BLayout L;
  const int T = kBatchTokens, k = s->top_k, parts = (T + kBRun - 1) / kBRun;
  const int sint = n_shared ? s->shared_inter : 0;
  L.kc_r = (s->inter + kBChunkK - 1) / kBChunkK;
  L.kc_s = (sint + kBChunkK - 1) / kBChunkK;
  auto align = [](size_t v) { return (v + 255) & ~(size_t)255; };
  size_t o = 0;
  L.head = o; o = align(o + sizeof(BHead));
  L.seg1 = o; o = align(o + sizeof(BSeg) * (size_t)(T * k + n_shared * parts));
  L.seg2 = o; o = align(o + sizeof(BSeg) * (size_t)(T * k * L.kc_r + n_shared * parts * L.kc_s));
  L.pos = o;  o = align(o + sizeof(int2) * T * (k + n_shared));
  L.gate = o; o = align(o + sizeof(float) * T);
  L.xdig = o; o = align(o + (size_t)T * 3 * s->hidden);
  L.xsum = o; o = align(o + sizeof(float) * (size_t)T * 2 * (s->hidden / s->group));
  L.xinv = o; o = align(o + sizeof(float) * (size_t)T * (s->hidden / 128));
  L.h = o;    o = align(o + sizeof(float) * (size_t)T * ((size_t)k * s->inter + (size_t)n_shared * sint));
  L.yrow = o; o = align(o + sizeof(float) * (size_t)T * ((size_t)k * L.kc_r + (size_t)n_shared * L.kc_s) * s->hidden);
  L.total = o;
  return L;
}
size_t batch_workspace_bytes(const slicemoe_shape* s, int n_shared) { return batch_layout(s, n_shared).total; }

__device__ __forceinline__ void b_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void b_dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ---- plan ------------------------------------------------------------------------------------------------
struct BPlanParams {
  const int32_t* ids;
  const uint8_t* prec;
  const uint16_t* x;
  const float* gate_vec;  // or null
  int T, k, n_experts, n_shared, hidden, inter, shared_inter, kc_r, kc_s;
  const slicemoe_expert* experts;
  const slicemoe_expert* shared;
  BHead* head;
  BSeg *seg1, *seg2;
  int2* pos;
  float* gate;
  uint8_t* xdig;          // digits of x: [T][3 hidden]
  float *xsum, *xinv;     // their group sums [T][hidden / G][2], block scales [T][hidden / 128]
  BatchControl ctl;
};
__device__ __forceinline__ int b_chunk_cols(int inter, int kc) { return min(kBChunkK, inter - kc * kBChunkK); }
// Block-wide exclusive scans of four values, in place; `total` gets the sums.
__device__ void b_scan(unsigned (&v)[4], unsigned (*sums)[kBPlanThreads / 32], unsigned (&total)[4]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned inc[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) inc[i] = v[i];
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const unsigned a = __shfl_up_sync(0xffffffffu, inc[i], off);
      if (lane >= off) inc[i] += a;
    }
  }
  if (lane == 31) {
#pragma unroll
    for (int i = 0; i < 4; ++i) sums[i][warp] = inc[i];
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const unsigned w = lane < kBPlanThreads / 32 ? sums[i][lane] : 0u;
    total[i] = __reduce_add_sync(0xffffffffu, w);
    v[i] = __reduce_add_sync(0xffffffffu, lane < warp ? w : 0u) + inc[i] - v[i];
  }
}
// Block 0 plans; block 1 + t turns token t's x into digits and, with gated shared experts, works out its gate.
template <int G>
__global__ void __launch_bounds__(kBPlanThreads) batch_plan_kernel(const BPlanParams p) {
  __shared__ int s_e[kBPlanThreads];
  __shared__ unsigned s_high[kBPlanThreads], s_index[kBPlanThreads], s_prefix[kBPlanThreads], s_sums[4][kBPlanThreads / 32];
  __shared__ uint8_t s_tok[kBPlanThreads][kBRun];
  const int tid = threadIdx.x, lane = tid & 31;
  b_dep_launch();
  b_dep_wait();
  if (blockIdx.x > 0) {
    const int t = blockIdx.x - 1, nkb = p.hidden >> 7;
    const uint16_t* x = p.x + (size_t)t * p.hidden;
    float dot = 0.f;
    for (int b = tid >> 5; b < nkb; b += kBPlanThreads / 32) {
      const uint2 raw = *reinterpret_cast<const uint2*>(x + b * 128 + 4 * lane);
      const float v[4] = {__uint_as_float(raw.x << 16), __uint_as_float(raw.x & 0xffff0000u), __uint_as_float(raw.y << 16),
                          __uint_as_float(raw.y & 0xffff0000u)};
      if (p.gate_vec) {
#pragma unroll
        for (int j = 0; j < 4; ++j) dot = fmaf(p.gate_vec[b * 128 + 4 * lane + j], v[j], dot);
      }
      const BlockDigits d = block_digits(v);
      store_digits(d, b * 128 + 4 * lane, p.xdig + (size_t)t * 3 * p.hidden);
      int s0, s1, s2;
      group_digit_sums<G>(d, lane, s0, s1, s2);
      if ((lane & (G / 4 - 1)) == 0) {
        float* sum = p.xsum + ((size_t)t * (p.hidden / G) + b * (128 / G) + lane / (G / 4)) * 2;
        sum[0] = fmaf(256.f, (float)s1, (float)s0);
        sum[1] = 65536.f * (float)s2;
      }
      if (lane == 0) p.xinv[t * nkb + b] = d.inv;
    }
    if (p.gate_vec) {  // sigmoid(gate_vec . x[t])
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, off);
      float* part = reinterpret_cast<float*>(s_sums[0]);
      if (lane == 0) part[tid >> 5] = dot;
      __syncthreads();
      if (tid == 0) {
        float sum = 0.f;
        for (int w = 0; w < kBPlanThreads / 32; ++w) sum += part[w];
        p.gate[t] = 1.f / (1.f + expf(-sum));
      }
    }
    return;
  }
  const int npairs = p.T * p.k, slots = p.k + p.n_shared;
  const bool off = *p.ctl.extra_arrivals != 0u;
  int e = -1;
  unsigned hi = 0u;
  if (tid < npairs) {
    e = p.ids[tid];
    hi = p.prec[tid] != 0 ? 1u : 0u;
    if (e < 0 || e >= p.n_experts) {
      e = -1;
      atomicOr(p.ctl.status, (unsigned)SLICEMOE_STATUS_BAD_EXPERT_ID);
    }
  }
  s_e[tid] = e;
  s_high[tid] = 0u;
  // the expert's planes (the shared experts' for the threads that list those): asked for now, used at the end
  const int parts = (p.T + kBRun - 1) / kBRun, n_sh = p.n_shared * parts;
  // (the shared experts are listed by the last threads, which have a pair of their own only in the largest batches)
  const int sid = tid - (kBPlanThreads - n_sh);
  const slicemoe_expert* ex = e >= 0 ? p.experts + e : nullptr;
  const slicemoe_expert* exs = sid >= 0 ? p.shared + sid / parts : nullptr;
  const uint8_t* planes[3][4];
  auto fetch = [&](const slicemoe_expert* x) {
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const slicemoe_mat& mat = m == 0 ? x->gate : m == 1 ? x->up : x->down;
      planes[m][0] = reinterpret_cast<const uint8_t*>(mat.msb);
      planes[m][1] = reinterpret_cast<const uint8_t*>(mat.lsb);
      planes[m][2] = reinterpret_cast<const uint8_t*>(mat.scale);
      planes[m][3] = mat.zp;
    }
  };
  if (ex) fetch(ex);
  else if (exs) fetch(exs);
  __syncthreads();
  int rank = 0, count = 0, first = tid;
  for (int j = 0; j < npairs; ++j) {
    if (s_e[j] == e) {
      if (j < first) first = j;
      rank += j < tid;
      ++count;
    }
  }
  const bool valid = e >= 0;
  // pairs of one expert in list order, eight to a run; the run goes by the thread of its first pair
  int leader = first;
  if (valid && rank >= kBRun) {
    int seen = 0;
    for (int j = first; j < tid; ++j)
      if (s_e[j] == e && seen++ == (rank & ~(kBRun - 1))) leader = j;
    if ((rank & (kBRun - 1)) == 0) leader = tid;
  }
  if (valid) {
    atomicOr(&s_high[leader], hi << (rank & (kBRun - 1)));
    s_tok[leader][rank & (kBRun - 1)] = (uint8_t)(tid / p.k);
  }
  __syncthreads();
  const bool lead = valid && leader == tid;
  const int n = lead ? min(kBRun, count - rank) : 0;
  const unsigned bc = lead ? b_block_cost(n, s_high[tid]) : 0u;
  const unsigned u1 = 2u * bc * (p.hidden >> 7) + kBFixedCost;
  unsigned c2 = 0;
  if (lead) c2 = (bc * (p.inter >> 7) + kBFixedCost * p.kc_r) * (p.hidden / 16);
  unsigned sc[4] = {lead ? 1u : 0u, (unsigned)n, lead ? u1 * (p.inter / 16) : 0u, c2}, tot[4];
  b_scan(sc, s_sums, tot);
  const unsigned index = sc[0], prefix = sc[1], start1 = sc[2], start2 = sc[3], n_runs = tot[0], t1 = tot[2], t2 = tot[3];
  // a run's segments: one for gate and up, one for each chunk of down's columns
  auto emit = [&](BSeg g, unsigned block_cost, unsigned st1, unsigned st2, BSeg* to1, BSeg* to2, int kc_n, int yrow) {
    g.lsb = g.high != 0u;
    g.pad_[0] = g.pad_[1] = 0;
    auto point = [&](int to, int m) {
#pragma unroll
      for (int i = 0; i < 4; ++i) g.ptr[to][i] = planes[m][i];
      if (g.lsb && !g.ptr[to][1]) {  // both slices asked of an expert without LSB planes: defined garbage, reported
        g.ptr[to][1] = g.ptr[to][0];
        atomicOr(p.ctl.status, (unsigned)SLICEMOE_STATUS_MISSING_LSB);
      }
    };
    point(0, 0);
    point(1, 1);
    g.start = st1;
    g.ucost = 2u * block_cost * (p.hidden >> 7) + kBFixedCost;
    g.units = g.inter / 16;
    g.yrow = 0;
    g.kb0 = 0;
    g.nkb = g.row_kb = p.hidden >> 7;
    *to1 = g;
    point(0, 2);
    g.row_kb = g.inter >> 7;
    g.units = p.hidden / 16;
    for (int kc = 0; kc < kc_n; ++kc) {
      g.kb0 = kc * (kBChunkK / 128);
      g.nkb = b_chunk_cols(g.inter, kc) >> 7;
      g.start = st2;
      g.ucost = block_cost * g.nkb + kBFixedCost;
      g.yrow = yrow + kc * g.n;
      to2[kc] = g;
      st2 += g.ucost * (p.hidden / 16);
    }
  };
  if (lead) {
    BSeg g;
    g.n = n;
    g.high = s_high[tid];
    g.inter = p.inter;
    g.hoff = (int)prefix * p.inter;
    for (int i = 0; i < kBRun; ++i) g.tok[i] = i < n ? s_tok[tid][i] : s_tok[tid][0];
    emit(g, bc, start1, start2, p.seg1 + index, p.seg2 + index * p.kc_r, p.kc_r, (int)prefix * p.kc_r);
    s_index[tid] = (unsigned)n;
    s_prefix[tid] = prefix;
  }
  __syncthreads();
  if (tid < npairs)
    p.pos[(tid / p.k) * slots + tid % p.k] =
        valid ? make_int2((int)s_prefix[leader] * p.kc_r + (rank & (kBRun - 1)), (int)s_index[leader]) : make_int2(-1, 0);
  // shared experts: all tokens, both slices
  const unsigned bs = b_block_cost(min(p.T, kBRun), 0xffu);
  const unsigned cs1 = (2u * bs * (p.hidden >> 7) + kBFixedCost) * (p.shared_inter / 16);
  const unsigned cs2 = (bs * (p.shared_inter >> 7) + kBFixedCost * p.kc_s) * (p.hidden / 16);
  if (sid >= 0) {
    const int j = sid / parts, t0 = sid % parts * kBRun, ns = min(kBRun, p.T - t0);
    const int before = j * p.T + t0;  // pairs of shared experts before this run
    BSeg g;
    g.n = ns;
    g.high = 0xffu;
    g.inter = p.shared_inter;
    g.hoff = npairs * p.inter + before * p.shared_inter;
    for (int i = 0; i < kBRun; ++i) g.tok[i] = (uint8_t)(t0 + (i < ns ? i : 0));
    if (ex) fetch(exs);
    emit(g, bs, t1 + (unsigned)sid * cs1, t2 + (unsigned)sid * cs2, p.seg1 + n_runs + sid,
         p.seg2 + n_runs * p.kc_r + sid * p.kc_s, p.kc_s, npairs * p.kc_r + before * p.kc_s);
  }
  for (int i = tid; i < p.T * p.n_shared; i += kBPlanThreads) {
    const int t = i / p.n_shared, j = i % p.n_shared, t0 = t / kBRun * kBRun, ns = min(kBRun, p.T - t0);
    p.pos[t * slots + p.k + j] = make_int2(npairs * p.kc_r + (j * p.T + t0) * p.kc_s + (t - t0), ns);
  }
  if (tid == 0) {
    BHead h;
    const int sign = off ? -1 : 1;
    h.nseg[0] = sign * ((int)n_runs + n_sh);
    h.nseg[1] = sign * ((int)n_runs * p.kc_r + n_sh * p.kc_s);
    h.total[0] = t1 + (unsigned)n_sh * cs1;
    h.total[1] = t2 + (unsigned)n_sh * cs2;
    h.off = off ? 1 : 0;
    *p.head = h;
  }
}

// ---- the projections --------------------------------------------------------------------------------------
struct BParams {
  const BHead* head;
  const BSeg* segs;
  const uint8_t* xdig;
  const float *xsum, *xinv;
  float* h;
  float* yrow;
  BatchControl ctl;
  int hidden, K, shift;  // K: widest vector of digits (hidden, or a chunk of the intermediate width)
  int stages;            // per group
  int max_segs;          // entries the list can have
};
template <int G, int PHASE>
struct BSmem {
  static constexpr int kMeta = 8 * (128 / G) * 48;         // scales, then zero-points, of up to 8 blocks
  static constexpr int kStage = kBPlane + kMeta;
  static constexpr int kMats = PHASE == 1 ? 2 : 1;
  static constexpr int kPart = kBGroupWarps * kMats * kBRun * 20;  // floats: [warp][matrix][token][16 rows, padded]
  static constexpr int shares = 0;                                    // segments of the share ...
  static constexpr int range = shares + kBMaxSegs * (int)sizeof(BSeg);  // ... and their first and last row block of it
  static constexpr int ctl = range + kBMaxSegs * 8;                   // first and last segment, dead flag
  static constexpr int bars = ctl + 32;
  static constexpr int kMaxStages = 8;
  static constexpr int part = (bars + 2 * kBGroups * kMaxStages * 8 + 127) & ~127;
  static constexpr int dig = part + kBGroups * 2 * kPart * 4;
  __host__ __device__ static constexpr int tok_stride(int K) { return 3 * K + 32; }  // eight tokens' digit rows spread over the banks
  __host__ __device__ static constexpr int sums(int K) { return dig + kBRun * tok_stride(K); }            // float [K / G][digits 0 and 1, digit 2][8]
  __host__ __device__ static constexpr int inv(int K) { return sums(K) + 2 * (K / G) * kBRun * 4; }       // float [K / 128][8]
  __host__ __device__ static constexpr int ring(int K) { return (inv(K) + K / 128 * kBRun * 4 + 127) & ~127; }
};

constexpr unsigned long long kBCopyCycles = 2000000ull;  // a millisecond: far more than any copy takes
struct BWait {
  volatile int* dead;
  unsigned long long limit;
  unsigned* status;
  // true: the phase is there; false: it is not, and nobody waits any more
  __device__ __forceinline__ bool wait(uint32_t bar, uint32_t parity) const {
    const long long t0 = clock64();
    while (!*dead) {
      for (int i = 0; i < 64; ++i)
        if (mbar_try(bar, parity)) return true;
      if ((unsigned long long)(clock64() - t0) > limit) {
        *dead = 1;
        atomicOr(status, (unsigned)SLICEMOE_STATUS_WAIT_TIMEOUT);
      }
    }
    return false;
  }
};
// The consumers' wait: a call where the first look fails, not six copies of the loop (8 tokens of a 512-wide layer of 512-wide
// experts, top-4, G 64: 19.8 us, in line 20.7).
__device__ __noinline__ void b_wait_slow(uint32_t bar, uint32_t parity, BWait w) { w.wait(bar, parity); }
__device__ __forceinline__ void b_wait(uint32_t bar, uint32_t parity, const BWait& w) {
  if (!mbar_try(bar, parity)) b_wait_slow(bar, parity, w);
}
// The producers': their four lanes go on together or stop together.
__device__ __forceinline__ bool b_wait_lanes(uint32_t bar, uint32_t parity, const BWait& w) {
  return __all_sync(0xfu, mbar_try(bar, parity)) || __all_sync(0xfu, w.wait(bar, parity));
}

// One 16 x 128 block for eight tokens: acc[2 row half + token] += the block's contribution (lane (g, c): rows g and
// g + 8, tokens 2 c and 2 c + 1).
//   kModeHigh   all pairs use both slices: the nibbles are put together into 8-bit codes first, one MMA per 32 columns and
//               digit, and nothing to add up afterwards;
//   kModeLow    none does: the MSB nibbles alone, worth 2^shift;
//   kModeMixed  both products, and a pair's column takes the LSB product or not.
// Where nibbles are used as they are (low, mixed) the A fragment of rows g + 8 is the raw bytes, 16 x their nibble plus row
// g's: the difference of the accumulator rows is 16 C[g + 8], and the row's scale is divided by 16.
// WIDE: column n of the B operand is token n, an MMA per digit.  Otherwise, for up to two tokens, columns 4 t .. 4 t + 2 are the
// digits of token t, one MMA for all: even lanes c get digits 0 and 1 of token c / 2, odd ones digit 2.  The two exchange a
// row half's, so that an even lane finishes row g in acc[0] and an odd one row g + 8; `sc` and `zp` are at that row.
// Every form gives a token the same bits: the same exact integers (times a power of two that the row's scale takes back), rounded
// at the same points, blocks in the same order.  So what else is in a run does not show in a token's result.
enum { kModeLow = 0, kModeMixed = 1, kModeHigh = 2 };
template <int G, int MODE, bool WIDE>
__device__ __forceinline__ void b_block(const uint8_t* msb, const uint8_t* lsb, const uint8_t* sc, const uint8_t* zp, const uint8_t* dig,
                                        const float* X, const float* inv, int shift, int odd, unsigned low0, unsigned low1,
                                        float (&acc)[4]) {
  constexpr int SG = 128 / G, KS = G / 32;
  constexpr uint32_t kLow = 0x0f0f0f0fu;
  float2 iv;
  if (WIDE) iv = *reinterpret_cast<const float2*>(inv);
  else iv.x = *inv;
  constexpr int ND = WIDE ? 3 : 1;
#pragma unroll
  for (int sg = 0; sg < SG; ++sg) {
    // the group's words of the lane, 16 columns each: [plane], or [row half] of the codes
    constexpr int W = G / 16;
    uint32_t a[2][W];
    if (W == 2) {  // half of a 64-column tile
      const uint2 v = *reinterpret_cast<const uint2*>(msb + (sg >> 1) * 512 + (sg & 1) * 8);
      a[0][0] = v.x; a[0][1] = v.y;
      if (MODE != kModeLow) {
        const uint2 u = *reinterpret_cast<const uint2*>(lsb + (sg >> 1) * 512 + (sg & 1) * 8);
        a[1][0] = u.x; a[1][1] = u.y;
      }
    } else {
#pragma unroll
      for (int h = 0; h < W / 4; ++h) {
        const uint4 v = *reinterpret_cast<const uint4*>(msb + (sg * (W / 4) + h) * 512);
        a[0][(4 * h) % W] = v.x; a[0][(4 * h + 1) % W] = v.y; a[0][(4 * h + 2) % W] = v.z; a[0][(4 * h + 3) % W] = v.w;
        if (MODE != kModeLow) {
          const uint4 u = *reinterpret_cast<const uint4*>(lsb + (sg * (W / 4) + h) * 512);
          a[1][(4 * h) % W] = u.x; a[1][(4 * h + 1) % W] = u.y; a[1][(4 * h + 2) % W] = u.z; a[1][(4 * h + 3) % W] = u.w;
        }
      }
    }
    if (MODE == kModeHigh) {
      // a slice narrower than four bits leaves the top of its nibble zero, so what the masks let through beyond it is zero
      const uint32_t mask = kLow << shift;
      const int back = 4 - shift;
#pragma unroll
      for (int w = 0; w < W; ++w) {
        const uint32_t m = a[0][w], l = a[1][w];
        a[0][w] = ((m << shift) & mask) | (l & ~mask);
        a[1][w] = ((m >> back) & mask) | ((l >> 4) & ~mask);
      }
    }
    int v[ND][4];
#pragma unroll
    for (int d = 0; d < ND; ++d) {
      int m[4], l[4];
#pragma unroll
      for (int s = 0; s < KS; ++s) {
        const int ks = sg * KS + s;
        const uint2 b = *reinterpret_cast<const uint2*>(dig + ks * 96 + d * 32);
        const uint32_t w0 = a[0][2 * s], w1 = a[0][2 * s + 1], u0 = a[1][2 * s], u1 = a[1][2 * s + 1];
        if (MODE == kModeHigh) {
          if (s == 0) mma_u8s8_first(m, w0, u0, w1, u1, b.x, b.y);
          else mma_u8s8(m, w0, u0, w1, u1, b.x, b.y);
        } else {
          if (s == 0) mma_u8s8_first(m, w0 & kLow, w0, w1 & kLow, w1, b.x, b.y);
          else mma_u8s8(m, w0 & kLow, w0, w1 & kLow, w1, b.x, b.y);
          if (MODE == kModeMixed) {
            if (s == 0) mma_u8s8_first(l, u0 & kLow, u0, u1 & kLow, u1, b.x, b.y);
            else mma_u8s8(l, u0 & kLow, u0, u1 & kLow, u1, b.x, b.y);
          }
        }
      }
      if (MODE != kModeHigh) {
        m[2] -= m[0];
        m[3] -= m[1];
      }
      if (MODE == kModeMixed) {
        l[2] -= l[0];
        l[3] -= l[1];
#pragma unroll
        for (int i = 0; i < 4; ++i) m[i] = (m[i] << shift) + (l[i] & ((i & 1) ? ~low1 : ~low0));
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) v[d][i] = m[i];
    }
    // rows g and g + 8; in the narrow form the lane's own row, twice
    float s0 = __half2float(*reinterpret_cast<const __half*>(sc + sg * 32)), s1 = WIDE ? __half2float(*reinterpret_cast<const __half*>(sc + sg * 32 + 16)) : s0;
    unsigned z0 = zp[sg * 16], z1 = WIDE ? zp[sg * 16 + 8] : z0;
    if (MODE == kModeLow) {  // 2^shift (q_msb - (zp >> shift)): the power of two goes into the scale
      const float two = (float)(1 << shift);
      z0 >>= shift;
      z1 >>= shift;
      s0 *= two;
      s1 *= two;
    }
    if (MODE != kModeHigh) {
      s1 *= 0.0625f;
      z1 <<= 4;
    }
    // a pair at MSB precision among others at both slices: 2^shift (zp >> shift)
    const unsigned drop = (1u << shift) - 1u;
    // Digits 0 and 1 go together in 32 bits: 255 x 128 x 128 x 257 at most.  Not so in the rows of a mixed run that carry a factor
    // of 16.  Digit 2 joins in fp32.
    if (WIDE) {
      const float2 xl = *reinterpret_cast<const float2*>(X + sg * 2 * kBRun), xh = *reinterpret_cast<const float2*>(X + sg * 2 * kBRun + kBRun);
      const float x0 = xl.x + xh.x, x1 = xl.y + xh.y;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const bool mixed16 = MODE == kModeMixed && i >= 2;
        float t = mixed16 ? fmaf((float)v[ND - 1][i], 65536.f, fmaf((float)v[ND / 2][i], 256.f, (float)v[0][i]))
                          : fmaf((float)v[ND - 1][i], 65536.f, (float)(v[0][i] + v[ND / 2][i] * 256));
        unsigned z = i >= 2 ? z1 : z0;
        if (MODE == kModeMixed) z &= ~(((i & 1) ? low1 : low0) & (i >= 2 ? drop << 4 : drop));
        t = fmaf(-(float)z, (i & 1) ? x1 : x0, t);
        acc[i] = fmaf((i >= 2 ? s1 : s0) * ((i & 1) ? iv.y : iv.x), t, acc[i]);
      }
    } else {
      // digits 0 and 1 of both row halves in an even lane, digit 2 of both in an odd one
      const float f0 = (float)(odd ? v[0][0] : v[0][0] + v[0][1] * 256);
      const float f1 = odd ? (float)v[0][2]
                           : MODE == kModeMixed ? fmaf((float)v[0][3], 256.f, (float)v[0][2]) : (float)(v[0][2] + v[0][3] * 256);
      const float got = __shfl_xor_sync(0xffffffffu, odd ? f0 : f1, 1);
      const float x = X[sg * 2 * kBRun] + X[sg * 2 * kBRun + kBRun];
      float t = odd ? fmaf(f1, 65536.f, got) : fmaf(got, 65536.f, f0);
      unsigned z = odd ? z1 : z0;
      if (MODE == kModeMixed) z &= ~(low0 & (odd ? drop << 4 : drop));
      t = fmaf(-(float)z, x, t);
      acc[0] = fmaf((odd ? s1 : s0) * iv.x, t, acc[0]);
    }
  }
}

// A consumer warp's part of a share's row blocks `u`, u + kBGroups, ... below `last`.
struct BState {
  int st, half;   // stage, buffer of partial rows
  uint32_t par;   // parity of the stage's use
};
template <int G, int PHASE, int MODE, bool WIDE>
__device__ __forceinline__ void b_rows(const BParams& p, const BSeg& sh, int u, int last, uint32_t fb, const uint8_t* ring, float* part,
                                       const uint8_t* dig, const float* X, const float* inv, int stride, int group, int gw, int lane,
                                       const BWait& wait, BState& state) {
  using S = BSmem<G, PHASE>;
  constexpr int SG = 128 / G;
  constexpr int per = MODE == kModeLow ? 8 : 4;  // blocks of a stage
  const int g8 = lane >> 2, c = lane & 3, n = sh.n, nkb = sh.nkb, shift = p.shift;
  // the lane's tokens: 2 c and 2 c + 1, or c / 2
  const int tk0 = WIDE ? 2 * c : c >> 1, tk1 = WIDE ? 2 * c + 1 : c >> 1;
  const unsigned low0 = (sh.high >> tk0) & 1u ? 0u : 0xffffffffu, low1 = (sh.high >> tk1) & 1u ? 0u : 0xffffffffu;
  // columns without a token repeat the last one's; the narrow form's fourth column repeats a digit
  const uint8_t* my_dig = dig + c * 8 + (WIDE ? min(g8, n - 1) * stride : min(g8 >> 2, n - 1) * stride + min(g8 & 3, 2) * 32);
  const float* my_X = X + (WIDE ? 2 * c : c >> 1);
  const int my_row = WIDE ? g8 : g8 + 8 * (c & 1);  // first row of the lane
  const float* my_inv = inv + tk0;
  int st = state.st, half = state.half;
  uint32_t par = state.par;
  for (; u < last; u += kBGroups) {
    float* pb = part + half * S::kPart;
#pragma unroll 1
    for (int m = 0; m < S::kMats; ++m) {
      float acc[4] = {0.f, 0.f, 0.f, 0.f};
      for (int b0 = 0; b0 < nkb; b0 += per) {
        b_wait(fb + 16 * st, par, wait);
        const uint8_t* stage = ring + st * S::kStage;
        const int nb = min(per, nkb - b0);
#pragma unroll 1
        for (int b = gw; b < nb; b += kBGroupWarps)
          b_block<G, MODE, WIDE>(stage + b * 1024 + lane * 16, stage + kBPlane / 2 + b * 1024 + lane * 16, stage + kBPlane + b * (SG * 32) + my_row * 2,
                                 stage + kBPlane + 8 * SG * 32 + b * (SG * 16) + my_row, my_dig + (b0 + b) * 384, my_X + (b0 + b) * SG * 2 * kBRun,
                                 my_inv + (b0 + b) * kBRun, shift, c & 1, low0, low1, acc);
        __syncwarp();
        if (lane == 0) mbar_arrive(fb + 16 * st + 8);
        if (++st == p.stages) { st = 0; par ^= 1; }
      }
      float* w = pb + (gw * S::kMats + m) * (kBRun * 20);
      if (WIDE) {
        w[(2 * c) * 20 + g8] = acc[0];
        w[(2 * c + 1) * 20 + g8] = acc[1];
        w[(2 * c) * 20 + g8 + 8] = acc[2];
        w[(2 * c + 1) * 20 + g8 + 8] = acc[3];
      } else {
        w[(c >> 1) * 20 + my_row] = acc[0];
      }
    }
    // the four warps' shares of the columns, added in warp order by a thread per (token, row); two buffers take turns
    asm volatile("bar.sync %0, %1;" ::"r"(2 + group), "n"(32 * kBGroupWarps) : "memory");
    const int t = (gw * 32 + lane) >> 4, row = lane & 15;
    if (t < n) {
      float s[2] = {0.f, 0.f};
#pragma unroll
      for (int w = 0; w < kBGroupWarps; ++w)
#pragma unroll
        for (int m = 0; m < S::kMats; ++m) s[m] += pb[(w * S::kMats + m) * (kBRun * 20) + t * 20 + row];
      if (PHASE == 1) p.h[sh.hoff + (size_t)t * sh.inter + u * 16 + row] = s[0] / (1.f + expf(-s[0])) * s[1];  // silu(gate) * up
      else p.yrow[(size_t)(sh.yrow + t) * p.hidden + u * 16 + row] = s[0];
    }
    half ^= 1;
  }
  state.st = st;
  state.half = half;
  state.par = par;
}

template <int G, int PHASE>
__global__ void __launch_bounds__(kBThreads, 1) batch_ffn_kernel(const __grid_constant__ BParams p) {
  using S = BSmem<G, PHASE>;
  constexpr int SG = 128 / G;
  extern __shared__ __align__(128) uint8_t smem[];
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  BSeg* shares = reinterpret_cast<BSeg*>(smem + S::shares);
  int2* range = reinterpret_cast<int2*>(smem + S::range);
  int* ctl = reinterpret_cast<int*>(smem + S::ctl);
  volatile int* dead = ctl + 2;
  const uint32_t bars = smem_u32(smem + S::bars);
  if (tid == 0) {
    ctl[0] = 0x7fffffff;
    ctl[1] = -1;
    *dead = 0;
    for (int i = 0; i < kBGroups * p.stages; ++i) {
      mbar_init(bars + 16 * i, 1);                // full: the producer's arrive, and the bytes
      mbar_init(bars + 16 * i + 8, kBGroupWarps); // empty
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncthreads();
  // The gate/up launch waits for the plan before it lets the next launch start.  So the down launch, when it starts, finds the
  // plan complete: it looks up its share and streams its weights while gate/up is still running, and waits only for h.
  if (PHASE == 1) {
    b_dep_wait();
    b_dep_launch();
  }
  const unsigned long long lim = *p.ctl.wait_cycles;
  BWait wait;
  wait.dead = dead;
  wait.limit = lim != 0ull ? lim : kWaitCycles;
  wait.status = p.ctl.status;
  bool off;
  // This CTA's share: the row blocks whose start, in cost, lies in its window.  A thread per segment; everything a role needs
  // to know about a segment is in its entry, so the way to the first copy is two trips to L2.
  {
    const uint4 head = tid < p.max_segs ? __ldcg(reinterpret_cast<const uint4*>(p.segs + tid)) : make_uint4(0u, 1u, 0u, 0u);
    const int said = __ldcg(&p.head->nseg[PHASE - 1]), nseg = abs(said);
    off = said < 0;
    const unsigned long long total = __ldcg(&p.head->total[PHASE - 1]);
    const unsigned lo = (unsigned)((total * blockIdx.x + gridDim.x - 1) / gridDim.x);
    const unsigned hi = (unsigned)((total * (blockIdx.x + 1) + gridDim.x - 1) / gridDim.x);
    int2 r = make_int2(0, 0);
    if (tid < nseg) {
      auto ord = [&](unsigned at) { return at <= head.x ? 0 : (int)min(head.z, (at - head.x + head.y - 1) / head.y); };
      r = make_int2(ord(lo), ord(hi));
    }
    if (r.y > r.x) {
      atomicMin(&ctl[0], tid);
      atomicMax(&ctl[1], tid);
    }
    __syncthreads();
    const int s0 = ctl[0], n = min(ctl[1] - s0 + 1, kBMaxSegs);
    if (r.y > r.x && tid - s0 < kBMaxSegs) range[tid - s0] = r;
    for (int i = warp; i < n; i += kBThreads / 32)
      reinterpret_cast<uint32_t*>(shares + i)[lane] = __ldcg(reinterpret_cast<const uint32_t*>(p.segs + s0 + i) + lane);
    __syncthreads();
  }
  const int ns = ctl[1] < 0 ? 0 : min(ctl[1] - ctl[0] + 1, kBMaxSegs);
  uint8_t* ring0 = smem + S::ring(p.K);

  if (warp >= kBConsumers) {
    // ---- producer of a group: lane 0 the MSB plane, 1 the LSB plane, 2 the scales, 3 the zero-points ----
    if (lane >= 4) return;
    if (off) return;  // the time-out exercise: nothing is asked for, and the consumers' waits run out
    const int group = warp - kBConsumers;
    const uint32_t fb = bars + 16 * group * p.stages;
    const uint32_t ring = smem_u32(ring0 + (size_t)group * p.stages * S::kStage);
    const uint64_t pol = l2_evict_first_policy();
    const unsigned per_block = lane < 2 ? 1024u : (lane == 2 ? SG * 32u : SG * 16u);
    int st = 0, ord = 0;
    uint32_t par = 1, used = 0;
    bool ok = true;
    for (int i = 0; i < ns && ok; ++i) {
      const BSeg& sh = shares[i];
      const int u0 = range[i].x, u1 = range[i].y;
      const int nkb = sh.nkb, per = sh.lsb ? 4 : 8;
      const bool active = lane != 1 || sh.lsb;
      const unsigned dst0 = lane == 0 ? 0u : lane == 1 ? kBPlane / 2 : lane == 2 ? kBPlane : kBPlane + 8 * SG * 32;
      // the group's row blocks: every kBGroups-th of the share
      for (int u = u0 + ((group - ord) & (kBGroups - 1)); u < u1 && ok; u += kBGroups) {
#pragma unroll 1
        for (int m = 0; m < S::kMats && ok; ++m) {
          const uint8_t* src = sh.ptr[m][lane] + ((size_t)u * sh.row_kb + sh.kb0) * per_block;
          for (int b0 = 0; b0 < nkb; b0 += per) {
            const unsigned nb = (unsigned)min(per, nkb - b0);
            // the down launch's first lap round the ring finds it empty; after that space is the consumers' doing, who wait for
            // the gate/up launch first: that is no part of the limit on this wait
            if (PHASE == 2 && used == (uint32_t)p.stages) b_dep_wait();
            ok = b_wait_lanes(fb + 16 * st + 8, par, wait);
            if (!ok) break;
            if (lane == 0) mbar_arrive_expect_tx(fb + 16 * st, nb * ((sh.lsb ? 2048u : 1024u) + SG * 48u));
            __syncwarp(0xfu);
            if (active) bulk_g2s(ring + st * S::kStage + dst0, src, nb * per_block, fb + 16 * st, pol);
            src += nb * per_block;
            ++used;
            if (++st == p.stages) { st = 0; par ^= 1; }
          }
        }
      }
      ord += u1 - u0;
    }
    // no copy may be on its way when the CTA ends (in the normal case the consumers have seen them all land)
    const unsigned long long drain = wait.limit > kBCopyCycles ? wait.limit : kBCopyCycles;
    for (uint32_t i = used > (uint32_t)p.stages ? used - p.stages : 0; i < used; ++i) {
      const long long t0 = clock64();
      while (!mbar_try(fb + 16 * (i % p.stages), (i / p.stages) & 1) && (unsigned long long)(clock64() - t0) < drain) {}
    }
    return;
  }

  // ---- consumers ----
  const int group = warp / kBGroupWarps, gw = warp % kBGroupWarps;
  const uint32_t fb = bars + 16 * group * p.stages;
  const uint8_t* ring = ring0 + (size_t)group * p.stages * S::kStage;
  float* part = reinterpret_cast<float*>(smem + S::part) + group * 2 * S::kPart;
  uint8_t* dig = smem + S::dig;
  float* X = reinterpret_cast<float*>(smem + S::sums(p.K));
  float* inv = reinterpret_cast<float*>(smem + S::inv(p.K));
  const int stride = S::tok_stride(p.K);
  if (PHASE == 2) {
    b_dep_wait();  // h
    b_dep_launch();
  }
  BState state = {0, 0, 0u};
  int ord = 0;
  for (int i = 0; i < ns; ++i) {
    const BSeg& sh = shares[i];
    const int u0 = range[i].x, u1 = range[i].y, n = sh.n, nkb = sh.nkb;
    if (i > 0) asm volatile("bar.sync 1, %0;" ::"n"(32 * kBConsumers) : "memory");  // the digits of the run before have been used
    // the run's vectors as digits: x's are copied (the plan launch has worked them out), h's are worked out here.  Several
    // loads in flight together: each is a trip to L2
    if (PHASE == 1) {
      const int per = 3 * p.hidden / 16, ngrp = p.hidden / G;
      for (int at = tid; at < per; at += 32 * kBConsumers)
        for (int t0 = 0; t0 < n; t0 += 4) {
          uint4 raw[4];
#pragma unroll
          for (int t = 0; t < 4; ++t)
            if (t0 + t < n) raw[t] = __ldcg(reinterpret_cast<const uint4*>(p.xdig + (size_t)sh.tok[t0 + t] * 3 * p.hidden) + at);
#pragma unroll
          for (int t = 0; t < 4; ++t)
            if (t0 + t < n) *(reinterpret_cast<uint4*>(dig + (t0 + t) * stride) + at) = raw[t];
        }
      for (int at = tid; at < n * 2 * ngrp; at += 32 * kBConsumers) {
        const int t = at / (2 * ngrp), g = at - t * 2 * ngrp;
        X[g * kBRun + t] = __ldcg(p.xsum + (size_t)sh.tok[t] * 2 * ngrp + g);
      }
      for (int at = tid; at < n * nkb; at += 32 * kBConsumers) {
        const int t = at / nkb, b = at - t * nkb;
        inv[b * kBRun + t] = __ldcg(p.xinv + sh.tok[t] * nkb + b);
      }
    } else {
      constexpr int kAhead = 4;
      for (int blk0 = warp; blk0 < n * nkb; blk0 += kAhead * kBConsumers) {
        uint4 raw[kAhead];
#pragma unroll
        for (int a = 0; a < kAhead; ++a) {
          const int blk = blk0 + a * kBConsumers, t = blk / nkb, b = blk - t * nkb;
          if (blk < n * nkb) raw[a] = __ldcg(reinterpret_cast<const uint4*>(p.h + sh.hoff + (size_t)t * sh.inter + (sh.kb0 + b) * 128) + lane);
        }
#pragma unroll
        for (int a = 0; a < kAhead; ++a) {
          const int blk = blk0 + a * kBConsumers, t = blk / nkb, b = blk - t * nkb;
          if (blk >= n * nkb) break;
          const float v[4] = {__uint_as_float(raw[a].x), __uint_as_float(raw[a].y), __uint_as_float(raw[a].z), __uint_as_float(raw[a].w)};
          const BlockDigits d = block_digits(v);
          store_digits(d, b * 128 + 4 * lane, dig + t * stride);
          int s0, s1, s2;
          group_digit_sums<G>(d, lane, s0, s1, s2);
          if ((lane & (G / 4 - 1)) == 0) {
            float* x = X + (b * SG + lane / (G / 4)) * 2 * kBRun + t;
            x[0] = fmaf(256.f, (float)s1, (float)s0);
            x[kBRun] = 65536.f * (float)s2;
          }
          if (lane == 0) inv[b * kBRun + t] = d.inv;
        }
      }
    }
    asm volatile("bar.sync 1, %0;" ::"n"(32 * kBConsumers) : "memory");
    const unsigned all = (1u << n) - 1u;
    const int first = u0 + ((group - ord) & (kBGroups - 1));
    const bool high = (sh.high & all) == all;
    auto rows = [&](auto mode, auto wide) {
      b_rows<G, PHASE, decltype(mode)::value, decltype(wide)::value>(p, sh, first, u1, fb, ring, part, dig, X, inv, stride, group, gw, lane, wait, state);
    };
    using std::integral_constant;
    if (n > 2) {
      if (!sh.lsb) rows(integral_constant<int, kModeLow>(), std::true_type());
      else if (high) rows(integral_constant<int, kModeHigh>(), std::true_type());
      else rows(integral_constant<int, kModeMixed>(), std::true_type());
    } else {
      if (!sh.lsb) rows(integral_constant<int, kModeLow>(), std::false_type());
      else if (high) rows(integral_constant<int, kModeHigh>(), std::false_type());
      else rows(integral_constant<int, kModeMixed>(), std::false_type());
    }
    ord += u1 - u0;
  }
}

// ---- combine ---------------------------------------------------------------------------------------------
constexpr int kBCombineThreads = 256;
struct BCombine {
  const BHead* head;
  const float* yrow;
  const int2* pos;
  const float* weights;
  const float* gate;  // or null
  float* y;
  int k, n_shared, hidden, kc_r, kc_s;
};
__global__ void __launch_bounds__(kBCombineThreads) batch_combine_kernel(const BCombine p) {
  const int t = blockIdx.y, col = (blockIdx.x * kBCombineThreads + threadIdx.x) * 2, slots = p.k + p.n_shared;
  b_dep_launch();
  b_dep_wait();
  __shared__ int4 s_at[SLICEMOE_MAX_TOP_K + SLICEMOE_MAX_SHARED];  // first row, rows from chunk to chunk, chunks, weight
  if (threadIdx.x < slots) {
    const int j = threadIdx.x;
    const int2 at = p.pos[t * slots + j];
    const float w = j < p.k ? p.weights[t * p.k + j] : p.gate ? p.gate[t] : 1.f;
    s_at[j] = make_int4(at.x, at.y, j < p.k ? p.kc_r : p.kc_s, __float_as_int(w));
  }
  const bool off = p.head->off != 0;
  __syncthreads();
  if (col >= p.hidden || off) return;
  float2 a = make_float2(0.f, 0.f);
  for (int j0 = 0; j0 < slots; j0 += 4) {
    float2 v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (j0 + j < slots && s_at[j0 + j].x >= 0) v[j] = __ldcg(reinterpret_cast<const float2*>(p.yrow + (size_t)s_at[j0 + j].x * p.hidden + col));
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (j0 + j >= slots || s_at[j0 + j].x < 0) continue;
      const int4 at = s_at[j0 + j];
      for (int kc = 1; kc < at.z; ++kc) {
        const float2 u = __ldcg(reinterpret_cast<const float2*>(p.yrow + (size_t)(at.x + kc * at.y) * p.hidden + col));
        v[j].x += u.x;
        v[j].y += u.y;
      }
      a.x = fmaf(__int_as_float(at.w), v[j].x, a.x);
      a.y = fmaf(__int_as_float(at.w), v[j].y, a.y);
    }
  }
  float* y = p.y + (size_t)t * p.hidden + col;
  if ((reinterpret_cast<uintptr_t>(y) & 7) == 0) {
    *reinterpret_cast<float2*>(y) = a;
  } else {  // a caller's y that starts on any float, as the batch-1 kernel takes it
    y[0] = a.x;
    y[1] = a.y;
  }
}

// ---- host side ---------------------------------------------------------------------------------------------
template <class P>
static int b_launch(void (*kernel)(P), dim3 grid, unsigned threads, size_t smem, cudaStream_t st, const P& params) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  SM_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, params));
  return SLICEMOE_OK;
}

constexpr int kBSmemMax = 227 * 1024;
constexpr int kBMaxHidden = 4096;
template <int G, int PHASE>
static int b_launch_ffn(BParams p, int sms, cudaStream_t st) {
  static bool attr_set[64];
  int dev = 0;
  SM_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return SLICEMOE_E_UNSUPPORTED;
  if (!attr_set[dev]) {
    SM_CUDA_TRY(cudaFuncSetAttribute(batch_ffn_kernel<G, PHASE>, cudaFuncAttributeMaxDynamicSharedMemorySize, kBSmemMax));
    attr_set[dev] = true;
  }
  using S = BSmem<G, PHASE>;
  // As many stages as shared memory holds beside the digits of eight tokens: bytes in flight are what the bandwidth needs.
  // Gate/up: three per group at hidden 2048, two at 4096, one at 4096 with G 32, where copy and arithmetic take turns (four
  // tokens that share none of their experts of 1408: 84 us, token after token 80, the one layer of 30 where that is ahead).
  static_assert(S::ring(PHASE == 1 ? kBMaxHidden : kBChunkK) + kBGroups * S::kStage <= kBSmemMax, "one stage at least");
  p.stages = (kBSmemMax - S::ring(p.K)) / (kBGroups * S::kStage);
  if (p.stages > S::kMaxStages) p.stages = S::kMaxStages;
  return b_launch(batch_ffn_kernel<G, PHASE>, dim3((unsigned)sms), kBThreads,
                  (size_t)S::ring(p.K) + (size_t)kBGroups * p.stages * S::kStage, st, p);
}

template <int G>
static int b_launch_all(const BPlanParams& pp, BParams p1, BParams p2, int sms, cudaStream_t st) {
  int rc = b_launch(batch_plan_kernel<G>, dim3((unsigned)(1 + pp.T)), kBPlanThreads, 0, st, pp);
  if (rc == SLICEMOE_OK) rc = b_launch_ffn<G, 1>(p1, sms, st);
  if (rc == SLICEMOE_OK) rc = b_launch_ffn<G, 2>(p2, sms, st);
  return rc;
}

int batch_layer(const slicemoe_shape* s, const slicemoe_expert* experts, const slicemoe_expert* shared, int n_shared,
                const float* gate_vec, const uint16_t* x, int T, const int32_t* ids, const uint8_t* prec, const float* weights,
                float* y, void* workspace, const BatchControl& ctl, int sms, void* stream) {
  const BLayout L = batch_layout(s, n_shared);
  uint8_t* ws = reinterpret_cast<uint8_t*>(workspace);
  cudaStream_t st = (cudaStream_t)stream;
  const bool gated = n_shared > 0 && s->shared_sigmoid_gate;
  BPlanParams pp;
  pp.ids = ids;
  pp.prec = prec;
  pp.x = x;
  pp.gate_vec = gated ? gate_vec : nullptr;
  pp.T = T;
  pp.k = s->top_k;
  pp.n_experts = s->n_experts;
  pp.n_shared = n_shared;
  pp.hidden = s->hidden;
  pp.inter = s->inter;
  pp.shared_inter = n_shared ? s->shared_inter : 0;
  pp.kc_r = L.kc_r;
  pp.kc_s = L.kc_s;
  pp.head = reinterpret_cast<BHead*>(ws + L.head);
  pp.experts = experts;
  pp.shared = shared;
  pp.seg1 = reinterpret_cast<BSeg*>(ws + L.seg1);
  pp.seg2 = reinterpret_cast<BSeg*>(ws + L.seg2);
  pp.pos = reinterpret_cast<int2*>(ws + L.pos);
  pp.gate = reinterpret_cast<float*>(ws + L.gate);
  pp.xdig = ws + L.xdig;
  pp.xsum = reinterpret_cast<float*>(ws + L.xsum);
  pp.xinv = reinterpret_cast<float*>(ws + L.xinv);
  pp.ctl = ctl;
  BParams p;
  p.head = pp.head;
  p.segs = pp.seg1;
  p.xdig = pp.xdig;
  p.xsum = pp.xsum;
  p.xinv = pp.xinv;
  p.h = reinterpret_cast<float*>(ws + L.h);
  p.yrow = reinterpret_cast<float*>(ws + L.yrow);
  p.ctl = ctl;
  p.hidden = s->hidden;
  p.K = s->hidden;
  p.shift = s->b_high - s->b_low;
  p.stages = 0;
  const int parts = (T + kBRun - 1) / kBRun;
  p.max_segs = T * s->top_k + n_shared * parts;
  BParams p2 = p;
  p2.segs = pp.seg2;
  p2.max_segs = T * s->top_k * L.kc_r + n_shared * parts * L.kc_s;
  const int widest = s->inter > pp.shared_inter ? s->inter : pp.shared_inter;
  p2.K = widest < kBChunkK ? widest : kBChunkK;
  const int rc = s->group == 128 ? b_launch_all<128>(pp, p, p2, sms, st)
                 : s->group == 64 ? b_launch_all<64>(pp, p, p2, sms, st) : b_launch_all<32>(pp, p, p2, sms, st);
  if (rc != SLICEMOE_OK) return rc;
  BCombine c;
  c.head = pp.head;
  c.yrow = p.yrow;
  c.pos = pp.pos;
  c.weights = weights;
  c.gate = gated ? pp.gate : nullptr;
  c.y = y;
  c.k = s->top_k;
  c.n_shared = n_shared;
  c.hidden = s->hidden;
  c.kc_r = L.kc_r;
  c.kc_s = L.kc_s;
  return b_launch(batch_combine_kernel, dim3((unsigned)((s->hidden / 2 + kBCombineThreads - 1) / kBCombineThreads), (unsigned)T),
                  kBCombineThreads, 0, st, c);
}

}  // namespace slicemoe
