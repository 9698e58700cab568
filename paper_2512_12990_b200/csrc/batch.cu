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
// The two projections are one kernel.  A CTA (one per SM) takes an equal share, by bytes, of the row blocks of all runs.
// Four groups of a producer warp and four consumer warps each take the share's row blocks in turn: the producer
// streams the planes, scales and zero-points through the group's own ring with bulk copies, never waiting for anything but
// space; the consumers split a row block's 128-column blocks.  The arithmetic is the batch-1 kernel's: activations
// as 23-bit fixed point per 128-element block in three base-256 digits (int8), integer MMAs on the raw nibbles,
// scale and zero-point once per group.  Column n of the MMA's B operand is token n, one MMA per digit: a lane ends up
// with all digits of its two tokens, so the digits are put together in its registers and a row block's result is two
// values per lane, row half and matrix.  A pair at MSB precision shares the run with pairs at both slices: its columns
// leave out the LSB sums and the zero-point's low bits.
//
// Bound: HBM.  Per 16 x 128 block of both planes (2 KB, 89 cycles of an SM's share of the bandwidth) a warp issues about 125
// instructions, 24 of them MMAs (53 cycles of the integer tensor pipe).
// Measured, 8 tokens, 64 x 1408 top-6 + 2 shared, hidden 2048: eight batch-1 launches 133 us, this BATCH_US.
//
// Bounded waits: when one runs out the CTA's dead flag goes up and SLICEMOE_STATUS_WAIT_TIMEOUT is set; from then on nobody
// waits for data, the consumers walk through the rest of their work and the producers stop and wait for their copies.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "batch.cuh"
#include "common.cuh"
#include "decode_common.cuh"

namespace slicemoe {

constexpr int kBRun = 8;                 // pairs of a run: the columns of an MMA
constexpr int kBGroups = 4, kBGroupWarps = 4, kBConsumers = kBGroups * kBGroupWarps;
constexpr int kBThreads = 32 * (kBConsumers + kBGroups);
constexpr int kBChunkK = 2048;           // columns of a down projection's task; wider experts are several
constexpr int kBPlane = 8192;            // plane bytes of a stage: 4 blocks of both slices or 8 of the MSB slice
constexpr int kBMaxSegs = 40;            // runs that a CTA's share can touch
constexpr int kBFixedCost = 4;           // a row block's cost besides its plane blocks, in plane blocks
constexpr int kBPlanThreads = 256;
static_assert(kBatchTokens * SLICEMOE_MAX_TOP_K <= kBPlanThreads, "a thread per pair");

struct __align__(16) BRun {
  int expert;          // routed: 0 .., shared: n_experts ..
  int n;
  unsigned high;       // bit per pair: both slices
  int inter;
  int hoff;            // first h of the run: [n][inter]
  int pad_;
  uint8_t tok[kBRun];
};
struct __align__(16) BSeg {  // the row blocks of a run in one projection (down: for one chunk of columns)
  int run, kc;
  unsigned start, ucost;     // cost before the segment, cost of a row block
  int units;
  int yrow;                  // down: first result row of the segment
  int pad_[2];
};
struct BHead {
  int nseg[2];
  unsigned total[2];
  int off;                   // nothing is to be computed
};

struct BLayout {
  size_t head, runs, seg1, seg2, pos, gate, h, yrow, total;
  int kc_r, kc_s, max_runs, max_seg2;
};
static inline BLayout batch_layout(const slicemoe_shape* s, int n_shared) {
  BLayout L;
  const int T = kBatchTokens, k = s->top_k, parts = (T + kBRun - 1) / kBRun;
  const int sint = n_shared ? s->shared_inter : 0;
  L.kc_r = (s->inter + kBChunkK - 1) / kBChunkK;
  L.kc_s = (sint + kBChunkK - 1) / kBChunkK;
  L.max_runs = T * k + n_shared * parts;
  L.max_seg2 = T * k * L.kc_r + n_shared * parts * L.kc_s;
  auto align = [](size_t v) { return (v + 255) & ~(size_t)255; };
  size_t o = 0;
  L.head = o; o = align(o + sizeof(BHead));
  L.runs = o; o = align(o + sizeof(BRun) * L.max_runs);
  L.seg1 = o; o = align(o + sizeof(BSeg) * L.max_runs);
  L.seg2 = o; o = align(o + sizeof(BSeg) * L.max_seg2);
  L.pos = o;  o = align(o + sizeof(int2) * T * (k + n_shared));
  L.gate = o; o = align(o + sizeof(float) * T);
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
  BHead* head;
  BRun* runs;
  BSeg *seg1, *seg2;
  int2* pos;
  float* gate;
  BatchControl ctl;
};
__device__ __forceinline__ unsigned b_cost1(int planes, int hidden) { return 2u * planes * (hidden >> 7) + kBFixedCost; }
__device__ __forceinline__ int b_chunk_cols(int inter, int kc) { return min(kBChunkK, inter - kc * kBChunkK); }
__device__ __forceinline__ unsigned b_cost2(int planes, int cols) { return planes * (cols >> 7) + kBFixedCost; }
// Block-wide exclusive scan; *total gets the sum.
__device__ unsigned b_scan(unsigned v, unsigned* sums, unsigned* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned inc = v;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const unsigned a = __shfl_up_sync(0xffffffffu, inc, off);
    if (lane >= off) inc += a;
  }
  __syncthreads();
  if (lane == 31) sums[warp] = inc;
  __syncthreads();
  const unsigned w = lane < kBPlanThreads / 32 ? sums[lane] : 0u;
  *total = __reduce_add_sync(0xffffffffu, w);
  return __reduce_add_sync(0xffffffffu, lane < warp ? w : 0u) + inc - v;
}
// Block 0 plans; block 1 + t, with gated shared experts, works out token t's gate.
__global__ void __launch_bounds__(kBPlanThreads) batch_plan_kernel(const BPlanParams p) {
  __shared__ int s_e[kBPlanThreads];
  __shared__ unsigned s_high[kBPlanThreads], s_index[kBPlanThreads], s_prefix[kBPlanThreads], s_sums[32];
  __shared__ uint8_t s_tok[kBPlanThreads][kBRun];
  const int tid = threadIdx.x, lane = tid & 31;
  b_dep_launch();
  b_dep_wait();
  if (blockIdx.x > 0) {  // sigmoid(gate_vec . x[t])
    const int t = blockIdx.x - 1;
    float dot = 0.f;
    for (int i = tid; i < p.hidden / 2; i += kBPlanThreads) {
      const uint32_t raw = *reinterpret_cast<const uint32_t*>(p.x + (size_t)t * p.hidden + 2 * i);
      dot = fmaf(p.gate_vec[2 * i], __uint_as_float(raw << 16), dot);
      dot = fmaf(p.gate_vec[2 * i + 1], __uint_as_float(raw & 0xffff0000u), dot);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, off);
    float* part = reinterpret_cast<float*>(s_sums);
    if (lane == 0) part[tid >> 5] = dot;
    __syncthreads();
    if (tid == 0) {
      float sum = 0.f;
      for (int w = 0; w < kBPlanThreads / 32; ++w) sum += part[w];
      p.gate[t] = 1.f / (1.f + expf(-sum));
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
  const int planes = lead && s_high[tid] ? 2 : 1;
  const unsigned u1 = b_cost1(planes, p.hidden);
  unsigned c2 = 0;
  if (lead)
    for (int kc = 0; kc < p.kc_r; ++kc) c2 += b_cost2(planes, b_chunk_cols(p.inter, kc)) * (p.hidden / 16);
  unsigned n_runs, n_pairs, t1, t2;
  const unsigned index = b_scan(lead ? 1u : 0u, s_sums, &n_runs);
  const unsigned prefix = b_scan((unsigned)n, s_sums, &n_pairs);
  const unsigned start1 = b_scan(lead ? u1 * (p.inter / 16) : 0u, s_sums, &t1);
  unsigned start2 = b_scan(c2, s_sums, &t2);
  if (lead) {
    BRun r;
    r.expert = e;
    r.n = n;
    r.high = s_high[tid];
    r.inter = p.inter;
    r.hoff = (int)prefix * p.inter;
    r.pad_ = 0;
    for (int i = 0; i < kBRun; ++i) r.tok[i] = i < n ? s_tok[tid][i] : s_tok[tid][0];
    p.runs[index] = r;
    BSeg g;
    g.pad_[0] = g.pad_[1] = 0;
    g.run = (int)index;
    g.kc = 0;
    g.start = start1;
    g.ucost = u1;
    g.units = p.inter / 16;
    g.yrow = 0;
    p.seg1[index] = g;
    g.units = p.hidden / 16;
    for (int kc = 0; kc < p.kc_r; ++kc) {
      g.kc = kc;
      g.start = start2;
      g.ucost = b_cost2(planes, b_chunk_cols(p.inter, kc));
      g.yrow = (int)prefix * p.kc_r + kc * n;
      p.seg2[index * p.kc_r + kc] = g;
      start2 += g.ucost * (p.hidden / 16);
    }
    s_index[tid] = (unsigned)n;
    s_prefix[tid] = prefix;
  }
  __syncthreads();
  if (tid < npairs)
    p.pos[(tid / p.k) * slots + tid % p.k] =
        valid ? make_int2((int)s_prefix[leader] * p.kc_r + (rank & (kBRun - 1)), (int)s_index[leader]) : make_int2(-1, 0);
  // shared experts: all tokens, both slices
  const int parts = (p.T + kBRun - 1) / kBRun;
  const unsigned us1 = b_cost1(2, p.hidden);
  unsigned cs2 = 0;
  for (int kc = 0; kc < p.kc_s; ++kc) cs2 += b_cost2(2, b_chunk_cols(p.shared_inter, kc)) * (p.hidden / 16);
  const int n_sh = p.n_shared * parts;
  if (tid < n_sh) {
    const int j = tid / parts, part = tid % parts, t0 = part * kBRun, ns = min(kBRun, p.T - t0);
    const int before = j * p.T + t0;  // pairs of shared experts before this run
    BRun r;
    r.expert = p.n_experts + j;
    r.n = ns;
    r.high = 0xffu;
    r.inter = p.shared_inter;
    r.hoff = npairs * p.inter + before * p.shared_inter;
    r.pad_ = 0;
    for (int i = 0; i < kBRun; ++i) r.tok[i] = (uint8_t)(t0 + (i < ns ? i : 0));
    const int idx = (int)n_runs + tid;
    p.runs[idx] = r;
    BSeg g;
    g.pad_[0] = g.pad_[1] = 0;
    g.run = idx;
    g.kc = 0;
    g.start = t1 + (unsigned)tid * us1 * (p.shared_inter / 16);
    g.ucost = us1;
    g.units = p.shared_inter / 16;
    g.yrow = 0;
    p.seg1[idx] = g;
    unsigned st = t2 + (unsigned)tid * cs2;
    g.units = p.hidden / 16;
    for (int kc = 0; kc < p.kc_s; ++kc) {
      g.kc = kc;
      g.start = st;
      g.ucost = b_cost2(2, b_chunk_cols(p.shared_inter, kc));
      g.yrow = npairs * p.kc_r + before * p.kc_s + kc * ns;
      p.seg2[n_runs * p.kc_r + tid * p.kc_s + kc] = g;
      st += g.ucost * (p.hidden / 16);
    }
  }
  for (int i = tid; i < p.T * p.n_shared; i += kBPlanThreads) {
    const int t = i / p.n_shared, j = i % p.n_shared, t0 = t / kBRun * kBRun, ns = min(kBRun, p.T - t0);
    p.pos[t * slots + p.k + j] = make_int2(npairs * p.kc_r + (j * p.T + t0) * p.kc_s + (t - t0), ns);
  }
  if (tid == 0) {
    BHead h;
    h.nseg[0] = off ? 0 : (int)n_runs + n_sh;
    h.nseg[1] = off ? 0 : (int)n_runs * p.kc_r + n_sh * p.kc_s;
    h.total[0] = t1 + (unsigned)n_sh * us1 * (p.n_shared ? p.shared_inter / 16 : 0);
    h.total[1] = t2 + (unsigned)n_sh * cs2;
    h.off = off ? 1 : 0;
    *p.head = h;
    if (off) atomicOr(p.ctl.status, (unsigned)SLICEMOE_STATUS_WAIT_TIMEOUT);
  }
}

// ---- the projections --------------------------------------------------------------------------------------
struct BShare {  // a part of a CTA's share: row blocks first .. last - 1 of a segment
  const uint8_t* ptr[2][4];  // [gate, up / down][MSB, LSB, scales, zero-points]
  int first, last;
  int n;
  unsigned high;
  int inter, hoff, yrow;
  int kb0, nkb, row_kb;      // first 128-column block, their number, blocks of a whole row
  int lsb;                   // some pair uses both slices
  uint8_t tok[kBRun];
};
struct BParams {
  const slicemoe_expert* experts;
  const slicemoe_expert* shared;
  const uint16_t* x;
  const BHead* head;
  const BRun* runs;
  const BSeg* segs;
  float* h;
  float* yrow;
  BatchControl ctl;
  int n_experts, hidden, K, shift;  // K: widest vector of digits (hidden, or a chunk of the intermediate width)
  int stages;                       // per group
};
template <int G, int PHASE>
struct BSmem {
  static constexpr int kMeta = 8 * (128 / G) * 48;         // scales, then zero-points, of up to 8 blocks
  static constexpr int kStage = kBPlane + kMeta;
  static constexpr int kMats = PHASE == 1 ? 2 : 1;
  static constexpr int kPart = kBGroupWarps * kMats * kBRun * 20;  // floats: [warp][matrix][token][16 rows, padded]
  static constexpr int shares = 0;
  static constexpr int ctl = shares + kBMaxSegs * (int)sizeof(BShare);  // number of shares, dead flag, wait limit
  static constexpr int bars = ctl + 32;
  static constexpr int kMaxStages = 8;
  static constexpr int part = (bars + 2 * kBGroups * kMaxStages * 8 + 127) & ~127;
  static constexpr int dig = part + kBGroups * 2 * kPart * 4;
  __host__ __device__ static int tok_stride(int K) { return 3 * K + 32; }  // eight tokens' digit rows spread over the banks
  __host__ __device__ static int sums(int K) { return dig + kBRun * tok_stride(K); }            // float [K / G][8]
  __host__ __device__ static int inv(int K) { return sums(K) + K / G * kBRun * 4; }             // float [K / 128][8]
  __host__ __device__ static int ring(int K) { return (inv(K) + K / 128 * kBRun * 4 + 127) & ~127; }
};
static_assert(sizeof(BShare) % 8 == 0, "alignment");

struct BWait {
  volatile int* dead;
  unsigned long long limit;
  unsigned* status;
  // true: the phase is there; false: it is not, and nobody waits any more
  __device__ __forceinline__ bool operator()(uint32_t bar, uint32_t parity) const {
    if (mbar_try(bar, parity)) return true;
    const long long t0 = clock64();
    for (;;) {
      for (int i = 0; i < 64; ++i)
        if (mbar_try(bar, parity)) return true;
      if (*dead) return false;
      if ((unsigned long long)(clock64() - t0) > limit) {
        *dead = 1;
        atomicOr(status, (unsigned)SLICEMOE_STATUS_WAIT_TIMEOUT);
        return false;
      }
    }
  }
};

// One 16 x 128 block for eight tokens: acc[2 row half + token] += the block's contribution (lane (g, c): rows g and
// g + 8, tokens 2 c and 2 c + 1).  As in the batch-1 kernel the A fragment of rows g + 8 is the bytes as they are, 16 x
// their nibble plus row g's: the difference of the accumulator rows is 16 C[g + 8], and the row's scale is divided by 16.
template <int G, bool LSB>
__device__ __forceinline__ void b_block(const uint8_t* msb, const uint8_t* lsb, const uint8_t* sc, const uint8_t* zp, const uint8_t* dig,
                                        const float* X, const float* inv, int shift, unsigned low0, unsigned low1, float (&acc)[4]) {
  constexpr int SG = 128 / G, KS = G / 32;
  constexpr uint32_t kLow = 0x0f0f0f0fu;
  uint32_t a[2][8];  // [plane][words of the lane: 16 columns each]
  {
    const uint4 v0 = *reinterpret_cast<const uint4*>(msb), v1 = *reinterpret_cast<const uint4*>(msb + 512);
    a[0][0] = v0.x; a[0][1] = v0.y; a[0][2] = v0.z; a[0][3] = v0.w;
    a[0][4] = v1.x; a[0][5] = v1.y; a[0][6] = v1.z; a[0][7] = v1.w;
  }
  if (LSB) {
    const uint4 v0 = *reinterpret_cast<const uint4*>(lsb), v1 = *reinterpret_cast<const uint4*>(lsb + 512);
    a[1][0] = v0.x; a[1][1] = v0.y; a[1][2] = v0.z; a[1][3] = v0.w;
    a[1][4] = v1.x; a[1][5] = v1.y; a[1][6] = v1.z; a[1][7] = v1.w;
  }
  const float2 iv = *reinterpret_cast<const float2*>(inv);
#pragma unroll
  for (int sg = 0; sg < SG; ++sg) {
    float t[4];
#pragma unroll
    for (int d = 2; d >= 0; --d) {
      int m[4], l[4];
#pragma unroll
      for (int s = 0; s < KS; ++s) {
        const int ks = sg * KS + s;
        const uint2 b = *reinterpret_cast<const uint2*>(dig + ks * 96 + d * 32);
        const uint32_t w0 = a[0][2 * ks], w1 = a[0][2 * ks + 1];
        if (s == 0) mma_u8s8_first(m, w0 & kLow, w0, w1 & kLow, w1, b.x, b.y);
        else mma_u8s8(m, w0 & kLow, w0, w1 & kLow, w1, b.x, b.y);
        if (LSB) {
          const uint32_t u0 = a[1][2 * ks], u1 = a[1][2 * ks + 1];
          if (s == 0) mma_u8s8_first(l, u0 & kLow, u0, u1 & kLow, u1, b.x, b.y);
          else mma_u8s8(l, u0 & kLow, u0, u1 & kLow, u1, b.x, b.y);
        }
      }
      m[2] -= m[0];
      m[3] -= m[1];
      if (LSB) {
        l[2] -= l[0];
        l[3] -= l[1];
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        int v = m[i] << shift;
        if (LSB) v += l[i] & ((i & 1) ? ~low1 : ~low0);
        t[i] = d == 2 ? (float)v : fmaf(t[i], 256.f, (float)v);
      }
    }
    const float2 xs = *reinterpret_cast<const float2*>(X + sg * kBRun);
    const float s0 = __half2float(*reinterpret_cast<const __half*>(sc + sg * 32));
    const float s1 = __half2float(*reinterpret_cast<const __half*>(sc + sg * 32 + 16)) * 0.0625f;
    const unsigned z0 = zp[sg * 16], z1 = zp[sg * 16 + 8];
    // MSB slice alone: 2^shift (zp >> shift)
    const unsigned drop = (1u << shift) - 1u;
    const float za = (float)(z0 & ~(low0 & drop)), zb = (float)(z0 & ~(low1 & drop));
    const float zc = (float)((z1 & ~(low0 & drop)) << 4), zd = (float)((z1 & ~(low1 & drop)) << 4);
    acc[0] = fmaf(s0 * iv.x, fmaf(-za, xs.x, t[0]), acc[0]);
    acc[1] = fmaf(s0 * iv.y, fmaf(-zb, xs.y, t[1]), acc[1]);
    acc[2] = fmaf(s1 * iv.x, fmaf(-zc, xs.x, t[2]), acc[2]);
    acc[3] = fmaf(s1 * iv.y, fmaf(-zd, xs.y, t[3]), acc[3]);
  }
}

template <int G, int PHASE>
__global__ void __launch_bounds__(kBThreads, 1) batch_ffn_kernel(const __grid_constant__ BParams p) {
  using S = BSmem<G, PHASE>;
  constexpr int SG = 128 / G;
  extern __shared__ __align__(128) uint8_t smem[];
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  BShare* shares = reinterpret_cast<BShare*>(smem + S::shares);
  int* n_shares = reinterpret_cast<int*>(smem + S::ctl);
  volatile int* dead = n_shares + 1;
  const uint32_t bars = smem_u32(smem + S::bars);
  if (tid == 0) {
    *dead = 0;
    for (int i = 0; i < kBGroups * p.stages; ++i) {
      mbar_init(bars + 16 * i, 1);                // full: the producer's arrive, and the bytes
      mbar_init(bars + 16 * i + 8, kBGroupWarps); // empty
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
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
  if (warp == 0) {
    // this CTA's share: the row blocks whose start, in cost, lies in its window
    const int nseg = __ldcg(&p.head->nseg[PHASE - 1]);
    const unsigned long long total = __ldcg(&p.head->total[PHASE - 1]);
    const unsigned lo = (unsigned)((total * blockIdx.x + gridDim.x - 1) / gridDim.x);
    const unsigned hi = (unsigned)((total * (blockIdx.x + 1) + gridDim.x - 1) / gridDim.x);
    int count = 0;
    for (int s0 = 0; s0 < nseg; s0 += 32) {
      int first = 0, last = 0;
      BSeg g{};
      if (s0 + lane < nseg) {
        const uint4* src = reinterpret_cast<const uint4*>(p.segs + s0 + lane);
        reinterpret_cast<uint4*>(&g)[0] = __ldcg(src);
        reinterpret_cast<uint4*>(&g)[1] = __ldcg(src + 1);
        auto ord = [&](unsigned at) { return at <= g.start ? 0 : (int)min((unsigned)g.units, (at - g.start + g.ucost - 1) / g.ucost); };
        first = ord(lo);
        last = ord(hi);
      }
      const unsigned has = __ballot_sync(0xffffffffu, last > first);
      const int at = count + __popc(has & ((1u << lane) - 1u));
      if (last > first && at < kBMaxSegs) {
        BRun r;
        const uint4* src = reinterpret_cast<const uint4*>(p.runs + g.run);
#pragma unroll
        for (int i = 0; i < (int)(sizeof(BRun) / 16); ++i) reinterpret_cast<uint4*>(&r)[i] = __ldcg(src + i);
        BShare& sh = shares[at];
        const slicemoe_expert* ex = r.expert >= p.n_experts ? p.shared + (r.expert - p.n_experts) : p.experts + r.expert;
        sh.lsb = r.high != 0u;
#pragma unroll
        for (int m = 0; m < S::kMats; ++m) {
          const slicemoe_mat* mat = PHASE == 1 ? (m ? &ex->up : &ex->gate) : &ex->down;
          sh.ptr[m][0] = reinterpret_cast<const uint8_t*>(mat->msb);
          sh.ptr[m][1] = reinterpret_cast<const uint8_t*>(mat->lsb);
          sh.ptr[m][2] = reinterpret_cast<const uint8_t*>(mat->scale);
          sh.ptr[m][3] = mat->zp;
          if (sh.lsb && !sh.ptr[m][1]) {  // both slices asked of an expert without LSB planes: defined garbage, reported
            sh.ptr[m][1] = sh.ptr[m][0];
            atomicOr(p.ctl.status, (unsigned)SLICEMOE_STATUS_MISSING_LSB);
          }
        }
        sh.first = first;
        sh.last = last;
        sh.n = r.n;
        sh.high = r.high;
        sh.inter = r.inter;
        sh.hoff = r.hoff;
        sh.yrow = g.yrow;
        sh.row_kb = (PHASE == 1 ? p.hidden : r.inter) >> 7;
        sh.kb0 = PHASE == 1 ? 0 : g.kc * (kBChunkK / 128);
        sh.nkb = PHASE == 1 ? sh.row_kb : b_chunk_cols(r.inter, g.kc) >> 7;
#pragma unroll
        for (int i = 0; i < kBRun; ++i) sh.tok[i] = r.tok[i];
      }
      count += __popc(has);
    }
    if (lane == 0) *n_shares = min(count, kBMaxSegs);
  }
  __syncthreads();
  const int ns = *n_shares;
  uint8_t* ring0 = smem + S::ring(p.K);

  if (warp >= kBConsumers) {
    // ---- producer of a group: lane 0 the MSB plane, 1 the LSB plane, 2 the scales, 3 the zero-points ----
    if (lane >= 4) return;
    const int group = warp - kBConsumers;
    const uint32_t fb = bars + 16 * group * p.stages;
    const uint32_t ring = smem_u32(ring0 + (size_t)group * p.stages * S::kStage);
    const uint64_t pol = l2_evict_first_policy();
    const unsigned per_block = lane < 2 ? 1024u : (lane == 2 ? SG * 32u : SG * 16u);
    int st = 0, ord = 0;
    uint32_t par = 1, used = 0;
    bool ok = true;
    for (int i = 0; i < ns && ok; ++i) {
      const BShare& sh = shares[i];
      const int nkb = sh.nkb, per = sh.lsb ? 4 : 8;
      const bool active = lane != 1 || sh.lsb;
      const unsigned dst0 = lane == 0 ? 0u : lane == 1 ? kBPlane / 2 : lane == 2 ? kBPlane : kBPlane + 8 * SG * 32;
      // the group's row blocks: every kBGroups-th of the share
      for (int u = sh.first + ((group - ord) & (kBGroups - 1)); u < sh.last && ok; u += kBGroups) {
#pragma unroll 1
        for (int m = 0; m < S::kMats && ok; ++m) {
          const uint8_t* src = sh.ptr[m][lane] + ((size_t)u * sh.row_kb + sh.kb0) * per_block;
          for (int b0 = 0; b0 < nkb; b0 += per) {
            const unsigned nb = (unsigned)min(per, nkb - b0);
            if (!wait(fb + 16 * st + 8, par)) { ok = false; break; }
            if (lane == 0) mbar_arrive_expect_tx(fb + 16 * st, nb * ((sh.lsb ? 2048u : 1024u) + SG * 48u));
            __syncwarp(0xfu);
            if (active) bulk_g2s(ring + st * S::kStage + dst0, src, nb * per_block, fb + 16 * st, pol);
            src += nb * per_block;
            ++used;
            if (++st == p.stages) { st = 0; par ^= 1; }
          }
        }
      }
      ord += sh.last - sh.first;
    }
    // no copy may be on its way when the CTA ends (in the normal case the consumers have seen them all land)
    for (uint32_t i = used > (uint32_t)p.stages ? used - p.stages : 0; i < used; ++i) {
      const long long t0 = clock64();
      while (!mbar_try(fb + 16 * (i % p.stages), (i / p.stages) & 1) && (unsigned long long)(clock64() - t0) < wait.limit) {}
    }
    return;
  }

  // ---- consumers ----
  const int group = warp / kBGroupWarps, gw = warp % kBGroupWarps, g8 = lane >> 2, c = lane & 3;
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
  int st = 0, ord = 0, half = 0;
  uint32_t par = 0;
  for (int i = 0; i < ns; ++i) {
    const BShare& sh = shares[i];
    const int n = sh.n, nkb = sh.nkb;
    if (i > 0) asm volatile("bar.sync 1, %0;" ::"n"(32 * kBConsumers) : "memory");  // the digits of the run before have been used
    for (int blk = warp; blk < n * nkb; blk += kBConsumers) {
      const int t = blk / nkb, b = blk - t * nkb;
      float v[4];
      if (PHASE == 1) {
        const uint2 raw = *reinterpret_cast<const uint2*>(p.x + (size_t)sh.tok[t] * p.hidden + b * 128 + 4 * lane);
        v[0] = __uint_as_float(raw.x << 16);
        v[1] = __uint_as_float(raw.x & 0xffff0000u);
        v[2] = __uint_as_float(raw.y << 16);
        v[3] = __uint_as_float(raw.y & 0xffff0000u);
      } else {
        const float4 raw = __ldcg(reinterpret_cast<const float4*>(p.h + sh.hoff + (size_t)t * sh.inter + (sh.kb0 + b) * 128) + lane);
        v[0] = raw.x; v[1] = raw.y; v[2] = raw.z; v[3] = raw.w;
      }
      const BlockDigits d = block_digits(v);
      store_digits(d, b * 128 + 4 * lane, dig + t * stride);
      int s0, s1, s2;
      group_digit_sums<G>(d, lane, s0, s1, s2);
      if ((lane & (G / 4 - 1)) == 0)
        X[(b * SG + lane / (G / 4)) * kBRun + t] = fmaf(65536.f, (float)s2, fmaf(256.f, (float)s1, (float)s0));
      if (lane == 0) inv[b * kBRun + t] = d.inv;
    }
    asm volatile("bar.sync 1, %0;" ::"n"(32 * kBConsumers) : "memory");
    const unsigned low0 = (sh.high >> (2 * c)) & 1u ? 0u : 0xffffffffu, low1 = (sh.high >> (2 * c + 1)) & 1u ? 0u : 0xffffffffu;
    const bool lsb = sh.lsb != 0;
    const int per = lsb ? 4 : 8;
    const uint8_t* my_dig = dig + min(g8, n - 1) * stride + c * 8;  // columns without a token repeat the last one's
    for (int u = sh.first + ((group - ord) & (kBGroups - 1)); u < sh.last; u += kBGroups) {
      float* pb = part + half * S::kPart;
#pragma unroll 1
      for (int m = 0; m < S::kMats; ++m) {
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        for (int b0 = 0; b0 < nkb; b0 += per) {
          wait(fb + 16 * st, par);
          const uint8_t* stage = ring + st * S::kStage;
          const int nb = min(per, nkb - b0);
          for (int b = gw; b < nb; b += kBGroupWarps) {
            const uint8_t* sc = stage + kBPlane + b * (SG * 32) + g8 * 2;
            const uint8_t* zp = stage + kBPlane + 8 * SG * 32 + b * (SG * 16) + g8;
            const uint8_t* dg = my_dig + (b0 + b) * 384;
            const float* xp = X + (b0 + b) * SG * kBRun + 2 * c;
            const float* ip = inv + (b0 + b) * kBRun + 2 * c;
            const uint8_t* ap = stage + b * 1024 + lane * 16;
            if (lsb) b_block<G, true>(ap, ap + kBPlane / 2, sc, zp, dg, xp, ip, p.shift, low0, low1, acc);
            else b_block<G, false>(ap, nullptr, sc, zp, dg, xp, ip, p.shift, 0xffffffffu, 0xffffffffu, acc);
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(fb + 16 * st + 8);
          if (++st == p.stages) { st = 0; par ^= 1; }
        }
        float* w = pb + (gw * S::kMats + m) * (kBRun * 20);
        w[(2 * c) * 20 + g8] = acc[0];
        w[(2 * c + 1) * 20 + g8] = acc[1];
        w[(2 * c) * 20 + g8 + 8] = acc[2];
        w[(2 * c + 1) * 20 + g8 + 8] = acc[3];
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
    ord += sh.last - sh.first;
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
  if (col >= p.hidden || p.head->off) return;
  float2 a = make_float2(0.f, 0.f);
  const float gate = p.gate ? p.gate[t] : 1.f;
#pragma unroll 4
  for (int j = 0; j < slots; ++j) {
    const int2 at = p.pos[t * slots + j];
    if (at.x < 0) continue;
    const float w = j < p.k ? p.weights[t * p.k + j] : gate;
    const int kc_n = j < p.k ? p.kc_r : p.kc_s;
    float2 v = __ldcg(reinterpret_cast<const float2*>(p.yrow + (size_t)at.x * p.hidden + col));
    for (int kc = 1; kc < kc_n; ++kc) {
      const float2 u = __ldcg(reinterpret_cast<const float2*>(p.yrow + (size_t)(at.x + kc * at.y) * p.hidden + col));
      v.x += u.x;
      v.y += u.y;
    }
    a.x = fmaf(w, v.x, a.x);
    a.y = fmaf(w, v.y, a.y);
  }
  *reinterpret_cast<float2*>(p.y + (size_t)t * p.hidden + col) = a;
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
  // as many stages as shared memory holds: bytes in flight are what the bandwidth needs
  p.stages = (kBSmemMax - S::ring(p.K)) / (kBGroups * S::kStage);
  if (p.stages > S::kMaxStages) p.stages = S::kMaxStages;
  return b_launch(batch_ffn_kernel<G, PHASE>, dim3((unsigned)sms), kBThreads,
                  (size_t)S::ring(p.K) + (size_t)kBGroups * p.stages * S::kStage, st, p);
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
  pp.runs = reinterpret_cast<BRun*>(ws + L.runs);
  pp.seg1 = reinterpret_cast<BSeg*>(ws + L.seg1);
  pp.seg2 = reinterpret_cast<BSeg*>(ws + L.seg2);
  pp.pos = reinterpret_cast<int2*>(ws + L.pos);
  pp.gate = reinterpret_cast<float*>(ws + L.gate);
  pp.ctl = ctl;
  int rc = b_launch(batch_plan_kernel, dim3(gated ? 1 + T : 1), kBPlanThreads, 0, st, pp);
  if (rc != SLICEMOE_OK) return rc;
  BParams p;
  p.experts = experts;
  p.shared = shared;
  p.x = x;
  p.head = pp.head;
  p.runs = pp.runs;
  p.segs = pp.seg1;
  p.h = reinterpret_cast<float*>(ws + L.h);
  p.yrow = reinterpret_cast<float*>(ws + L.yrow);
  p.ctl = ctl;
  p.n_experts = s->n_experts;
  p.hidden = s->hidden;
  p.K = s->hidden;
  p.shift = s->b_high - s->b_low;
  p.stages = 0;
  BParams p2 = p;
  p2.segs = pp.seg2;
  const int widest = s->inter > pp.shared_inter ? s->inter : pp.shared_inter;
  p2.K = widest < kBChunkK ? widest : kBChunkK;
  if (s->group == 128) {
    rc = b_launch_ffn<128, 1>(p, sms, st);
    if (rc == SLICEMOE_OK) rc = b_launch_ffn<128, 2>(p2, sms, st);
  } else if (s->group == 64) {
    rc = b_launch_ffn<64, 1>(p, sms, st);
    if (rc == SLICEMOE_OK) rc = b_launch_ffn<64, 2>(p2, sms, st);
  } else {
    rc = b_launch_ffn<32, 1>(p, sms, st);
    if (rc == SLICEMOE_OK) rc = b_launch_ffn<32, 2>(p2, sms, st);
  }
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
