// Batch-1 decode of one MoE layer from bit-sliced AMAT weights (Section 4.1 of the paper: an expert
// runs from MSB+LSB slices at full precision or from the MSB slice alone), as ONE persistent kernel.
//
// The work is a pure weight stream: every plane byte is used once, so the bound is HBM bandwidth and
// everything else is arranged so that the stream never stops.
//   * One CTA per SM: 16 consumer warps in 4 groups, one epilogue warp, two producer warps (6 lanes each,
//     one per bulk copy of a chunk) and a warp that requests the down tiles.  The 4 warps of a group split a chunk's 128-column blocks, so the
//     per-chunk bookkeeping is paid by 4 warps, not 16, while 4 chunks are in work at any time.  The
//     schedule is a pure function of the slot table, so every role enumerates it for itself and only
//     data and barrier phases pass between them.  The producer streams chunks - 16 rows x <=2048 columns: the MSB plane tile,
//     the LSB plane tile when the expert runs at 8 bits (<=16 KB each, one contiguous run thanks to the
//     tiled layout), scales and zero-points - into a ring of eight 19 KB units with cp.async.bulk +
//     mbarriers.  Nobody waits for the gate/up -> down dependency to request tiles, so down-projection tiles are
//     already in flight (up to the whole ring) while the grid exchanges h.
//   * Integer arithmetic on the tensor pipe.  The activation vector (x, later h) is converted once,
//     per 128-element block, to fixed point relative to the block's largest magnitude and split into
//     three balanced base-256 digits (int8).  The digits sit in separate columns of the B operand of
//     mma.sync m16n8k32 (u8 x s8 -> s32); the A operand is the raw nibble plane: the layout stores
//     the two row halves of a fragment in the low and high nibbles of each byte, so `w & 0x0f0f0f0f`
//     and `w` itself are the whole unpack (the second half then carries 16 x its rows plus the first
//     half's, which one subtraction and the fold weight undo).  Sums are exact in int32; MSB and LSB planes combine as
//     16 * Cm + Cl.  Scale and zero-point are applied once per (row, group):
//        sum_k x_k s (q_k - zp) = s (sum_k q_k x_k - zp sum_{k in group} x_k).
//     The plain ALUs could not unpack + convert + FMA two weights per byte at HBM rate; this costs
//     about seven instructions per 512 weights.
//   * Phase 1 (gate/up + SwiGLU): tasks are (expert slot, 16-row block), dealt to the CTAs one by one in slot order, so that h is
//     complete slot after slot and part of it is in digits before the last of it is written.  (A window of consecutive
//     tasks per CTA - all slots complete at the end - and all of h converted then: a launch of a 2048-wide layer of 1408-wide
//     experts, top-6 + 2 shared, 16.4 us; dealt, with the warp that requests the down tiles at once: 15.8; with a gated shared
//     expert of 5632, 18.5 / 16.1; 1024-wide, top-8 of 512, 11.1 / 9.6; 256-wide, 6.45 / 5.9.)  The epilogue warp adds the warps' partial rows, applies SwiGLU and writes h (fp32) to
//     the workspace.  There is no barrier between the phases: readers poll the h words themselves (two
//     buffers used by alternate launches, each left "empty" by the launch before; every wait bounded).
//   * Phase 2 (down + weighted combine): a task is a 16-row block of the OUTPUT over ALL slots, so
//     the top-k combine stays inside the CTA: no atomics, no cross-CTA reduction, fixed summation
//     order (results are bit-reproducible).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "batch.cuh"
#include "common.cuh"
#include "decode_common.cuh"
#include "decode_schedule.cuh"
#include "route.cuh"

namespace slicemoe {

constexpr int kConsumerWarps = 16;
// kGroups consumer groups: a phase-1 task belongs to one group, phase-2 chunks go round-robin
constexpr int kGroupWarps = 4;   // warps of a group; they split the 128-column blocks of the chunk
static_assert(kGroups * kGroupWarps == kConsumerWarps, "groups");
constexpr int kEpilogueWarp = kConsumerWarps;
constexpr int kProducerWarp = kConsumerWarps + 1;  // first of kProducers producer warps
constexpr int kDownWarp = kProducerWarp + kProducers;  // fetches the routed experts' pointers, then requests the down tiles
constexpr int kThreads = 32 * (kDownWarp + 1);
constexpr int kUnits2 = 16;                        // at most this many (smaller) units in phase 2
constexpr int kFull2PerGroup = 8;  // >= chunks that a group can have in flight in phase 2 (of kUnits2 units)
constexpr int kUnits = 8;                                 // ring units; a chunk takes one per plane
constexpr int kChunkK = 2048;                             // K columns per chunk (16 blocks of 128)
constexpr int kBlocksPerWarp = kChunkK / 128 / kGroupWarps;
constexpr int kPlaneUnitBytes = 16 * kChunkK / 2;         // 16384
constexpr int kScaleUnitBytes = 16 * (kChunkK / 32) * 2;  // 2048 (group 32 is the worst case)
constexpr int kZpUnitBytes = 16 * (kChunkK / 32);         // 1024
constexpr int kUnitBytes = kPlaneUnitBytes + kScaleUnitBytes + kZpUnitBytes;  // 19456
constexpr int kMaxSlots = SLICEMOE_MAX_TOP_K + SLICEMOE_MAX_SHARED;
constexpr int kMaxHidden = 4096;
constexpr int kHCap = 12288;  // sum of intermediate widths over all slots of a layer
constexpr int kMaxMine = 32;   // phase-2 chunks one consumer group can have: (slots + kHCap / kChunkK) chunks per
                               // output row block, at most 4 row blocks per CTA, shared by 4 groups

// ---- optional time stamps ------------------------------------------------------------------------
// A build with -DSLICEMOE_TRACE records, per CTA and for the most recent launch, when its roles passed a few
// points: clock64 relative to the CTA's start (and the global timer at three of them).  slicemoe_trace_read hands
// the table out; `python -m paper_2512_12990_b200.trace` prints the timeline.  The ordinary build has none of it.
#ifdef SLICEMOE_TRACE
constexpr int kTraceSlots = 48;
__device__ long long g_trace[256][kTraceSlots];
__shared__ long long s_trace_t0;
__device__ __forceinline__ long long trace_gtime() {
  long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
#define SM_TRACE(i)                                                                   \
  do {                                                                                \
    if ((threadIdx.x & 31) == 0 && blockIdx.x < 256) g_trace[blockIdx.x][i] = clock64() - s_trace_t0; \
  } while (0)
#define SM_TRACE_G(i)                                                                 \
  do {                                                                                \
    if ((threadIdx.x & 31) == 0 && blockIdx.x < 256) g_trace[blockIdx.x][i] = trace_gtime(); \
  } while (0)
#else
#define SM_TRACE(i) do { } while (0)
#define SM_TRACE_G(i) do { } while (0)
#endif
// stamp numbers (clock64 unless noted): 1 dependency wait over, 2 plan built, 3 x as digits (warp 3),
// 4 prologue barrier passed, 5-8 gate/up phase done (consumer groups 0-3), 9 list of down chunks built (warp 0),
// 10 no block of h left to take on (warp 0), 11 down phase done (warp 0), 12 last h value written, 13 y written;
// 14-17 no block of h left (first warp of consumer groups 0-3), 23-26 the h blocks of the group's last down chunk
// flagged, 27-30 down phase done (first warp of groups 0-3), 31 the request of the down tiles begins, 18 all down tiles
// requested, 32-39 producer 0 has requested its gate/up chunk 0-7; global timer: 20 kernel entry, 21 dependency
// wait over, 22 y written

// ---- workspace --------------------------------------------------------------------------------
struct WsHeader {
  unsigned readers;     // CTAs of the running launch that have read `epoch` (the last one moves it on)
  unsigned epoch;       // launches so far on this workspace; its parity selects the h buffer
  unsigned status;      // SLICEMOE_STATUS_* bits
  unsigned extra_arrivals;         // != 0: h never counts as complete (slicemoe_workspace_set_wait; 0 in real use)
  unsigned long long wait_cycles;  // limit of the device-side waits, 0 = kWaitCycles
};
// The intermediate vector h crosses the grid through the workspace without a barrier: there are two buffers,
// used by alternate launches; a buffer's words all hold kHEmpty when its launch begins (the launch before
// wrote that, after the launch before it had read them; slicemoe_workspace_init writes both), a CTA stores its
// h values with plain stores, and a reader polls the words it needs until none of them is kHEmpty any more.
// kHEmpty is a NaN pattern that no arithmetic produces (the sign bit of a generated NaN is clear).
constexpr unsigned kHEmpty = 0xffffffffu;
constexpr size_t kWsHOff = 2048;                              // float h[2][kHCap]
constexpr size_t kWsStageOff = kWsHOff + 2 * sizeof(float) * kHCap;
// host-step staging: x bf16[kMaxHidden] | logits f32[512] | ids i32[16] | w f32[16] | prec u8[16] | y f32[kMaxHidden]
constexpr size_t kWsStX = kWsStageOff;
constexpr size_t kWsStLogits = kWsStX + 2 * kMaxHidden;
constexpr size_t kWsStIds = kWsStLogits + 4 * 512;
constexpr size_t kWsStW = kWsStIds + 64;
constexpr size_t kWsStPrec = kWsStW + 64;
constexpr size_t kWsStY = kWsStPrec + 64;
constexpr size_t kWsBytes = kWsStY + 4 * kMaxHidden;
// Behind that, in a workspace of slicemoe_workspace_bytes(): the batch kernels' part, then the lists of a pass that is
// routed here: ids i32, w f32, prec u8, [kBatchTokens][SLICEMOE_MAX_TOP_K] each.
constexpr size_t kWsBatchOff = (kWsBytes + 255) & ~(size_t)255;
constexpr size_t kWsListEntries = (size_t)kBatchTokens * SLICEMOE_MAX_TOP_K;
constexpr size_t kWsListBytes = kWsListEntries * 9;
// From this many tokens on a layer call takes the batch kernels (four launches) instead of a launch of the batch-1 kernel
// per token.  Measured, us, loop / batch at T = 4, 8 with tokens that share no expert until all are named: 2048-wide layer of
// 1408-wide experts 62 / 45, 123 / 60; 1024 wide 33 / 19, 66 / 23; 256 wide 24 / 14, 47 / 16; groups of 32, 2048 wide 82 / 51, 163 / 69.
// Of 30 shapes, widths 256 to 4096 and all groups, the batch was ahead from four tokens on at all but one: 4096 wide, groups
// of 32, four experts of 1408 a token 79.5 / 83.6 (T = 5 99 / 103, T = 8 159 / 134), where its ring has one stage a group.  By time
// alone the line would lie at three (the first three shapes, let in there: 47 / 40, 25 / 20, 18 / 14); it lies at four because
// slicemoe_layer_static, which has no room for the batch, gives the bits of slicemoe_layer up to three tokens, as its header says.
constexpr int kBatchMinTokens = 4;
static_assert(sizeof(WsHeader) <= kWsHOff, "workspace header");
static_assert(kWsStLogits + 4 * 512 <= kWsStIds, "x and the logits fit the staging area back to back too");

// ---- kernel parameters -------------------------------------------------------------------------
struct DecodeParams {
  const slicemoe_expert* experts;
  const slicemoe_expert* shared;
  const float* gate_vec;
  const uint16_t* x;
  const int32_t* ids;
  const uint8_t* prec;
  const float* weights;
  float* y;
  WsHeader* ws;
  float* ws_h;
  int n_experts, n_shared, k;
  int hidden, inter, shared_inter, group;
  int sigmoid_gate;
  int shift;  // b_high - b_low: the MSB slice is worth 2^shift of the LSB slice's units
  // the routing lists were complete before the work ahead of this kernel in the stream began: they are read, and
  // the routed experts' tiles requested, while that work is still running
  int lists_resident;
  // fused routing (logits != nullptr): the list is computed from the router logits in the prologue instead of
  // read from ids / prec / weights, and written to the *_out arrays (each may be null) by one CTA
  const float* logits;
  const float* bias;
  int renorm, rank_high;
  float tau;
  int32_t* ids_out;
  uint8_t* prec_out;
  float* weights_out;
};

struct Slot {
  const uint8_t* ptr[3][4];  // [gate, up, down][MSB plane, LSB plane, scales, zero-points]: slicemoe_expert's pointers
  int inter;
  int prec;
  float coef;
  int hoff;   // offset of this slot's h in the workspace / in the digit buffer
  int gated;  // 1: the combine weight is sigmoid(gate_vec . x)
  int pad_;
};

// The schedule of a CTA.
//   phase 1: tasks are 16-row blocks of gate and up, numbered slot after slot - shared, routed from both slices, routed from the
//     MSB slice alone - so that task o of the grid writes h[16 o ..].  Deal says which of them a CTA has.  How many tasks of the
//     shared experts a CTA has (count_s) follows from the shape alone, so their tiles are requested before the routing list is known.  A
//     both-slice task is 2 * nch chunks (gate then up; nch = 2048-column chunks of hidden), each two
//     units (MSB tile, LSB tile); an MSB-only task is nch chunks, each two units (the gate's MSB tile
//     and the up's).  Every phase-1 chunk takes two units.  Which producer and which group a task goes to says TaskPlace;
//     which units and barriers a chunk uses is stated at `struct Bars`.
//   phase 2: tasks m = 0 .. count2-1 are the output row blocks blockIdx.x + m * gridDim.x; each is one run of
//     chunks over the slots in order (p2c[j] chunks and p2u[j] units come before slot j), two units per
//     chunk for 8-bit slots and one for 4-bit slots.  Chunk number c is consumed by group c % kGroups.
//     Phase 2 re-cuts the ring into nunits2 units of unit2_bytes, just large enough for the widest down
//     chunk (plane area, then scales at scale2_off, zero-points at zp2_off), so that more - for the
//     benchmark shapes all - of the phase's tiles are in shared memory before h arrives.
struct Plan {
  int count_s;      // phase-1 tasks of this CTA of the shared experts
  Deal deal;        // its phase-1 tasks
  int hpar;         // which h buffer this launch uses
  int never_ready;  // the time-out exercise: treat h as never complete
  int count2;
  int nslots;
  int htotal;   // sum of the slots' intermediate widths
  int unit2_bytes, nunits2, scale2_off, zp2_off;
  short p2c[kMaxSlots + 1], p2u[kMaxSlots + 1];
};

struct SmemLayout {
  // offsets into dynamic shared memory
  static constexpr int ring = 0;
  static constexpr int hdig = ring + kUnits * kUnitBytes;    // int8 [kHCap/32][3 digits][32]
  static constexpr int xdig = hdig + kHCap * 3;              // int8 [kMaxHidden/32][3][32]
  static constexpr int hsumw = xdig + kMaxHidden * 3;        // float [kHCap/32][2]: weighted digit sums per group
  static constexpr int xsumw = hsumw + (kHCap / 32) * 8;     // float [kMaxHidden/32][2]
  static constexpr int hinv = xsumw + (kMaxHidden / 32) * 8;  // float [kHCap/128]: 2^-e of each 128-block of h
  static constexpr int xinv = hinv + (kHCap / 128) * 4;       // float [kMaxHidden/128]
  static constexpr int partial = xinv + (kMaxHidden / 128) * 4;  // float2 [warps][16]
  // float [warps][16], phase 2's, apart from phase 1's: the epilogue warp takes a CTA's tasks in order and may still be at another
  // group's when a group without a chunk in the first row block, and without a block of h to take on, writes its share of it.
  // (A wait for that instead cost 0.1 us a launch.)
  static constexpr int partial2 = partial + kConsumerWarps * 16 * 2 * 4;
  static constexpr int p2list = partial2 + kConsumerWarps * 16 * 4;  // uint4 [warps][kMaxMine]: a warp's phase-2 chunks
  static constexpr int slots = p2list + kConsumerWarps * kMaxMine * 16;
  static constexpr int plan = slots + kMaxSlots * (int)sizeof(Slot);
  static constexpr int bars = (plan + (int)sizeof(Plan) + 15) & ~15;  // uint64 barriers
  static constexpr int nbars = 2 * kUnits + kGroups * kFull2PerGroup + kUnits2 + 2 * kGroups + 5;
  static constexpr int dead = bars + nbars * 8;  // int dead flag; 8 bytes on, the wait limit in cycles
  static constexpr int hready = dead + 16;       // uint8 [kHCap / 128]: the 128-block of h is in shared memory as digits
  static constexpr int hnext = hready + kHCap / 128;  // int: the next block of h that nobody has taken on
  static constexpr int gate = hnext + 16;            // float [kMaxHidden / 128]: a block's share of gate_vec . x
  static constexpr int total = gate + kMaxHidden / 128 * 4;
};
static_assert(SmemLayout::total <= 227 * 1024, "shared memory budget");
static_assert(sizeof(Slot) % 8 == 0, "slot alignment");
static_assert(SmemLayout::slots % 8 == 0 && SmemLayout::hdig % 16 == 0 && SmemLayout::xdig % 16 == 0 &&
                  SmemLayout::plan % 8 == 0 && SmemLayout::partial % 8 == 0 && SmemLayout::partial2 % 4 == 0 && SmemLayout::p2list % 16 == 0,
              "alignment");

// Barriers.  Every barrier has ONE waiter that meets its phases strictly in order, so a parity wait can never
// be a phase off (mbarrier.try_wait.parity only tells the current phase from the one before it):
//   - a chunk's "full" barrier belongs to the consumer group that consumes it: group g's i-th chunk of a phase
//     uses full[g][i % 2] in phase 1, armed with the chunk's bytes by producer g % kProducers, and
//     full2[g][i % kFull2PerGroup] in phase 2, armed by the down warp;
//   - an "empty" barrier belongs to the warp that refills the space.  Phase 1: producer P owns half of the ring and
//     walks it in order: its j-th chunk takes the unit pair (4 P + 2 (j % 2), + 1) and waits on
//     empty[2 P + j % 2]; phase 2: the down warp takes the nunits2 units in running order, one
//     empty2 barrier per unit (an arrive from each warp of the group that consumed it).
// pfull1 / pempty1 per group (phase-1 partial rows to the epilogue warp and back), pfull2 / pempty2 (phase-2
// partial rows of all warps), p1_done (every consumer warp is through with phase 1, so the ring may be re-cut), plan_ready (the
// routed part of the plan and the routed slots stand: waited for after the shared experts' tasks), head_ready (what the workspace
// header says is in the plan).  The last two have one phase, and several waiters.
struct Bars {
  static constexpr int full = 0, empty = kUnits, full2 = 2 * kUnits, empty2 = full2 + kGroups * kFull2PerGroup,
                       pfull1 = empty2 + kUnits2,
                       pempty1 = pfull1 + kGroups, pfull2 = pempty1 + kGroups, pempty2 = pfull2 + 1, head_ready = pfull2 + 2,
                       p1_done = pfull2 + 3, plan_ready = pfull2 + 4, count = pfull2 + 5;
};

static_assert(Bars::count <= SmemLayout::nbars, "barrier storage");

// ---- fixed-point activations (see decode_common.cuh) ----------------------------------------------------
// One warp converts one 128-element block whose first element has index k0 in its vector: digits in B-fragment order,
// the weighted digit sums of every group of G elements (the zero-point term of the fold) and the block's 2^-e.
template <int G>
__device__ __forceinline__ void block_to_digits(const float (&v)[4], int k0, int lane, uint8_t* dig, float* sumw,
                                                float* inv) {
  const BlockDigits b = block_digits(v);
  const int k = k0 + 4 * lane;
  store_digits(b, k, dig);
  int s0, s1, s2;
  group_digit_sums<G>(b, lane, s0, s1, s2);
  if ((lane & (G / 4 - 1)) == 0) {
    sumw[(k / G) * 2 + 0] = (float)s0 + 256.f * (float)s1;
    sumw[(k / G) * 2 + 1] = 65536.f * (float)s2;
  }
  if (lane == 0) inv[k0 >> 7] = b.inv;
}

// ---- schedule enumeration (identical in every role) ----------------------------------------------------
__device__ __forceinline__ int nchunks_of(int K) { return (K + kChunkK - 1) / kChunkK; }
enum ChunkMode { kModeSingle = 0, kModeBoth = 1, kModePair = 2 };

// ---- consumers -----------------------------------------------------------------------------------
// Phase change: the consumer warps take 128-blocks of the grid's h on, a few at a time in order, poll them in the
// workspace until all of a block's values have been written (see kHEmpty), and turn the block into digits at once.  The tasks are
// dealt so that h is complete slot after slot, and a warp whose group is through with phase 1 early begins with the early slots.
// A block's flag in `hready` tells the other warps that its digits
// stand; nobody waits for the whole of h (see wait_h_blocks).  Returns false if the (bounded) wait ran out.
// (Four warps that did nothing else than this while gate/up ran took its issue slots: 20.8 -> 23.9 us where groups are 32 wide.
// Chunks that were ready consumed before more of h was taken on: 15.9 -> 17.0, a look at h is a trip of over a microsecond.)
template <int G>
__device__ bool fetch_h(const DecodeParams& p, uint8_t* smem, int lane, int htotal, const float* hbuf, bool never_ready,
                        volatile int* dead, unsigned* status) {
  const int nblk = htotal >> 7;
  // Loads in flight together, fewer where there would not be some for every warp.  The line lies where the digit sums of a block
  // begin to cost.  Four / two, us a launch, the layer alone: groups of 128, 2048-wide with two shared experts 15.67 / 15.95, with a
  // gated one of 5632 15.93 / 16.31, 1024-wide 9.58 / 9.47; groups of 64, 4096-wide 16.8 / 16.65 (experts of 1024), 29.85 / 29.83
  // (of 1408), 2048-wide 18.6 / 18.67, 1024-wide 11.05 / 10.73 (top-8 of 512), 19.78 / 19.85 (of 1408); groups of 32, 2048-wide
  // 22.4 / 21.64, 2688-wide 16.86 / 16.77.
  constexpr int kTake = G == 128 ? 4 : 2;
  const int take = max(1, min(kTake, nblk / kConsumerWarps));
  const long long t0 = clock64();
  for (;;) {
    int b0 = 0;
    if (lane == 0) b0 = atomicAdd(reinterpret_cast<int*>(smem + SmemLayout::hnext), take);
    b0 = __shfl_sync(0xffffffffu, b0, 0);
    if (b0 >= nblk) return true;
    unsigned pending = (1u << min(take, nblk - b0)) - 1u, before = 0u;  // warp-uniform
    while (pending != 0u) {
      if (pending == before) __nanosleep(100);  // (others are still at work on phase 1, whose way to memory this is, too)
      before = pending;
      float4 v[kTake];
#pragma unroll
      for (int i = 0; i < kTake; ++i)  // L2 is the point of coherence
        if ((pending >> i) & 1u) v[i] = __ldcg(reinterpret_cast<const float4*>(hbuf) + (b0 + i) * 32 + lane);
#pragma unroll
      for (int i = 0; i < kTake; ++i) {
        if ((pending >> i) & 1u) {
          const bool mine = __float_as_uint(v[i].x) != kHEmpty && __float_as_uint(v[i].y) != kHEmpty &&
                            __float_as_uint(v[i].z) != kHEmpty && __float_as_uint(v[i].w) != kHEmpty;
          if (__all_sync(0xffffffffu, mine) && !never_ready) {
            const float q[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
            block_to_digits<G>(q, (b0 + i) * 128, lane, smem + SmemLayout::hdig, reinterpret_cast<float*>(smem + SmemLayout::hsumw),
                               reinterpret_cast<float*>(smem + SmemLayout::hinv));
            pending &= ~(1u << i);
            __syncwarp();  // every lane's digits of the block are written ...
            if (lane == 0) {
              __threadfence_block();  // ... and visible before the flag is
              *reinterpret_cast<volatile uint8_t*>(smem + SmemLayout::hready + b0 + i) = 1;
            }
          }
        }
      }
      if (pending != 0u) {
        if (*dead) return false;
        if ((unsigned long long)(clock64() - t0) > wait_limit(dead)) {
          *dead = 1;
          atomicOr(status, (unsigned)SLICEMOE_STATUS_WAIT_TIMEOUT);
          return false;
        }
      }
    }
  }
}

// Waits (bounded) until the `n` (<= 32) 128-blocks of h from block `b0` on are in shared memory as digits.
__device__ __forceinline__ bool wait_h_blocks(const uint8_t* smem, int b0, int n, int lane, volatile int* dead,
                                              unsigned* status) {
  const volatile uint8_t* flag = reinterpret_cast<const volatile uint8_t*>(smem + SmemLayout::hready) + b0 + min(lane, n - 1);
  if (!__all_sync(0xffffffffu, *flag != 0)) {
    const long long t0 = clock64();
    while (!__all_sync(0xffffffffu, *flag != 0)) {
      if (*dead) return false;
      if ((unsigned long long)(clock64() - t0) > wait_limit(dead)) {
        *dead = 1;
        atomicOr(status, (unsigned)SLICEMOE_STATUS_WAIT_TIMEOUT);
        return false;
      }
    }
  }
  __threadfence_block();
  return true;
}

// Per-lane constants of the fold (see consume_chunk).
struct LaneRole {
  int c, r, cq, boff;
  float w0, w1;
};

// One chunk: this warp's 128-column blocks of the 16-row tile(s) in unit0 (and unit1).  The A operand is
// the nibble plane, the B operand the activation digits starting at `dig`; `sumw` / `binv` are the
// digits' weighted group sums and block scales for the same columns.
//   kModeSingle: MSB tile only           -> *out0 += 2^shift s (Cm - (zp >> shift) X)
//   kModeBoth:   MSB tile, LSB tile      -> *out0 += s (2^shift Cm + Cl - zp X)
// with shift = b_high - b_low (4 for 8-bit codes with 4-bit slices; a narrower slice sits in the low bits of its
// nibble, so the planes and everything below are the same for all widths)
//   kModePair:   two matrices' MSB tiles -> *out0 += first, *out1 += second (each with its own scales)
// Unpacking: a plane byte holds row g's nibble (low) and row g + 8's (high).  The fragment registers of
// row g are the bytes masked to their low nibble; those of row g + 8 are the bytes as they are, worth
// 16 * high + low, so that accumulator rows g + 8 come out as 16 * C[g + 8] + C[g] and one subtraction per
// folded value recovers 16 * C[g + 8] (the 16 goes into the lane's fold weight).  One AND per register pair.
// Lane roles: lanes with c in {0, 1} fold row g, lanes with c in {2, 3} row g + 8; even c holds digits 0
// and 1, odd c digit 2 (and the unused fourth column).  The caller adds the two digit halves (a shuffle
// with lane ^ 1) once per task.
template <int G>
__device__ __forceinline__ void pass_mma(int (&acc)[128 / G][4], const uint8_t* ap, const uint2& bv0, const uint2& bv1,
                                         const uint2& bv2, const uint2& bv3) {
  const uint4 wlo = *reinterpret_cast<const uint4*>(ap);
  const uint4 whi = *reinterpret_cast<const uint4*>(ap + 512);
  constexpr uint32_t kLow = 0x0f0f0f0fu;
  mma_u8s8_first(acc[0], wlo.x & kLow, wlo.x, wlo.y & kLow, wlo.y, bv0.x, bv0.y);
  if (G == 32) {
    mma_u8s8_first(acc[32 / G], wlo.z & kLow, wlo.z, wlo.w & kLow, wlo.w, bv1.x, bv1.y);
    mma_u8s8_first(acc[64 / G], whi.x & kLow, whi.x, whi.y & kLow, whi.y, bv2.x, bv2.y);
    mma_u8s8_first(acc[96 / G], whi.z & kLow, whi.z, whi.w & kLow, whi.w, bv3.x, bv3.y);
  } else if (G == 64) {
    mma_u8s8_first(acc[64 / G], whi.x & kLow, whi.x, whi.y & kLow, whi.y, bv2.x, bv2.y);
    mma_u8s8(acc[0], wlo.z & kLow, wlo.z, wlo.w & kLow, wlo.w, bv1.x, bv1.y);
    mma_u8s8(acc[64 / G], whi.z & kLow, whi.z, whi.w & kLow, whi.w, bv3.x, bv3.y);
  } else {
    mma_u8s8(acc[0], wlo.z & kLow, wlo.z, wlo.w & kLow, wlo.w, bv1.x, bv1.y);
    mma_u8s8(acc[0], whi.x & kLow, whi.x, whi.y & kLow, whi.y, bv2.x, bv2.y);
    mma_u8s8(acc[0], whi.z & kLow, whi.z, whi.w & kLow, whi.w, bv3.x, bv3.y);
  }
}

// (The mode is a template argument: with one body for down's two modes a 2048-wide layer took 15.8 us instead of 15.5, of groups of
// 32 21.1 instead of 20.3, 512-wide ones 15.8 instead of 14.95.)
// Blocks of two planes one after the other in a loop, not unrolled: another kernel between two launches - the routing - leaves fewer
// of this one's instructions in the caches, and a launch runs most of them once.  With the routing launch, unrolled / as a loop, us:
// 2048-wide, top-6 + 2 shared 18.15 / 17.43, gated shared expert 19.07 / 17.97, groups of 64 21.1 / 20.85, of 32 24.5 / 23.5;
// 4096-wide 18.75 / 18.4.  Where no other kernel comes between, the loop costs up to 0.9 % of some and saves others more: the layer
// alone 15.55 / 15.66, 15.85 / 15.92, 18.66 / 18.66, 21.42 / 21.64, 16.59 / 16.63 (2688-wide, groups of 32: 17.17 / 16.77), with resident
// lists 15.21 / 15.35, 15.87 / 15.96, 18.22 / 18.26, 21.29 / 21.29, 15.53 / 15.58 (16.37 / 15.91).
template <int G, int MODE>
__device__ __forceinline__ void consume_chunk(const LaneRole& lr, int lane, int gw, int rot, int nblocks,
                                              const uint8_t* unit0, const uint8_t* unit1, int scale_off, int zp_off,
                                              const uint8_t* dig, const float* sumw, const float* binv, float* out0,
                                              float* out1, int shift) {
  constexpr int SG = 128 / G;
  constexpr bool p8 = MODE == kModeBoth, pair = MODE == kModePair;
  const float pfix = p8 ? 1.f : (float)(1 << shift);
  const int zsh = p8 ? 0 : shift;
  const bool hi = (lr.c >> 1) != 0;
  float acc0 = 0.f, acc1 = 0.f;
#pragma unroll (MODE == kModeSingle ? kBlocksPerWarp : 1)
  for (int j = 0; j < kBlocksPerWarp; ++j) {
    const int b = (gw + kGroupWarps - rot) % kGroupWarps + kGroupWarps * j;  // 128-column block of the chunk
    if (b < nblocks) {
      const uint8_t* bp = dig + lr.boff + b * 384;
      const uint2 bv0 = *reinterpret_cast<const uint2*>(bp);
      const uint2 bv1 = *reinterpret_cast<const uint2*>(bp + 96);
      const uint2 bv2 = *reinterpret_cast<const uint2*>(bp + 192);
      const uint2 bv3 = *reinterpret_cast<const uint2*>(bp + 288);
      int m[SG][4], l[SG][4];
      pass_mma<G>(m, unit0 + b * 1024 + lane * 16, bv0, bv1, bv2, bv3);
      if (MODE != kModeSingle) pass_mma<G>(l, unit1 + b * 1024 + lane * 16, bv0, bv1, bv2, bv3);
      const float sfix = pfix * binv[b];
      const uint16_t* ms = reinterpret_cast<const uint16_t*>(unit0 + scale_off) + (b * SG) * 16 + lr.r;
      const uint8_t* mz = unit0 + zp_off + (b * SG) * 16 + lr.r;
#pragma unroll
      for (int sg = 0; sg < SG; ++sg) {
        // this lane's row (g, or 16 x row g + 8) and digit columns
        int ca = hi ? m[sg][2] - m[sg][0] : m[sg][0];
        int cb = hi ? m[sg][3] - m[sg][1] : m[sg][1];
        int ca1 = 0, cb1 = 0;
        if (MODE != kModeSingle) {
          ca1 = hi ? l[sg][2] - l[sg][0] : l[sg][0];
          cb1 = hi ? l[sg][3] - l[sg][1] : l[sg][1];
        }
        if (p8) {  // both slices: 2^shift Cm + Cl
          ca = (ca << shift) + ca1;
          cb = (cb << shift) + cb1;
        }
        const float x0 = sumw[(b * SG + sg) * 2 + lr.cq];
        {
          const float t = fmaf((float)cb, lr.w1, (float)ca * lr.w0);
          const float sc = __half2float(__ushort_as_half(ms[sg * 16])) * sfix;
          const float z = (float)((int)mz[sg * 16] >> zsh);
          // both slices: s (2^shift Cm + Cl - zp X); MSB only: 2^shift s (Cm - (zp >> shift) X)
          acc0 = fmaf(sc, fmaf(-z, x0, t), acc0);
        }
        if (pair) {  // the second matrix' scales / zero-points travel in the second unit
          const uint16_t* ms1 = reinterpret_cast<const uint16_t*>(unit1 + scale_off) + (b * SG) * 16 + lr.r;
          const uint8_t* mz1 = unit1 + zp_off + (b * SG) * 16 + lr.r;
          const float t = fmaf((float)cb1, lr.w1, (float)ca1 * lr.w0);
          const float sc = __half2float(__ushort_as_half(ms1[sg * 16])) * sfix;
          const float z = (float)((int)mz1[sg * 16] >> shift);  // pair chunks are MSB-only
          acc1 = fmaf(sc, fmaf(-z, x0, t), acc1);
        }
      }
    }
  }
  *out0 += acc0;
  *out1 += acc1;
}

template <int G>
__device__ void consumer_loop(const DecodeParams& p, uint8_t* smem, int warp, int lane) {
  constexpr int LG = G == 128 ? 7 : (G == 64 ? 6 : 5);
  const Slot* slots = reinterpret_cast<const Slot*>(smem + SmemLayout::slots);
  const Plan& plan = *reinterpret_cast<const Plan*>(smem + SmemLayout::plan);
  float2* partial = reinterpret_cast<float2*>(smem + SmemLayout::partial);
  float* partial2 = reinterpret_cast<float*>(smem + SmemLayout::partial2);
  volatile int* dead = reinterpret_cast<volatile int*>(smem + SmemLayout::dead);
  const uint32_t bars = smem_u32(smem + SmemLayout::bars);
  const uint32_t full0 = bars + 8 * Bars::full, empty0 = bars + 8 * Bars::empty;
  unsigned* status = &p.ws->status;
  const int group = warp / kGroupWarps, gw = warp % kGroupWarps;
  LaneRole lr;
  lr.c = lane & 3;
  const int g8 = lane >> 2;
  lr.r = g8 + 8 * (lr.c >> 1);
  lr.cq = lr.c & 1;
  const float rowfix = (lr.c >> 1) ? 0.0625f : 1.f;
  lr.w0 = (lr.cq ? 65536.f : 1.f) * rowfix;
  lr.w1 = (lr.cq ? 0.f : 256.f) * rowfix;
  // B column n = g8 takes digit n % 4; the fourth is unused, so those lanes re-read digit 0 and are ignored
  lr.boff = ((g8 & 3) == 3 ? 0 : (g8 & 3)) * 32 + lr.c * 8;

  // ---- phase 1: the tasks of this group ----
  const int nch = nchunks_of(p.hidden);
  const int prod = group % kProducers;  // the producer that serves this group
  {
    int cn = 0, end = plan.count_s;  // the shared experts' tasks are known from the start, the others once the plan stands
    int jp = 0;  // chunks of this group's producer so far (they fix the unit pair)
    int ig = 0;  // chunks of this group so far (they fix the full barrier)
    for (int n = 0;; ++n) {
      if (n == plan.count_s) {
        if (!mbar_wait(bars + 8 * Bars::plan_ready, 0, dead, status)) return;
        end = plan.deal.count1;
        if (plan.nslots == 0 && blockIdx.x == 0)
          for (int i = threadIdx.x; i < p.hidden; i += 32 * kConsumerWarps) p.y[i] = 0.f;
      }
      if (n >= end) break;
      const bool shared = n < plan.count_s, both = shared || n < plan.deal.count_both;
      const int nchunks = both ? 2 * nch : nch;
      const TaskPlace at(shared ? n + 1 : plan.deal.count_both, n);
      if (at.group() == group) {
        float part0 = 0.f, part1 = 0.f, unused = 0.f;
        for (int q = 0; q < nchunks; ++q, ++jp, ++ig) {
          const int c = cn + q;
          const int kc = q % nch;  // which 2048-column chunk of hidden
          if (!mbar_wait(full0 + 8 * (2 * group + (ig & 1)), (ig >> 1) & 1, dead, status)) return;
          const int u0 = 4 * prod + 2 * (jp & 1);
          const int nblocks = min(kChunkK, p.hidden - kc * kChunkK) >> 7;
          const uint8_t* dig = smem + SmemLayout::xdig + kc * (kChunkK * 3);
          const float* sumw = reinterpret_cast<const float*>(smem + SmemLayout::xsumw) + kc * (kChunkK >> LG) * 2;
          const float* binv = reinterpret_cast<const float*>(smem + SmemLayout::xinv) + kc * (kChunkK >> 7);
          const uint8_t* unit0 = smem + SmemLayout::ring + u0 * kUnitBytes;
          if (both) {
            consume_chunk<G, kModeBoth>(lr, lane, gw, c % kGroupWarps, nblocks, unit0, unit0 + kUnitBytes, kPlaneUnitBytes,
                             kPlaneUnitBytes + kScaleUnitBytes, dig, sumw, binv, q < nch ? &part0 : &part1, &unused, p.shift);
          } else {
            consume_chunk<G, kModePair>(lr, lane, gw, c % kGroupWarps, nblocks, unit0, unit0 + kUnitBytes, kPlaneUnitBytes,
                             kPlaneUnitBytes + kScaleUnitBytes, dig, sumw, binv, &part0, &part1, p.shift);
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(empty0 + 8 * (2 * prod + (jp & 1)));
        }
        // hand the four warps' shares of the K split to the epilogue warp
        part0 += __shfl_xor_sync(0xffffffffu, part0, 1);  // digits 0,1 (even c) + digit 2 (odd c)
        part1 += __shfl_xor_sync(0xffffffffu, part1, 1);
        const int round = at.round();
        if (!mbar_wait(bars + 8 * (Bars::pempty1 + group), (round & 1) ^ 1, dead, status)) return;
        if (lr.cq == 0) partial[warp * 16 + lr.r] = make_float2(part0, part1);
        __syncwarp();
        if (lane == 0) mbar_arrive(bars + 8 * (Bars::pfull1 + group));
      } else if (at.producer == prod) {
        jp += nchunks;  // the other group this producer serves
      }
      cn += nchunks;
    }
  }
  __syncwarp();
  if (gw == 0) SM_TRACE(5 + group);
  if (lane == 0) mbar_arrive(bars + 8 * Bars::p1_done);  // this warp no longer reads phase-1 units
  if (plan.count2 == 0) return;

  // ---- ahead of the phase change: list this group's phase-2 chunks (the walk over all output row
  // blocks, slots and chunks costs more than consuming the group's own chunks, so it is done ahead of time) ----
  uint4* mylist = reinterpret_cast<uint4*>(smem + SmemLayout::p2list) + warp * kMaxMine;
  int nmine = 0;
  {
    const int chunks2 = plan.p2c[plan.nslots];
    const int units = plan.nunits2;
    int u = 0;                                    // the next chunk's first unit
    for (int m = 0; m < plan.count2; ++m) {
      for (int j = 0; j < plan.nslots; ++j) {
        const int nchj = plan.p2c[j + 1] - plan.p2c[j];
        const Slot& sl = slots[j];
        const int wu = sl.prec ? 2 : 1;
        for (int kc = 0; kc < nchj; ++kc) {
          const int c = m * chunks2 + plan.p2c[j] + kc;  // chunk number within the phase
          const int u0 = u, u1 = u + 1 == units ? 0 : u + 1;
          u += wu;
          if (u >= units) u -= units;
          if (c % kGroups != group) continue;
          const int ig = c / kGroups;  // this group's ordinal of the chunk
          if (lane == 0 && nmine < kMaxMine) {
            // slot, row block, rotation of the warps | the chunk's units, full barrier, parity | 128-column blocks,
            // both slices? | first column of the chunk in h
            const int k0 = kc * kChunkK;
            mylist[nmine] = make_uint4((unsigned)j | (unsigned)m << 16 | (unsigned)(ig % kGroupWarps) << 24,
                                       (unsigned)u0 | (unsigned)u1 << 8 |
                                           (unsigned)(ig % kFull2PerGroup) << 16 | (unsigned)((ig / kFull2PerGroup) & 1) << 24,
                                       (unsigned)(min(kChunkK, sl.inter - k0) >> 7) | (sl.prec ? 256u : 0u),
                                       (unsigned)(sl.hoff + k0));
          }
          ++nmine;
        }
      }
    }
    nmine = min(nmine, kMaxMine);  // the host refuses launch shapes that could exceed the list
  }
  __syncwarp();
  if (warp == 0) SM_TRACE(9);

  // ---- the grid's h ----
  if (!mbar_wait(bars + 8 * Bars::head_ready, 0, dead, status)) return;
  if (!fetch_h<G>(p, smem, lane, plan.htotal, p.ws_h + (size_t)plan.hpar * kHCap, plan.never_ready != 0, dead, status)) return;
  if (warp == 0) SM_TRACE(10);
  if (gw == 0) SM_TRACE(14 + group);

  // ---- phase 2: chunks round-robin over the groups, all warps contribute to every task ----
  const uint32_t full2 = bars + 8 * Bars::full2, empty2 = bars + 8 * Bars::empty2;
  float gate = 1.f;
  if (p.sigmoid_gate && p.n_shared > 0) {  // Qwen-style shared-expert gate: sigmoid(v . x)
    float dot = lane < (p.hidden >> 7) ? reinterpret_cast<const float*>(smem + SmemLayout::gate)[lane] : 0.f;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, off);
    gate = 1.f / (1.f + expf(-dot));
  }
  int i = 0;
  for (int m = 0; m < plan.count2; ++m) {
    float part = 0.f, unused = 0.f, sacc = 0.f;
    int jcur = -1;
    for (; i < nmine; ++i) {
      const uint4 d = mylist[i];
      if ((int)((d.x >> 16) & 0xffu) != m) break;
      const int j = d.x & 0xffffu, rot = d.x >> 24;
      if (j != jcur) {  // weighted combine, in slot order
        if (jcur >= 0) part = fmaf(slots[jcur].gated ? gate : slots[jcur].coef, sacc, part);
        jcur = j;
        sacc = 0.f;
      }
      const int u0 = d.y & 0xffu, u1 = (d.y >> 8) & 0xffu;
      const int nblocks = d.z & 0xffu, col = (int)d.w;
      const bool p8 = (d.z & 256u) != 0u;
      if (!mbar_wait(full2 + 8 * (kFull2PerGroup * group + ((d.y >> 16) & 0xffu)), d.y >> 24, dead, status)) return;
      if (!wait_h_blocks(smem, col >> 7, nblocks, lane, dead, status)) return;  // this chunk's part of h, no more
      if (gw == 0 && i == nmine - 1) SM_TRACE(23 + group);
      const uint8_t* dig = smem + SmemLayout::hdig + col * 3;
      const float* sumw = reinterpret_cast<const float*>(smem + SmemLayout::hsumw) + (col >> LG) * 2;
      const float* binv = reinterpret_cast<const float*>(smem + SmemLayout::hinv) + (col >> 7);
      const uint8_t *unit0 = smem + SmemLayout::ring + u0 * plan.unit2_bytes, *unit1 = smem + SmemLayout::ring + u1 * plan.unit2_bytes;
      if (p8) consume_chunk<G, kModeBoth>(lr, lane, gw, rot, nblocks, unit0, unit1, plan.scale2_off, plan.zp2_off, dig, sumw, binv, &sacc, &unused, p.shift);
      else consume_chunk<G, kModeSingle>(lr, lane, gw, rot, nblocks, unit0, unit1, plan.scale2_off, plan.zp2_off, dig, sumw, binv, &sacc, &unused, p.shift);
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(empty2 + 8 * u0);
        if (p8) mbar_arrive(empty2 + 8 * u1);
      }
    }
    if (jcur >= 0) part = fmaf(slots[jcur].gated ? gate : slots[jcur].coef, sacc, part);
    part += __shfl_xor_sync(0xffffffffu, part, 1);
    if (!mbar_wait(bars + 8 * Bars::pempty2, (m & 1) ^ 1, dead, status)) return;
    if (lr.cq == 0) partial2[warp * 16 + lr.r] = part;
    __syncwarp();
    if (lane == 0) mbar_arrive(bars + 8 * Bars::pfull2);
  }
  if (warp == 0) SM_TRACE(11);
  if (gw == 0) SM_TRACE(27 + group);
}

// ---- epilogue warp ---------------------------------------------------------------------------------
__device__ void epilogue_loop(const DecodeParams& p, uint8_t* smem, int lane) {
  const Plan& plan = *reinterpret_cast<const Plan*>(smem + SmemLayout::plan);
  const float2* partial = reinterpret_cast<const float2*>(smem + SmemLayout::partial);
  const float* partial2 = reinterpret_cast<const float*>(smem + SmemLayout::partial2);
  volatile int* dead = reinterpret_cast<volatile int*>(smem + SmemLayout::dead);
  const uint32_t bars = smem_u32(smem + SmemLayout::bars);
  unsigned* status = &p.ws->status;
  // This CTA's share of the OTHER h buffer goes back to "empty" for the next launch: its last readers were the
  // launch before this one.
  {
    uint4* other = reinterpret_cast<uint4*>(p.ws_h + (size_t)(plan.hpar ^ 1) * kHCap);
    constexpr int n16 = kHCap / 4;
    const int per = (n16 + (int)gridDim.x - 1) / (int)gridDim.x;
    const int lo = (int)blockIdx.x * per, hi = min(n16, lo + per);
    for (int i = lo + lane; i < hi; i += 32) other[i] = make_uint4(kHEmpty, kHEmpty, kHEmpty, kHEmpty);
  }
  float* hbuf = p.ws_h + (size_t)plan.hpar * kHCap;
  // phase 1: one group's four partial rows per task -> SwiGLU -> h
  {
    for (int n = 0; n < plan.deal.count1; ++n) {
      const int ord = plan.deal.ordinal(plan.count_s, n, (int)blockIdx.x, (int)gridDim.x);
      const TaskPlace place(plan.deal.count_both, n);
      const int group = place.group(), round = place.round();
      if (!mbar_wait(bars + 8 * (Bars::pfull1 + group), round & 1, dead, status)) return;
      float a = 0.f, b = 0.f;
      if (lane < 16) {
#pragma unroll
        for (int w = 0; w < kGroupWarps; ++w) {
          const float2 v = partial[(group * kGroupWarps + w) * 16 + lane];
          a += v.x;
          b += v.y;
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(bars + 8 * (Bars::pempty1 + group));
      if (lane < 16) hbuf[ord * 16 + lane] = a / (1.f + expf(-a)) * b;  // silu(gate) * up
    }
  }
  SM_TRACE(12);
  // phase 2: all warps' partial rows per output row block -> y
  for (int m = 0; m < plan.count2; ++m) {
    if (!mbar_wait(bars + 8 * Bars::pfull2, m & 1, dead, status)) return;
    float b = 0.f;
    if (lane < 16) {
#pragma unroll
      for (int w = 0; w < kConsumerWarps; ++w) b += partial2[w * 16 + lane];
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(bars + 8 * Bars::pempty2);
    if (lane < 16) p.y[(blockIdx.x + m * gridDim.x) * 16 + lane] = b;
  }
  SM_TRACE(13);
  SM_TRACE_G(22);
}

// ---- producer --------------------------------------------------------------------------------------
// What a producer lane copies, for a phase-1 chunk of matrix A (and, in a pair chunk, matrix B):
//   lane 0  A's MSB tile            -> first unit, plane area
//   lane 1  A's LSB tile (8-bit) or B's MSB tile (pair) -> second unit, plane area
//   lane 2  A's scales, lane 3 A's zero-points          -> first unit, after the plane area
//   lane 4  B's scales, lane 5 B's zero-points (pair)   -> second unit, after the plane area
// For all of them the source of (row block rb, column block kb of 128) is
// base + (rb * (K / 128) + kb) * bytes_per_block, because planes and scale / zero-point arrays are all
// stored [row block][column][16 rows].
constexpr int kProducerLanes = 6;
struct ProducerLane {
  uint32_t bytes_per_block;  // bytes per (16 rows x 128 columns)
  int field;                 // which of the matrix' four pointers
  bool second_unit;
};
// What a producer needs to wait: it starts before the kernels ahead of this one in the stream have completed, so
// a wait that does not pass at once is first the moment to wait for those (the consumers, on whom all of a
// producer's barriers depend, do not start earlier; and a bounded wait's clock must not run while an earlier
// kernel is still busy).
struct ProducerWait {
  volatile int* dead;
  unsigned* status;
  bool dep_waited;  // griddepcontrol.wait has been executed
  __device__ __forceinline__ bool operator()(uint32_t bar, uint32_t parity) {
    if (mbar_try(bar, parity)) return true;
    if (!dep_waited) {
      asm volatile("griddepcontrol.wait;" ::: "memory");
      dep_waited = true;
    }
    return mbar_wait(bar, parity, dead, status);
  }
};

// One phase-1 chunk of (slot, row block rb), columns from k0: both slices of matrix `mat`, or (mode kModePair) the MSB tiles of gate
// and up side by side, into the unit pair from `u` on, once it is empty.  Run by the first kProducerLanes lanes of a producer warp
// together.  Returns false if a wait ran out.
template <int G>
__device__ __forceinline__ bool produce_chunk(uint8_t* smem, int u, uint32_t empty_bar, uint32_t empty_parity, uint32_t bar, int lane,
                                              const ProducerLane& pl, const Slot& s, int mat, int mode, int K, int rb, int k0,
                                              ProducerWait& pw, uint64_t pol) {
  constexpr int SG = 128 / G;
  const bool pair = mode == kModePair;
  const uint8_t* src;
  if (lane == 1) {
    src = pair ? s.ptr[1][0] : s.ptr[mat][1];
    if (!pair && src == nullptr) {  // 8 bits asked of an expert without LSB planes: defined garbage, reported
      src = s.ptr[mat][0];
      atomicOr(pw.status, (unsigned)SLICEMOE_STATUS_MISSING_LSB);
    }
  } else {
    src = s.ptr[lane >= 4 ? 1 : mat][pl.field];
  }
  src += (size_t)((unsigned)rb * (unsigned)(K >> 7) + (unsigned)(k0 >> 7)) * pl.bytes_per_block;
  const uint32_t nblk = (uint32_t)(min(kChunkK, K - k0) >> 7);
  if (!pw(empty_bar, empty_parity)) return false;
  if (lane == 0) mbar_arrive_expect_tx(bar, nblk * (2048u + (pair ? 2u : 1u) * (SG * 48u)));
  __syncwarp((1u << kProducerLanes) - 1u);
  if (lane < 4 || pair) {
    const uint32_t at = pl.field < 2 ? 0u : pl.field == 2 ? kPlaneUnitBytes : kPlaneUnitBytes + kScaleUnitBytes;
    bulk_g2s(smem_u32(smem + SmemLayout::ring) + (uint32_t)(pl.second_unit ? u + 1 : u) * kUnitBytes + at, src, nblk * pl.bytes_per_block, bar, pol);
  }
  return true;
}

// Whether a copy that was asked for before `t0` is not going to land any more: a millisecond is far more than any takes.
__device__ __forceinline__ bool copy_overdue(long long t0, volatile int* dead) {
  const unsigned long long waited = (unsigned long long)(clock64() - t0);
  return waited > 2000000ull && (*dead || waited > wait_limit(dead));
}

// Producer warp `which` of kProducers (phase 1): every producer walks the whole schedule and issues its share.
template <int G>
__device__ void producer_loop(const DecodeParams& p, uint8_t* smem, int lane, int which) {
  constexpr int LG = G == 128 ? 7 : (G == 64 ? 6 : 5);
  const Slot* slots = reinterpret_cast<const Slot*>(smem + SmemLayout::slots);
  const Plan& plan = *reinterpret_cast<const Plan*>(smem + SmemLayout::plan);
  volatile int* dead = reinterpret_cast<volatile int*>(smem + SmemLayout::dead);
  const uint32_t bars = smem_u32(smem + SmemLayout::bars);
  ProducerWait pw;
  pw.dead = dead;
  pw.status = &p.ws->status;
  pw.dep_waited = false;
  const uint64_t pol = l2_evict_first_policy();
  ProducerLane pl;
  pl.field = lane < 2 ? lane : 2 + (lane & 1);  // lanes 2, 4: scales; lanes 3, 5: zero-points
  pl.bytes_per_block = lane < 2 ? 1024u : (pl.field == 2 ? (128u >> LG) * 32u : (128u >> LG) * 16u);
  pl.second_unit = lane == 1 || lane >= 4;
  bool ok = true;
  const int nch = nchunks_of(p.hidden);
  static_assert(kGroups == 2 * kProducers, "a producer serves the groups `which` and `which + kProducers`");
  int ig_lo = 0, ig_hi = 0;  // chunks armed so far for group `which` and for group `which + kProducers`
  {
    const int per_s = p.shared_inter / 16, per_r = p.inter / 16, shared_tasks = p.n_shared * per_s;  // tasks of a slot
    const float inv_r = 1.f / (float)per_r;
    int jp = 0;  // this warp's chunks so far
    // The shared experts' tasks are known from the start; what follows them - and how many tasks there are - once
    // the plan stands.
    int n_end = plan.count_s;
    for (int n = 0; ok; ++n) {
      if (n == plan.count_s) {
        ok = pw(bars + 8 * Bars::plan_ready, 0);
        if (!ok) break;
        n_end = plan.deal.count1;
      }
      if (n >= n_end) break;
      const TaskPlace place(n < plan.count_s ? n + 1 : plan.deal.count_both, n);
      if (place.producer == which) {
        const int ord = plan.deal.ordinal(plan.count_s, n, (int)blockIdx.x, (int)gridDim.x), routed = ord - shared_tasks;
        int slot, idx;
        if (routed < 0) {
          slot = ord / per_s;
          idx = ord - slot * per_s;
        } else {  // (the first request waits for this: no integer division)
          slot = (int)((float)routed * inv_r);
          idx = routed - slot * per_r;
          if (idx < 0) --slot, idx += per_r;
          if (idx >= per_r) ++slot, idx -= per_r;
          slot += p.n_shared;
        }
        const Slot& s = slots[slot];
        const int nchunks = s.prec ? 2 * nch : nch;
        const int g = place.group();
        for (int q = 0; q < nchunks && ok; ++q, ++jp) {
          int& igg = g == which ? ig_lo : ig_hi;
          ok = produce_chunk<G>(smem, 4 * which + 2 * (jp & 1), bars + 8 * (Bars::empty + 2 * which + (jp & 1)), ((jp >> 1) & 1) ^ 1,
                                bars + 8 * (Bars::full + 2 * g + (igg & 1)), lane, pl, s, s.prec ? q / nch : 0,
                                s.prec ? kModeBoth : kModePair, p.hidden, idx, (q % nch) * kChunkK, pw, pol);
          ++igg;
          if (which == 0 && lane == 0 && jp < 8) SM_TRACE(32 + jp);
        }
      }
    }
  }
  // Never leave the CTA with bulk copies still landing in its shared memory: wait (bounded) until every
  // barrier this warp may have armed has completed its last phase.  In the normal path they have long ago.
  for (int g = which; g < kGroups; g += kProducers) {
    const int n1 = g == which ? ig_lo : ig_hi;
    for (int i = max(0, n1 - 2); i < n1; ++i) {
      const long long t0 = clock64();
      while (!mbar_try(bars + 8 * (Bars::full + 2 * g + (i & 1)), (i >> 1) & 1)) {
        if (copy_overdue(t0, dead)) break;
      }
    }
  }
}

// The down tiles: rows of every slot for the output row blocks of this CTA, in the re-cut ring.  Nothing else is left to bring
// by then and everybody waits for these, so a lane asks for one array of one chunk: what it copies is worked out while phase 1
// still runs, and up to eight chunks are asked for by one instruction (a warp issues copies lane by lane, 60 cycles each; chunk
// after chunk, with what goes into one worked out in between, was 1700 cycles a chunk).
template <int G>
__device__ void down_loop(const DecodeParams& p, uint8_t* smem, int lane) {
  constexpr int SG = 128 / G;
  const Slot* slots = reinterpret_cast<const Slot*>(smem + SmemLayout::slots);
  const Plan& plan = *reinterpret_cast<const Plan*>(smem + SmemLayout::plan);
  volatile int* dead = reinterpret_cast<volatile int*>(smem + SmemLayout::dead);
  const uint32_t bars = smem_u32(smem + SmemLayout::bars);
  unsigned* status = &p.ws->status;
  if (!mbar_wait(bars + 8 * Bars::plan_ready, 0, dead, status) || plan.count2 == 0) return;
  const uint64_t pol = l2_evict_first_policy();
  const int units = plan.nunits2, chunks = plan.p2c[plan.nslots], chunk_units = plan.p2u[plan.nslots], total = plan.count2 * chunks;
  const int array = lane & 3;  // MSB plane, LSB plane, scales, zero-points
  const uint32_t block_bytes = array < 2 ? 1024u : array == 2 ? SG * 32u : SG * 16u;
  int done = 0;  // chunks asked for
  bool ok = true;
  while (done < total && ok) {
    // Up to eight chunks at a time.  A lane's chunk: row block m, slot j, columns from k0 on, first unit x of a running count.
    const int at = lane >> 2, base = done, c = base + at, n = min(8, total - base);
    const int m = c / chunks, r = c - m * chunks;
    int j = 0;
    while (j + 1 < plan.nslots && plan.p2c[j + 1] <= r) ++j;
    const Slot& s = slots[j];
    const int w = s.prec ? 2 : 1, k0 = (r - plan.p2c[j]) * kChunkK, x = m * chunk_units + plan.p2u[j] + (r - plan.p2c[j]) * w;
    const int nblk = min(kChunkK, s.inter - k0) >> 7;
    const uint8_t* src = s.ptr[2][array];
    if (at < n && array == 1 && s.prec && src == nullptr) {  // 8 bits asked of an expert without LSB planes: defined garbage, reported
      src = s.ptr[2][0];
      atomicOr(status, (unsigned)SLICEMOE_STATUS_MISSING_LSB);
    }
    src += (size_t)((unsigned)(blockIdx.x + m * gridDim.x) * (unsigned)(s.inter >> 7) + (unsigned)(k0 >> 7)) * block_bytes;
    const int lap0 = x / units, u0 = x - lap0 * units, u1 = u0 + 1 == units ? 0 : u0 + 1, lap1 = u1 == 0 ? lap0 + 1 : lap0;
    const uint32_t dst = smem_u32(smem + SmemLayout::ring) + (uint32_t)(array == 1 ? u1 : u0) * (uint32_t)plan.unit2_bytes +
                         (array < 2 ? 0u : (uint32_t)(array == 2 ? plan.scale2_off : plan.zp2_off));
    const uint32_t bar = bars + 8 * (Bars::full2 + kFull2PerGroup * (c % kGroups) + c / kGroups % kFull2PerGroup);
    const uint32_t bytes = (uint32_t)nblk * block_bytes, all_bytes = (uint32_t)nblk * ((w == 2 ? 2048u : 1024u) + SG * 48u);
    if (base == 0) {
      // The re-cut units lie over the phase-1 units: nothing of phase 2 lands before phase 1 has been consumed.
      ok = mbar_wait(bars + 8 * Bars::p1_done, 0, dead, status);
      SM_TRACE(31);
    }
    // what finds its units empty goes at once, the rest chunk by chunk as units become free
    const int fresh = __popc(__ballot_sync(0xffffffffu, at < n && x + w <= units)) >> 2;
    for (int q = 0; q < n; q = max(q + 1, fresh)) {
      const int end = max(q + 1, fresh);
      const bool mine = at >= q && at < end;
      if (ok && mine && lap0 > 0) ok = mbar_wait(bars + 8 * (Bars::empty2 + u0), (lap0 & 1) ^ 1, dead, status);
      if (ok && mine && w == 2 && lap1 > 0) ok = mbar_wait(bars + 8 * (Bars::empty2 + u1), (lap1 & 1) ^ 1, dead, status);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      if (mine && array == 0) mbar_arrive_expect_tx(bar, all_bytes);
      __syncwarp();
      if (mine && (array != 1 || w == 2)) bulk_g2s(dst, src, bytes, bar, pol);
      done += end - q;
    }
  }
  SM_TRACE(18);
  // no copy may still be landing when the CTA ends (in the normal path they have all been consumed); at most as many are on
  // their way as there are units
  const int c = done - 1 - lane;
  if (lane < kUnits2 && c >= 0) {
    const long long t0 = clock64();
    while (!mbar_try(bars + 8 * (Bars::full2 + kFull2PerGroup * (c % kGroups) + c / kGroups % kFull2PerGroup), (c / kGroups / kFull2PerGroup) & 1))
      if (copy_overdue(t0, dead)) break;
  }
}

// ---- prologue pieces ---------------------------------------------------------------------------------
// Slot order: shared experts, then the routed experts that run at 8 bits, then those that run at 4 bits,
// each group in list order.
//
// The routing list as one warp sees it: lane j < k holds entry j; out-of-range ids are dropped.
struct Routed {
  int e, pr;
  float w;
  bool valid;
  int pos;  // slot index of this lane's entry
  int nbig, nsmall;
};
template <bool FUSED>
__device__ __forceinline__ Routed read_routing(const DecodeParams& p, int lane, bool publish) {
  Routed rt;
  rt.e = -1;
  rt.pr = 0;
  rt.w = 0.f;
  if (FUSED) {
    // same arithmetic as the stand-alone routing kernel; the precision request is the precision
    const RouteSel sel = route_warp(RouteGlobal{p.logits}, p.n_experts, p.k, p.bias, p.renorm, p.tau, p.rank_high, lane);
    if (lane < p.k) {
      rt.e = sel.id;
      rt.pr = sel.prec_req;
      rt.w = sel.w;
      if (publish && blockIdx.x == 0) {
        if (p.ids_out) p.ids_out[lane] = sel.id;
        if (p.prec_out) p.prec_out[lane] = sel.prec_req;
        if (p.weights_out) p.weights_out[lane] = sel.w;
      }
    }
  } else if (lane < p.k) {
    rt.e = __ldcg(p.ids + lane);
    rt.pr = __ldcg(p.prec + lane);
    rt.w = __ldcg(p.weights + lane);
  }
  rt.valid = lane < p.k && rt.e >= 0 && rt.e < p.n_experts;
  const unsigned vmask = __ballot_sync(0xffffffffu, rt.valid);
  const unsigned bigmask = __ballot_sync(0xffffffffu, rt.valid && rt.pr != 0);
  const unsigned below = (1u << lane) - 1u;
  rt.nbig = __popc(bigmask);
  rt.nsmall = __popc(vmask) - rt.nbig;
  rt.pos = p.n_shared + (rt.pr != 0 ? __popc(bigmask & below) : rt.nbig + __popc(vmask & ~bigmask & below));
  return rt;
}

// The plane pointers of `count` slots from `first` on; each slot's expert is shared + slot, or what the slot table's first pointer
// names.  A slot's twelve pointers sit in slicemoe_expert in the order the slot table keeps them.
__device__ __forceinline__ void load_slot_pointers(const DecodeParams& p, Slot* slots, int lane, int first, int count, bool routed) {
  constexpr int kRounds = (kMaxSlots * 12 + 31) / 32;
  unsigned long long val[kRounds];
#pragma unroll
  for (int rd = 0; rd < kRounds; ++rd) {  // all loads in flight together
    if (rd * 32 >= count * 12) break;
    const int i = rd * 32 + lane;
    if (i < count * 12) {
      const int sl = first + i / 12, q = i % 12;
      const slicemoe_expert* ex = routed ? reinterpret_cast<const slicemoe_expert*>(slots[sl].ptr[0][0]) : p.shared + sl;
      val[rd] = __ldcg(reinterpret_cast<const unsigned long long*>(reinterpret_cast<const slicemoe_mat*>(ex) + (q >> 2)) + (q & 3));
    }
  }
  __syncwarp();  // every lane has read the experts' addresses before the first slot pointer overwrites one
#pragma unroll
  for (int rd = 0; rd < kRounds; ++rd) {
    if (rd * 32 >= count * 12) break;
    const int i = rd * 32 + lane;
    if (i < count * 12) slots[first + i / 12].ptr[(i % 12) >> 2][i & 3] = reinterpret_cast<const uint8_t*>(val[rd]);
  }
}

// What of the plan depends on the shape and the grid alone; one lane computes it while the kernel still waits
// for the grids before it.  Assumes at least one valid routed entry when k > 0 (build_plan redoes the unit
// size in the rare case that there is none).
__device__ __forceinline__ int phase2_unit_blocks(const DecodeParams& p, bool any_routed) {
  int maxblk = 1;
  if (p.n_shared) maxblk = max(maxblk, min(kChunkK, p.shared_inter) >> 7);
  if (any_routed) maxblk = max(maxblk, min(kChunkK, p.inter) >> 7);
  return maxblk;
}
__device__ __forceinline__ void plan_units2(const DecodeParams& p, Plan* plan, int maxblk) {
  const int meta_blk = 16 * (128 / p.group);  // scale entries per 128 columns
  plan->scale2_off = maxblk * 1024;
  plan->zp2_off = maxblk * 1024 + maxblk * meta_blk * 2;
  plan->unit2_bytes = (maxblk * (1024 + meta_blk * 3) + 127) & ~127;
  plan->nunits2 = min(kUnits2, (kUnits * kUnitBytes) / plan->unit2_bytes);
}
// Run by the epilogue warp, as what follows.
__device__ void build_plan_static(const DecodeParams& p, uint8_t* smem, int lane) {
  Slot* slots = reinterpret_cast<Slot*>(smem + SmemLayout::slots);
  Plan* plan = reinterpret_cast<Plan*>(smem + SmemLayout::plan);
  if (lane < p.n_shared) {
    Slot& s = slots[lane];
    s.inter = p.shared_inter;
    s.prec = 1;
    s.coef = 1.f;
    s.gated = p.sigmoid_gate;
    s.hoff = lane * p.shared_inter;
  }
  if (lane != 0) return;
  const int nrb = p.hidden / 16;
  plan->count2 = (int)blockIdx.x < nrb ? (nrb - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  plan_units2(p, plan, phase2_unit_blocks(p, p.k > 0));
  plan->count_s = dealt(p.n_shared * (p.shared_inter / 16), (int)blockIdx.x, (int)gridDim.x);
}

// The routed slots (all but the pointers) and the partition, in closed form.
template <bool FUSED>
__device__ __forceinline__ void build_plan(const DecodeParams& p, uint8_t* smem, int lane) {
  Slot* slots = reinterpret_cast<Slot*>(smem + SmemLayout::slots);
  Plan* plan = reinterpret_cast<Plan*>(smem + SmemLayout::plan);
  const Routed rt = read_routing<FUSED>(p, lane, true);
  if (rt.valid) {
    Slot& s = slots[rt.pos];
    s.inter = p.inter;
    s.prec = rt.pr != 0;
    s.coef = rt.w;
    s.gated = 0;
    s.hoff = p.n_shared * p.shared_inter + (rt.pos - p.n_shared) * p.inter;
  } else if (lane < p.k) {
    atomicOr(&p.ws->status, (unsigned)SLICEMOE_STATUS_BAD_EXPERT_ID);
  }
  __syncwarp();
  {
    const int nslots = p.n_shared + rt.nbig + rt.nsmall;
    // phase-2 chunk and unit counts before each slot: lane j handles slot j (8-bit: shared and the first nbig routed)
    {
      int cj = 0, uj = 0;
      if (lane < nslots) {
        const int inter = lane < p.n_shared ? p.shared_inter : p.inter;
        const bool p8 = lane < p.n_shared + rt.nbig;
        cj = nchunks_of(inter);
        uj = p8 ? 2 * cj : cj;
      }
      int ci = cj, ui = uj;  // inclusive scans
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const int a = __shfl_up_sync(0xffffffffu, ci, off), b = __shfl_up_sync(0xffffffffu, ui, off);
        if (lane >= off) {
          ci += a;
          ui += b;
        }
      }
      if (lane < nslots) {
        plan->p2c[lane + 1] = (short)ci;
        plan->p2u[lane + 1] = (short)ui;
      }
      if (lane == 0) plan->p2c[0] = plan->p2u[0] = 0;
    }
    if (lane == 0) {
      const int per = p.inter / 16;  // tasks of a routed slot
      plan->deal.set(p.n_shared * (p.shared_inter / 16) + rt.nbig * per, rt.nsmall * per, (int)blockIdx.x, (int)gridDim.x);
      if (nslots == 0) plan->count2 = 0;  // otherwise as build_plan_static left it
      plan->nslots = nslots;
      plan->htotal = p.n_shared * p.shared_inter + (rt.nbig + rt.nsmall) * p.inter;
      // phase-2 units: as large as the widest down chunk of any slot (set ahead of time for the usual case)
      if (rt.nbig + rt.nsmall == 0 && p.k > 0) plan_units2(p, plan, phase2_unit_blocks(p, false));
    }
  }
  __syncwarp();
  if (lane == 0) mbar_arrive(smem_u32(smem + SmemLayout::bars) + 8 * Bars::plan_ready);
}
// The routed slots' pointers.
template <bool FUSED>
__device__ __forceinline__ void routed_pointers(const DecodeParams& p, uint8_t* smem, int lane) {
  Slot* slots = reinterpret_cast<Slot*>(smem + SmemLayout::slots);
  const Routed rt = read_routing<FUSED>(p, lane, false);
  // lane j knows its entry's slot; every lane needs every slot's expert: passed through the slot table
  if (rt.valid) slots[rt.pos].ptr[0][0] = reinterpret_cast<const uint8_t*>(p.experts + rt.e);
  __syncwarp();
  load_slot_pointers(p, slots, lane, p.n_shared, rt.nbig + rt.nsmall, true);
  __syncwarp();
  if (lane == 0) mbar_arrive(smem_u32(smem + SmemLayout::bars) + 8 * Bars::plan_ready);
}

// ---- the kernel ------------------------------------------------------------------------------------
// FUSED: the routing list is computed from the router logits in the prologue (slicemoe_layer_routed); kept
// apart from the plain kernel so that the latter carries none of the routing code.
template <int G, bool FUSED>
__global__ void __launch_bounds__(kThreads, 1) decode_layer_kernel(const __grid_constant__ DecodeParams p) {
  extern __shared__ __align__(128) uint8_t smem[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  Plan* plan = reinterpret_cast<Plan*>(smem + SmemLayout::plan);

  // Programmatic dependent launch: the next kernel in the stream may start launching as soon as every CTA
  // of this grid has got here (its CTAs find room only where one of ours has exited), and this kernel does
  // all it can before it waits for the grids before it.  Nothing an earlier kernel may write is touched
  // before that wait: x and the workspace always, and the routing lists unless the caller has promised that
  // they were complete earlier (lists_resident).  The weights and expert tables are not written by a kernel in flight that
  // lets this one start: pack_kernel does not, and a caller's own kernels must not (slicemoe.h, "Order").
#ifdef SLICEMOE_TRACE
  if (tid == 0) s_trace_t0 = clock64();
  if (tid == 0 && blockIdx.x < 256) g_trace[blockIdx.x][20] = trace_gtime();
#endif
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const bool early_lists = !FUSED && p.lists_resident != 0;
  if (warp == kProducerWarp) {
    if (lane == 0) {
      *reinterpret_cast<int*>(smem + SmemLayout::dead) = 0;
      *reinterpret_cast<int*>(smem + SmemLayout::hnext) = 0;
      *reinterpret_cast<unsigned long long*>(smem + SmemLayout::dead + 8) = kWaitCycles;
      for (int i = 0; i < kHCap / 128; i += 8) *reinterpret_cast<unsigned long long*>(smem + SmemLayout::hready + i) = 0ull;
      const uint32_t bars = smem_u32(smem + SmemLayout::bars);
      for (int s = 0; s < kUnits; ++s) {
        mbar_init(bars + 8 * (Bars::full + s), 1);             // lane 0's expect_tx arrive
        mbar_init(bars + 8 * (Bars::empty + s), kGroupWarps);  // one arrive per warp of the consuming group
      }
      for (int s = 0; s < kGroups * kFull2PerGroup; ++s) mbar_init(bars + 8 * (Bars::full2 + s), 1);
      for (int s = 0; s < kUnits2; ++s) mbar_init(bars + 8 * (Bars::empty2 + s), kGroupWarps);
      for (int g = 0; g < kGroups; ++g) {
        mbar_init(bars + 8 * (Bars::pfull1 + g), kGroupWarps);
        mbar_init(bars + 8 * (Bars::pempty1 + g), 1);
      }
      mbar_init(bars + 8 * Bars::pfull2, kConsumerWarps);
      mbar_init(bars + 8 * Bars::pempty2, 1);
      mbar_init(bars + 8 * Bars::p1_done, kConsumerWarps);
      mbar_init(bars + 8 * Bars::plan_ready, 2);  // the plan, the pointers
      mbar_init(bars + 8 * Bars::head_ready, 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
  }
  // Ahead of the wait: what follows from the shape alone - the shared experts' slots, pointers and this CTA's share
  // of their tasks - and the routed experts' pointer table on its way into L2 (its entries are read right after the
  // wait).
  if (warp == kEpilogueWarp) {
    build_plan_static(p, smem, lane);
  } else if (warp == kDownWarp) {
    if (p.n_shared > 0) load_slot_pointers(p, reinterpret_cast<Slot*>(smem + SmemLayout::slots), lane, 0, p.n_shared, false);
  } else if (warp == 1 && p.experts != nullptr && p.k > 0 && !early_lists) {
    const char* tab = reinterpret_cast<const char*>(p.experts);
    const size_t bytes = (size_t)p.n_experts * sizeof(slicemoe_expert);
    for (size_t off = (size_t)lane * 128; off < bytes; off += 32 * 128)
      asm volatile("prefetch.global.L2 [%0];" ::"l"(tab + off));
  }
  __syncthreads();
  if (warp >= kProducerWarp && warp < kDownWarp) {
    // The producers start on the shared experts' tiles (and, with resident lists, go on to the routed experts')
    // while the kernels ahead are still running; see ProducerWait for where they wait for those.
    if (lane < kProducerLanes) producer_loop<G>(p, smem, lane, warp - kProducerWarp);
    return;
  }

  // Everyone else waits here.  Then the consumer warps turn x into digits, one or two 128-element blocks each, and go on to
  // the shared experts' tiles, while the epilogue warp reads the routing list, builds the routed slots and the partition and
  // tells everybody.  (With resident lists it does so first, while the producers are already busy with the shared experts'
  // tiles.)  What a kernel ahead may have written is read past L1: it may have run on this SM after this CTA began.
  if (warp == kDownWarp) {
    if (early_lists) routed_pointers<FUSED>(p, smem, lane);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // readers, epoch, status, extra_arrivals; a wait limit set by the host for this workspace
    const uint4 head = __ldcg(reinterpret_cast<const uint4*>(p.ws));
    const unsigned long long lim = __ldcg(&p.ws->wait_cycles);
    if (!early_lists) routed_pointers<FUSED>(p, smem, lane);
    if (lane == 0) {
      if (lim != 0ull) *reinterpret_cast<unsigned long long*>(smem + SmemLayout::dead + 8) = lim;
      // Which h buffer: the parity of the launch count.  The count moves on once every CTA of this launch has
      // read it (the last reader does it), so all of them see the same value, and the next launch the next.
      plan->hpar = (int)(head.y & 1u);
      plan->never_ready = head.w != 0u ? 1 : 0;
      mbar_arrive(smem_u32(smem + SmemLayout::bars) + 8 * Bars::head_ready);
      if (atomicAdd(&p.ws->readers, 1u) == gridDim.x - 1u) {
        p.ws->readers = 0u;
        p.ws->epoch = head.y + 1u;
        __threadfence();
      }
    }
    __syncwarp();
    down_loop<G>(p, smem, lane);
    return;
  }
  if (warp == kEpilogueWarp) {
    if (!early_lists) asm volatile("griddepcontrol.wait;" ::: "memory");
    build_plan<FUSED>(p, smem, lane);
    if (early_lists) asm volatile("griddepcontrol.wait;" ::: "memory");
    SM_TRACE(2);
    if (mbar_wait(smem_u32(smem + SmemLayout::bars) + 8 * Bars::head_ready, 0, reinterpret_cast<volatile int*>(smem + SmemLayout::dead), &p.ws->status))
      epilogue_loop(p, smem, lane);
    return;
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (warp == 3) {
    SM_TRACE(1);
    SM_TRACE_G(21);
  }
  {
    constexpr int kMine = kMaxHidden / 128 / kConsumerWarps;
    const bool gated = p.sigmoid_gate && p.n_shared > 0;
    uint2 raw[kMine];
    float gv[kMine][4];
#pragma unroll
    for (int i = 0; i < kMine; ++i)
      if ((warp + kConsumerWarps * i) * 128 < p.hidden)
        raw[i] = __ldcg(reinterpret_cast<const uint2*>(p.x + (warp + kConsumerWarps * i) * 128) + lane);
    if (gated) {
#pragma unroll
      for (int i = 0; i < kMine; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
          gv[i][j] = (warp + kConsumerWarps * i) * 128 < p.hidden ? __ldg(p.gate_vec + (warp + kConsumerWarps * i) * 128 + 4 * lane + j) : 0.f;
    }
#pragma unroll
    for (int i = 0; i < kMine; ++i) {
      const int blk = warp + kConsumerWarps * i;
      if (blk * 128 < p.hidden) {
        const float v[4] = {__uint_as_float(raw[i].x << 16), __uint_as_float(raw[i].x & 0xffff0000u),
                            __uint_as_float(raw[i].y << 16), __uint_as_float(raw[i].y & 0xffff0000u)};
        block_to_digits<G>(v, blk * 128, lane, smem + SmemLayout::xdig, reinterpret_cast<float*>(smem + SmemLayout::xsumw),
                           reinterpret_cast<float*>(smem + SmemLayout::xinv));
        if (gated) {
          float dot = 0.f;
#pragma unroll
          for (int j = 0; j < 4; ++j) dot = fmaf(gv[i][j], v[j], dot);
#pragma unroll
          for (int off = 16; off > 0; off >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, off);
          if (lane == 0) reinterpret_cast<float*>(smem + SmemLayout::gate)[blk] = dot;
        }
      }
    }
  }
  if (warp == 3) SM_TRACE(3);
  asm volatile("bar.sync 1, %0;" ::"n"(32 * kConsumerWarps) : "memory");
  if (warp == 3) SM_TRACE(4);
  consumer_loop<G>(p, smem, warp, lane);
}

// ---- inputs in host memory ---------------------------------------------------------------------------
// A decode step whose x and logits sit in device-mapped host memory: one block reads them over the bus, side by side, routes
// (so that the layer kernel, whose every CTA would otherwise work out the list for itself, just reads it) and leaves x and
// the list in the workspace.  The layer kernel's launch overlaps it.  Bound: one trip over the bus, about 2 us.  Against
// two copies and the layer kernel with the routing in its prologue - copies cannot overlap the launch, and the prologue
// is 3 us longer - a step of the 2048-wide layer takes 34 us instead of 38.
constexpr int kStageThreads = 256;
__global__ void __launch_bounds__(kStageThreads) stage_step_kernel(const uint32_t* x_host, const float* logits_host, int hidden, int E,
                                                                   int k, const float* bias, int renorm, float tau, int rank_high,
                                                                   uint32_t* x, int32_t* ids, float* weights, uint8_t* prec) {
  __shared__ float row[32 * ROUTE_MAX_VPT];
  const int tid = threadIdx.x, lane = tid & 31;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");  // the work ahead may be what writes the host buffers
  constexpr int kWords = kMaxHidden / 2 / kStageThreads;
  uint32_t v[kWords];
#pragma unroll
  for (int i = 0; i < kWords; ++i)
    if (i * kStageThreads + tid < hidden / 2) v[i] = __ldcv(x_host + i * kStageThreads + tid);
  for (int e = tid; e < E; e += kStageThreads) row[e] = __ldcv(logits_host + e);
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kWords; ++i)
    if (i * kStageThreads + tid < hidden / 2) x[i * kStageThreads + tid] = v[i];
  if (tid < 32) {
    const RouteSel sel = route_warp(RouteShared{row}, E, k, bias, renorm, tau, rank_high, lane);
    if (lane < k) {
      ids[lane] = sel.id;
      weights[lane] = sel.w;
      prec[lane] = sel.prec_req;
    }
  }
}

// ---- host side --------------------------------------------------------------------------------------
static int g_num_sms[64];
static bool g_attr_set[64][6];

static int device_setup(int* dev_out, int* sms_out) {
  int dev = 0;
  SM_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return SLICEMOE_E_UNSUPPORTED;
  if (g_num_sms[dev] == 0) {
    int sms = 0;
    SM_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    g_num_sms[dev] = sms;
  }
  *dev_out = dev;
  *sms_out = g_num_sms[dev];
  return SLICEMOE_OK;
}

template <int G, bool FUSED>
static int launch_decode(const DecodeParams& p, int dev, int sms, int gi, cudaStream_t st, bool cooperative = false) {
  bool& attr_set = g_attr_set[dev][2 * gi + (FUSED ? 1 : 0)];
  if (!attr_set) {
    SM_CUDA_TRY(cudaFuncSetAttribute(decode_layer_kernel<G, FUSED>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     SmemLayout::total));
    // Every CTA waits for h values that the other CTAs write, so all of them must be able to be resident at
    // once: one per SM needs the kernel to fit an SM at all.  (If another kernel holds SMs at the time, the
    // bounded wait for h ends the launch with SLICEMOE_STATUS_WAIT_TIMEOUT instead of a hang.)
    int per_sm = 0;
    SM_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, decode_layer_kernel<G, FUSED>, kThreads,
                                                              SmemLayout::total));
    if (per_sm < 1) return SLICEMOE_E_UNSUPPORTED;
    attr_set = true;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(sms);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = SmemLayout::total;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // see the top of the kernel
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  // On request the driver is asked to guarantee that all CTAs are resident together (they wait for one another's
  // h values): the launch then fails instead of timing out when the device cannot hold the grid, at the price of
  // the CTA-by-CTA hand-over between consecutive launches.
  attr[1].id = cudaLaunchAttributeCooperative;
  attr[1].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cooperative ? 2 : 1;
  SM_CUDA_TRY(cudaLaunchKernelEx(&cfg, decode_layer_kernel<G, FUSED>, p));
  return SLICEMOE_OK;
}

static int check_shape(const slicemoe_shape* s) {
  if (!s) return SLICEMOE_E_INVALID_ARG;
  if (!valid_widths(s->b_high, s->b_low)) return SLICEMOE_E_UNSUPPORTED;
  if (!valid_group(s->group)) return SLICEMOE_E_UNSUPPORTED;
  if (s->hidden <= 0 || s->inter <= 0 || s->n_experts <= 0 || s->top_k < 1) return SLICEMOE_E_INVALID_ARG;
  if (s->top_k > s->n_experts || s->top_k > SLICEMOE_MAX_TOP_K) return SLICEMOE_E_INVALID_ARG;
  if (s->n_shared < 0 || s->n_shared > SLICEMOE_MAX_SHARED) return SLICEMOE_E_INVALID_ARG;
  if ((s->hidden % 128) || (s->inter % 128)) return SLICEMOE_E_INVALID_ARG;
  if (s->n_shared > 0 && (s->shared_inter <= 0 || (s->shared_inter % 128))) return SLICEMOE_E_INVALID_ARG;
  if (s->hidden > kMaxHidden) return SLICEMOE_E_UNSUPPORTED;
  return SLICEMOE_OK;
}

// Routing computed in the kernel (run_layer's `fused` argument): logits [T, E] in, lists [T, k] out (optional).
struct FusedRouting {
  const float* logits;
  const float* bias;
  int renorm, rank_high;
  float tau;
  int32_t* ids_out;
  uint8_t* prec_out;
  float* weights_out;
};

// What a layer call refuses beyond missing arguments, of a checked shape; the device's index and number of SMs.
static int check_layer(const slicemoe_shape* shape, const slicemoe_expert* shared, int n_shared, const float* gate_vec, const void* x,
                       const void* workspace, size_t workspace_bytes, int* dev, int* sms) {
  if (n_shared > 0 && !shared) return SLICEMOE_E_INVALID_ARG;
  if (n_shared > 0 && shape->shared_sigmoid_gate && !gate_vec) return SLICEMOE_E_INVALID_ARG;
  if (workspace_bytes < kWsBytes || (reinterpret_cast<uintptr_t>(workspace) & 255)) return SLICEMOE_E_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(x) & 15) return SLICEMOE_E_INVALID_ARG;
  const long long hsum = (long long)shape->top_k * shape->inter + (long long)n_shared * shape->shared_inter;
  if (hsum > kHCap) return SLICEMOE_E_UNSUPPORTED;
  const int rc = device_setup(dev, sms);
  if (rc != SLICEMOE_OK) return rc;
  // at most 4 output row blocks per CTA: what the consumer groups' phase-2 chunk lists are sized for
  if ((shape->hidden / 16 + *sms - 1) / *sms > 4) return SLICEMOE_E_UNSUPPORTED;
  return SLICEMOE_OK;
}

static int run_layer(const slicemoe_shape* shape, const slicemoe_expert* experts, const slicemoe_expert* shared,
                     int n_shared, const float* gate_vec, const void* x, int T, const int32_t* ids,
                     const uint8_t* prec, const float* weights, float* y, void* workspace, size_t workspace_bytes,
                     void* stream, const FusedRouting* fused = nullptr, unsigned flags = 0u) {
  int rc = check_shape(shape);
  if (rc != SLICEMOE_OK) return rc;
  if (!experts || !x || !y || !workspace || T <= 0) return SLICEMOE_E_INVALID_ARG;
  if (fused ? !fused->logits : (!ids || !prec || !weights)) return SLICEMOE_E_INVALID_ARG;
  if (fused && shape->n_experts > 32 * ROUTE_MAX_VPT) return SLICEMOE_E_UNSUPPORTED;
  if ((flags & ~(unsigned)(SLICEMOE_LISTS_RESIDENT | SLICEMOE_COOPERATIVE)) != 0u || (fused && flags != 0u)) return SLICEMOE_E_INVALID_ARG;
  const bool coop = (flags & SLICEMOE_COOPERATIVE) != 0u;
  int dev, sms;
  rc = check_layer(shape, shared, n_shared, gate_vec, x, workspace, workspace_bytes, &dev, &sms);
  if (rc != SLICEMOE_OK) return rc;

  DecodeParams p;
  p.experts = experts;
  p.shared = shared;
  p.gate_vec = gate_vec;
  p.ws = reinterpret_cast<WsHeader*>(workspace);
  p.ws_h = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(workspace) + kWsHOff);
  p.n_experts = shape->n_experts;
  p.n_shared = n_shared;
  p.k = shape->top_k;
  p.hidden = shape->hidden;
  p.inter = shape->inter;
  p.shared_inter = n_shared > 0 ? shape->shared_inter : 0;
  p.group = shape->group;
  p.sigmoid_gate = (n_shared > 0 && shape->shared_sigmoid_gate) ? 1 : 0;
  p.lists_resident = (flags & SLICEMOE_LISTS_RESIDENT) ? 1 : 0;
  p.shift = shape->b_high - shape->b_low;
  cudaStream_t st = (cudaStream_t)stream;
  p.logits = nullptr;
  p.bias = fused ? fused->bias : nullptr;
  p.renorm = fused ? fused->renorm : 0;
  p.rank_high = fused ? fused->rank_high : 0;
  p.tau = fused ? fused->tau : 0.f;
  p.ids_out = nullptr;
  p.prec_out = nullptr;
  p.weights_out = nullptr;
  p.ids = nullptr;
  p.prec = nullptr;
  p.weights = nullptr;
  // A small batch: every expert is streamed once for all of a pass' tokens.  (A workspace of the batch-1 kernel's size, as
  // slicemoe_layer_static's, has no room for that: token after token then.)
  const size_t batch_bytes = batch_workspace_bytes(shape, n_shared);
  if (T >= kBatchMinTokens && workspace_bytes >= kWsBatchOff + batch_bytes + kWsListBytes &&
      batch_fits(shape, n_shared, T < kBatchTokens ? T : kBatchTokens, sms)) {
    uint8_t* bws = reinterpret_cast<uint8_t*>(workspace) + kWsBatchOff;
    uint8_t* lists = bws + batch_bytes;
    const BatchControl ctl = {&p.ws->status, &p.ws->extra_arrivals, &p.ws->wait_cycles};
    const int passes = (T + kBatchTokens - 1) / kBatchTokens, k = shape->top_k;
    for (int i = 0; i < passes; ++i) {
      const int t0 = (int)((long long)T * i / passes), n = (int)((long long)T * (i + 1) / passes) - t0;
      const size_t o = (size_t)t0 * k;
      const int32_t* pids = ids ? ids + o : nullptr;
      const uint8_t* pprec = prec ? prec + o : nullptr;
      const float* pw = weights ? weights + o : nullptr;
      if (fused) {
        int32_t* ri = fused->ids_out ? fused->ids_out + o : reinterpret_cast<int32_t*>(lists);
        float* rw = fused->weights_out ? fused->weights_out + o : reinterpret_cast<float*>(lists) + kWsListEntries;
        uint8_t* rp = fused->prec_out ? fused->prec_out + o : lists + 8 * kWsListEntries;
        rc = slicemoe_route_topk(fused->logits + (size_t)t0 * shape->n_experts, n, shape->n_experts, k, fused->bias, fused->renorm, fused->tau,
                                 fused->rank_high, ri, rw, rp, stream);
        if (rc != SLICEMOE_OK) return rc;
        pids = ri;
        pprec = rp;
        pw = rw;
      }
      rc = batch_layer(shape, experts, shared, n_shared, gate_vec, reinterpret_cast<const uint16_t*>(x) + (size_t)t0 * shape->hidden, n, pids,
                       pprec, pw, y + (size_t)t0 * shape->hidden, bws, ctl, sms, stream);
      if (rc != SLICEMOE_OK) return rc;
    }
    return SLICEMOE_OK;
  }
  for (int t = 0; t < T; ++t) {
    p.x = reinterpret_cast<const uint16_t*>(x) + (size_t)t * shape->hidden;
    if (fused) {
      const size_t o = (size_t)t * shape->top_k;
      p.logits = fused->logits + (size_t)t * shape->n_experts;
      p.ids_out = fused->ids_out ? fused->ids_out + o : nullptr;
      p.prec_out = fused->prec_out ? fused->prec_out + o : nullptr;
      p.weights_out = fused->weights_out ? fused->weights_out + o : nullptr;
    } else {
      p.ids = ids + (size_t)t * shape->top_k;
      p.prec = prec + (size_t)t * shape->top_k;
      p.weights = weights + (size_t)t * shape->top_k;
    }
    p.y = y + (size_t)t * shape->hidden;
    if (fused) {
      if (shape->group == 128) rc = launch_decode<128, true>(p, dev, sms, 0, st);
      else if (shape->group == 64) rc = launch_decode<64, true>(p, dev, sms, 1, st);
      else rc = launch_decode<32, true>(p, dev, sms, 2, st);
    } else {
      if (shape->group == 128) rc = launch_decode<128, false>(p, dev, sms, 0, st, coop);
      else if (shape->group == 64) rc = launch_decode<64, false>(p, dev, sms, 1, st, coop);
      else rc = launch_decode<32, false>(p, dev, sms, 2, st, coop);
    }
    if (rc != SLICEMOE_OK) return rc;
  }
  return SLICEMOE_OK;
}

}  // namespace slicemoe

using namespace slicemoe;

extern "C" int slicemoe_trace_read(long long* out_host, int max_ctas, int* slots_out) {
#ifdef SLICEMOE_TRACE
  if (!out_host || max_ctas <= 0) return SLICEMOE_E_INVALID_ARG;
  if (slots_out) *slots_out = kTraceSlots;
  const size_t n = (size_t)(max_ctas < 256 ? max_ctas : 256) * kTraceSlots * sizeof(long long);
  SM_CUDA_TRY(cudaMemcpyFromSymbol(out_host, g_trace, n));
  return SLICEMOE_OK;
#else
  (void)out_host;
  (void)max_ctas;
  (void)slots_out;
  return SLICEMOE_E_UNSUPPORTED;  // this build carries no time stamps
#endif
}

extern "C" size_t slicemoe_workspace_bytes(const slicemoe_shape* shape) {
  if (check_shape(shape) != SLICEMOE_OK) return kWsBytes;
  const long long hsum = (long long)shape->top_k * shape->inter + (long long)shape->n_shared * shape->shared_inter;
  if (hsum > kHCap) return kWsBytes;
  return kWsBatchOff + batch_workspace_bytes(shape, shape->n_shared) + kWsListBytes;
}

extern "C" int slicemoe_workspace_init(void* workspace, size_t workspace_bytes, void* stream) {
  if (!workspace || workspace_bytes < kWsBytes || (reinterpret_cast<uintptr_t>(workspace) & 255))
    return SLICEMOE_E_INVALID_ARG;
  // header to zero, both h buffers to "empty" (every byte 0xff: see kHEmpty)
  SM_CUDA_TRY(cudaMemsetAsync(workspace, 0, kWsHOff, (cudaStream_t)stream));
  SM_CUDA_TRY(cudaMemsetAsync(reinterpret_cast<uint8_t*>(workspace) + kWsHOff, 0xff, 2 * sizeof(float) * kHCap,
                              (cudaStream_t)stream));
  return SLICEMOE_OK;
}

extern "C" int slicemoe_workspace_set_wait(void* workspace, unsigned long long wait_cycles, unsigned extra_arrivals,
                                           void* stream) {
  if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255)) return SLICEMOE_E_INVALID_ARG;
  WsHeader* h = reinterpret_cast<WsHeader*>(workspace);
  cudaStream_t st = (cudaStream_t)stream;
  // small host-to-device copies from pageable memory are staged by the runtime before the call returns
  SM_CUDA_TRY(cudaMemcpyAsync(&h->wait_cycles, &wait_cycles, sizeof(wait_cycles), cudaMemcpyHostToDevice, st));
  SM_CUDA_TRY(cudaMemcpyAsync(&h->extra_arrivals, &extra_arrivals, sizeof(extra_arrivals), cudaMemcpyHostToDevice, st));
  return SLICEMOE_OK;
}

extern "C" int slicemoe_get_status(void* workspace, int* status_out, void* stream) {
  if (!workspace || !status_out) return SLICEMOE_E_INVALID_ARG;
  WsHeader* h = reinterpret_cast<WsHeader*>(workspace);
  unsigned v = 0;
  cudaStream_t st = (cudaStream_t)stream;
  SM_CUDA_TRY(cudaMemcpyAsync(&v, &h->status, sizeof(v), cudaMemcpyDeviceToHost, st));
  SM_CUDA_TRY(cudaMemsetAsync(&h->status, 0, sizeof(unsigned), st));
  SM_CUDA_TRY(cudaStreamSynchronize(st));
  *status_out = (int)v;
  return SLICEMOE_OK;
}

extern "C" int slicemoe_expert_ffn(const slicemoe_shape* shape, const slicemoe_expert* experts, const void* x, int T,
                                   const int32_t* ids, const uint8_t* prec, const float* weights, float* y,
                                   void* workspace, size_t workspace_bytes, void* stream) {
  return run_layer(shape, experts, nullptr, 0, nullptr, x, T, ids, prec, weights, y, workspace, workspace_bytes,
                   stream);
}

extern "C" int slicemoe_layer(const slicemoe_shape* shape, const slicemoe_expert* experts,
                              const slicemoe_expert* shared, const float* shared_gate_vec, const void* x, int T,
                              const int32_t* ids, const uint8_t* prec, const float* weights, float* y,
                              void* workspace, size_t workspace_bytes, void* stream) {
  if (!shape) return SLICEMOE_E_INVALID_ARG;
  return run_layer(shape, experts, shared, shape->n_shared, shared_gate_vec, x, T, ids, prec, weights, y, workspace,
                   workspace_bytes, stream);
}

extern "C" int slicemoe_layer_flags(const slicemoe_shape* shape, const slicemoe_expert* experts,
                                    const slicemoe_expert* shared, const float* shared_gate_vec, const void* x, int T,
                                    const int32_t* ids, const uint8_t* prec, const float* weights, float* y,
                                    void* workspace, size_t workspace_bytes, unsigned flags, void* stream) {
  if (!shape) return SLICEMOE_E_INVALID_ARG;
  return run_layer(shape, experts, shared, shape->n_shared, shared_gate_vec, x, T, ids, prec, weights, y, workspace,
                   workspace_bytes, stream, nullptr, flags);
}

extern "C" int slicemoe_layer_routed(const slicemoe_shape* shape, const slicemoe_expert* experts,
                                     const slicemoe_expert* shared, const float* shared_gate_vec, const void* x, int T,
                                     const float* logits, const float* bias, int renorm, float tau, int rank_high,
                                     int32_t* ids_out, uint8_t* prec_out, float* weights_out, float* y,
                                     void* workspace, size_t workspace_bytes, void* stream) {
  if (!shape) return SLICEMOE_E_INVALID_ARG;
  FusedRouting f;
  f.logits = logits;
  f.bias = bias;
  f.renorm = renorm;
  f.rank_high = rank_high;
  f.tau = tau;
  f.ids_out = ids_out;
  f.prec_out = prec_out;
  f.weights_out = weights_out;
  return run_layer(shape, experts, shared, shape->n_shared, shared_gate_vec, x, T, nullptr, nullptr, nullptr, y, workspace,
                   workspace_bytes, stream, &f);
}

namespace slicemoe {
// A caller's host buffer and where the device sees it.  Every page is asked about: of a buffer that is registered in part a
// kernel would touch pages that the device does not have (a copy of it fails as well, so such a call is refused).
struct HostBuffer {
  uint8_t* dev = nullptr;  // null: not registered
  bool look(const void* host, size_t bytes) {
    constexpr uintptr_t kPage = 4096;
    const uintptr_t at = reinterpret_cast<uintptr_t>(host);
    for (uintptr_t p = at; p < at + bytes; p = (p | (kPage - 1)) + 1) {
      cudaPointerAttributes attr;
      uint8_t* d = nullptr;
      if (cudaPointerGetAttributes(&attr, reinterpret_cast<const void*>(p)) != cudaSuccess) (void)cudaGetLastError();  // not registered
      else if (attr.type == cudaMemoryTypeHost && attr.devicePointer) d = static_cast<uint8_t*>(attr.devicePointer);
      if (p == at) dev = d;
      else if (d != (dev ? dev + (p - at) : nullptr)) return false;
    }
    return true;
  }
  bool mapped(unsigned align) const { return dev && (reinterpret_cast<uintptr_t>(dev) & (align - 1)) == 0; }
};
// Everything of a host step but its last synchronisation, on checked arguments.
static int enqueue_host_step(const slicemoe_shape* shape, const slicemoe_expert* experts, const slicemoe_expert* shared,
                             const float* shared_gate_vec, const void* x_host, const float* logits_host, const float* bias,
                             int renorm, float tau, int rank_high, float* y_host, void* workspace, size_t workspace_bytes,
                             void* stream) {
  uint8_t* ws = reinterpret_cast<uint8_t*>(workspace);
  cudaStream_t st = (cudaStream_t)stream;
  void* dx = ws + kWsStX;
  // logits_host == NULL: the logits follow x in the caller's buffer (x_host is bf16 [hidden] then float32 [E]) and
  // in the staging area alike, and one copy brings both
  float* dlogits = reinterpret_cast<float*>(logits_host ? ws + kWsStLogits : ws + kWsStX + 2 * (size_t)shape->hidden);
  int32_t* dids = reinterpret_cast<int32_t*>(ws + kWsStIds);
  float* dw = reinterpret_cast<float*>(ws + kWsStW);
  uint8_t* dprec = ws + kWsStPrec;
  float* dy = reinterpret_cast<float*>(ws + kWsStY);
  // y_host in pinned (device-mapped) host memory: the kernel writes its 16 output rows per CTA straight
  // into it and the copy back falls away; otherwise y goes through the staging area.  x and the logits likewise are read
  // where they are.
  const size_t x_bytes = 2 * (size_t)shape->hidden, logits_bytes = 4 * (size_t)shape->n_experts;
  HostBuffer hy, hx, hl;
  if (!hy.look(y_host, 4 * (size_t)shape->hidden) || !hx.look(x_host, x_bytes) ||
      !hl.look(logits_host ? static_cast<const void*>(logits_host) : static_cast<const uint8_t*>(x_host) + x_bytes, logits_bytes))
    return SLICEMOE_E_INVALID_ARG;
  const bool y_direct = hy.mapped(16);
  if (y_direct) dy = reinterpret_cast<float*>(hy.dev);
  const void* x_mapped = hx.dev;
  const float* logits_mapped = hx.mapped(4) && hl.mapped(4) ? reinterpret_cast<const float*>(hl.dev) : nullptr;
  if (logits_mapped) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1);
    cfg.blockDim = dim3(kStageThreads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    SM_CUDA_TRY(cudaLaunchKernelEx(&cfg, stage_step_kernel, reinterpret_cast<const uint32_t*>(x_mapped), logits_mapped, (int)shape->hidden,
                                   (int)shape->n_experts, (int)shape->top_k, bias, renorm, tau, rank_high,
                                   reinterpret_cast<uint32_t*>(dx), dids, dw, dprec));
    const int rc = slicemoe_layer(shape, experts, shared, shared_gate_vec, dx, 1, dids, dprec, dw, dy, workspace, workspace_bytes, stream);
    if (rc != SLICEMOE_OK) return rc;
    if (!y_direct) SM_CUDA_TRY(cudaMemcpyAsync(y_host, dy, 4 * (size_t)shape->hidden, cudaMemcpyDeviceToHost, st));
    return SLICEMOE_OK;
  }
  if (logits_host) {
    SM_CUDA_TRY(cudaMemcpyAsync(dx, x_host, 2 * (size_t)shape->hidden, cudaMemcpyHostToDevice, st));
    SM_CUDA_TRY(cudaMemcpyAsync(dlogits, logits_host, 4 * (size_t)shape->n_experts, cudaMemcpyHostToDevice, st));
  } else {
    SM_CUDA_TRY(cudaMemcpyAsync(dx, x_host, 2 * (size_t)shape->hidden + 4 * (size_t)shape->n_experts,
                                cudaMemcpyHostToDevice, st));
  }
  const int rc = slicemoe_layer_routed(shape, experts, shared, shared_gate_vec, dx, 1, dlogits, bias, renorm, tau, rank_high, dids,
                                       dprec, dw, dy, workspace, workspace_bytes, stream);
  if (rc != SLICEMOE_OK) return rc;
  if (!y_direct) SM_CUDA_TRY(cudaMemcpyAsync(y_host, dy, 4 * (size_t)shape->hidden, cudaMemcpyDeviceToHost, st));
  return SLICEMOE_OK;
}
}  // namespace slicemoe

extern "C" int slicemoe_decode_step_host(const slicemoe_shape* shape, const slicemoe_expert* experts,
                                         const slicemoe_expert* shared, const float* shared_gate_vec,
                                         const void* x_host, const float* logits_host, const float* bias, int renorm,
                                         float tau, int rank_high, float* y_host, void* workspace,
                                         size_t workspace_bytes, void* stream) {
  int rc = check_shape(shape);
  if (rc != SLICEMOE_OK) return rc;
  if (!x_host || !y_host || !workspace || workspace_bytes < kWsBytes) return SLICEMOE_E_INVALID_ARG;
  if (shape->n_experts > 512) return SLICEMOE_E_UNSUPPORTED;
  if (!experts) return SLICEMOE_E_INVALID_ARG;
  // all that the layer call would refuse is refused before a kernel that reads the caller's buffers is enqueued
  int dev, sms;
  rc = check_layer(shape, shared, shape->n_shared, shared_gate_vec, static_cast<uint8_t*>(workspace) + kWsStX, workspace, workspace_bytes,
                   &dev, &sms);
  if (rc != SLICEMOE_OK) return rc;
  rc = enqueue_host_step(shape, experts, shared, shared_gate_vec, x_host, logits_host, bias, renorm, tau, rank_high, y_host, workspace,
                         workspace_bytes, stream);
  // also after an error: the caller may free its buffers when the call returns, and part of the step may be enqueued
  const cudaError_t e = cudaStreamSynchronize((cudaStream_t)stream);
  if (rc == SLICEMOE_OK) SM_CUDA_TRY(e);
  return rc;
}

// ---- entry point for callers that cannot allocate -----------------------------------------------------
// The scratch that slicemoe_layer takes from the caller lives here, in the library image: kWsBytes bytes
// per GPU that loads the library, held until the process exits.
namespace slicemoe {
static __device__ __align__(256) unsigned char g_static_scratch[kWsBytes];
static void* g_static_scratch_ptr[64];  // device address of the array, per device, resolved once
}  // namespace slicemoe

extern "C" int slicemoe_layer_static(const slicemoe_shape* shape, const slicemoe_expert* experts,
                                     const slicemoe_expert* shared, const float* shared_gate_vec, const void* x, int T,
                                     const int32_t* ids, const uint8_t* prec, const float* weights, float* y,
                                     void* stream) {
  if (!shape) return SLICEMOE_E_INVALID_ARG;
  // The built-in scratch has one fixed size; a layer that would need more is refused, never truncated.
  const long long hsum = (long long)shape->top_k * shape->inter +
                         (long long)(shape->n_shared > 0 ? shape->n_shared : 0) * shape->shared_inter;
  if (shape->hidden > kMaxHidden || hsum > kHCap) return SLICEMOE_E_UNSUPPORTED;
  int dev = 0;
  SM_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return SLICEMOE_E_UNSUPPORTED;
  if (!g_static_scratch_ptr[dev]) {
    // In host code the array's name is only a handle; the address a kernel can use has to be asked for,
    // with the device that will run the kernel current.
    void* ptr = nullptr;
    SM_CUDA_TRY(cudaGetSymbolAddress(&ptr, g_static_scratch));
    if (!ptr) return SLICEMOE_E_CUDA;
    g_static_scratch_ptr[dev] = ptr;
  }
  void* ws = g_static_scratch_ptr[dev];
  // The array keeps whatever the previous call left: the header (launch count, status) must start at zero, and the
  // h buffer the first launch then uses must be empty (the launches clear the other one for their successors).
  SM_CUDA_TRY(cudaMemsetAsync(ws, 0, kWsHOff, (cudaStream_t)stream));
  SM_CUDA_TRY(cudaMemsetAsync(reinterpret_cast<uint8_t*>(ws) + kWsHOff, 0xff, sizeof(float) * kHCap, (cudaStream_t)stream));
  return run_layer(shape, experts, shared, shape->n_shared, shared_gate_vec, x, T, ids, prec, weights, y, ws, kWsBytes,
                   stream);
}
