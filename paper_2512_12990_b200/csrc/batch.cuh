// Decode of a small batch of tokens (batch.cu), called by the layer entry points (decode.cu).
#pragma once

#include <stddef.h>
#include <stdint.h>

#include "slicemoe.h"

#ifdef __CUDACC__
#define SM_HD __host__ __device__
#else
#define SM_HD
#endif

namespace slicemoe {

// Tokens of one pass; more are taken in several passes of equal size.
constexpr int kBatchTokens = 16;

constexpr int kBRun = 8;                 // pairs of a run: the columns of an MMA
constexpr int kBChunkK = 2048;           // columns of a down projection's task; wider experts are several
constexpr int kBMaxSegs = 40;            // runs that a CTA's share can touch
constexpr int kBMaxTasks = 640;          // runs of a pass in one projection

// What a 16 x 128 block of a run costs a CTA: the bytes it brings (an MSB tile 2, both slices 4) and its instructions - by
// measurement about half as much again for up to two pairs, the same for more, twice that where pairs of either precision
// meet.  (By bytes alone, CTAs with both-slice runs were done in 21,000 cycles and those with MSB runs in 34,000.)
SM_HD inline unsigned b_block_cost(int n, unsigned high) {
  const unsigned all = (1u << n) - 1u, compute = (n <= 2 ? 1u : 2u) << (high != 0u && (high & all) != all ? 1 : 0);
  return (high ? 4u : 2u) + compute;
}
constexpr unsigned kBFixedCost = 12;  // a row block's own: hand-shakes and the exchange between the four warps

// Whether no CTA's share can touch more runs than its list holds.  Shares are windows of total / sms on the costs of all runs
// one after the other; a pair costs most alone and from both slices, a run least alone and from the MSB slice.  On 148 SMs
// every permitted layer fits with room to spare; on a small part of a device some do not, and take the batch-1 kernel, token
// after token.
inline bool batch_fits(const slicemoe_shape* s, int n_shared, int T, int sms) {
  const int pairs = T * s->top_k, parts = (T + kBRun - 1) / kBRun, n_sh = n_shared * parts;
  unsigned long long total[2] = {0, 0}, least[2] = {~0ull, ~0ull};
  int tasks = 0;
  for (int shared = 0; shared < (n_shared > 0 ? 2 : 1); ++shared) {
    const int inter = shared ? s->shared_inter : s->inter, runs = shared ? n_sh : pairs;
    const unsigned most = shared ? b_block_cost(kBRun, 0xffu) : b_block_cost(1, 1u), low = shared ? b_block_cost(1, 1u) : b_block_cost(1, 0u);
    auto add = [&](int phase, unsigned blocks, unsigned rows) {
      const unsigned long long lo = (unsigned long long)(low * blocks + kBFixedCost) * rows;
      total[phase] += (unsigned long long)runs * (most * blocks + kBFixedCost) * rows;
      if (lo < least[phase]) least[phase] = lo;
    };
    add(0, 2u * (s->hidden / 128), inter / 16);
    for (int c0 = 0; c0 < inter; c0 += kBChunkK) {
      add(1, (inter - c0 < kBChunkK ? inter - c0 : kBChunkK) / 128, s->hidden / 16);
      tasks += runs;
    }
  }
  for (int phase = 0; phase < 2; ++phase)
    if (total[phase] / sms / least[phase] + 3 > (unsigned long long)kBMaxSegs) return false;
  return tasks <= kBMaxTasks;
}

// What the workspace header offers to the batch kernels.
struct BatchControl {
  unsigned* status;
  const unsigned* extra_arrivals;         // != 0: no weights are brought, so that the waits for them run out, and y is not written
  const unsigned long long* wait_cycles;  // limit of the device-side waits, 0 = the default
};

// Workspace of a pass, beyond what the batch-1 kernel takes.
size_t batch_workspace_bytes(const slicemoe_shape* s, int n_shared);

// One pass of T <= kBatchTokens tokens on checked arguments; `ws` has batch_workspace_bytes() bytes, 256-byte aligned.
int batch_layer(const slicemoe_shape* s, const slicemoe_expert* experts, const slicemoe_expert* shared, int n_shared,
                const float* gate_vec, const uint16_t* x, int T, const int32_t* ids, const uint8_t* prec, const float* weights,
                float* y, void* ws, const BatchControl& ctl, int sms, void* stream);

}  // namespace slicemoe
