// Decode of a small batch of tokens (batch.cu), called by the layer entry points (decode.cu).
#pragma once

#include <stddef.h>
#include <stdint.h>

#include "slicemoe.h"

namespace slicemoe {

// Tokens of one pass; more are taken in several passes of equal size.
constexpr int kBatchTokens = 16;

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
