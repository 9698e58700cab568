// Routing of one token by one warp: softmax + top-k with optional cache-priority bias and precision request
// (Section 4.1: gating scores decide which experts run and which of them matter most).  Shared by the
// stand-alone routing kernel and the decode kernel's fused prologue, so both give the same bits.
//
// Each lane keeps E/32 (<= 16) logits in registers; the softmax uses fp32 expf; selection runs k rounds of a
// warp arg-max on key = logit + bias (one fp32 add, NaN -> -inf) with ties broken towards the lower expert
// index, so the ids are a pure function of the keys.  A decode step waits for this, so what counts is the length of the
// dependent chain: a key is mapped to an integer of the same order, a round is two warp reductions (largest key, lowest
// index that has it), and the k probabilities are worked out side by side at the end.  (Rounds of five shuffle steps
// on (key, index) pairs with the probability in between made a decode step of two launches 20.8 us; this way 19.6.)
#pragma once

#include <math_constants.h>
#include <stdint.h>

namespace slicemoe {

constexpr int ROUTE_MAX_VPT = 16;  // values per lane -> E <= 512

struct RouteSel {  // lane j < k holds selection j
  int id;
  float w;
  uint8_t prec_req;
};

// Where a token's logits are: in global memory, read past L1 (a kernel that is launched early may run on an SM whose L1 still
// holds what the addresses held before), or in shared memory.
struct RouteGlobal {
  const float* row;
  __device__ __forceinline__ float operator[](int e) const { return __ldcg(row + e); }
};
struct RouteShared {
  const float* row;
  __device__ __forceinline__ float operator[](int e) const { return row[e]; }
};

// VPT: values per lane, a compile-time bound with 32 VPT >= E.  The result does not depend on it: a lane's
// values are visited in the same order, only the unrolled loops over absent values are shorter.
template <int VPT, class Row>
__device__ __forceinline__ RouteSel route_warp_vpt(const Row row, int E, int k, const float* bias, int renorm, float tau, int rank_high, int lane) {
  uint32_t key[VPT];  // ordered like the float keys; 0: no such expert, or taken
  float val[VPT];
  float vmax = -CUDART_INF_F;
#pragma unroll
  for (int v = 0; v < VPT; ++v) {
    const int e = v * 32 + lane;
    float l = -CUDART_INF_F;
    key[v] = 0u;
    if (e < E) {
      const float raw = row[e];
      l = isnan(raw) ? -CUDART_INF_F : raw;
      float kk = bias ? __fadd_rn(raw, __ldcg(bias + e)) : raw;
      if (isnan(kk)) kk = -CUDART_INF_F;
      const uint32_t b = __float_as_uint(kk + 0.0f);  // both zeros are one key
      key[v] = b ^ ((uint32_t)((int32_t)b >> 31) | 0x80000000u);
    }
    val[v] = l;
    vmax = fmaxf(vmax, l);
  }
  asm("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(vmax) : "f"(vmax));
  float sum = 0.0f;
#pragma unroll
  for (int v = 0; v < VPT; ++v) {
    const int e = v * 32 + lane;
    if (e < E) sum += expf(val[v] - vmax);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
  const float inv_sum = 1.0f / sum;

  int idsel = 0;  // lane j keeps selection j (k <= 16 < 32)
  for (int j = 0; j < k; ++j) {
    uint32_t best = key[0];
    int bv = 0;
#pragma unroll
    for (int v = 1; v < VPT; ++v) {
      if (key[v] > best) {  // ascending e within a lane: strict > keeps the lower index
        best = key[v];
        bv = v;
      }
    }
    const uint32_t top = __reduce_max_sync(0xffffffffu, best);
    const int e = (int)__reduce_min_sync(0xffffffffu, best == top ? (uint32_t)(bv * 32 + lane) : 0xffffffffu);
#pragma unroll
    for (int v = 0; v < VPT; ++v)
      if (e == v * 32 + lane) key[v] = 0u;
    if (lane == j) idsel = e;
  }
  float sel_val = 0.0f;  // the selection's logit, from the lane that holds it
#pragma unroll
  for (int v = 0; v < VPT; ++v) {
    const float got = __shfl_sync(0xffffffffu, val[v], idsel & 31);
    if ((idsel >> 5) == v) sel_val = got;
  }
  const float p = lane < k ? expf(sel_val - vmax) * inv_sum : 0.0f;
  float total = 1.0f;
  if (renorm) {  // added up in selection order
    total = 0.0f;
    for (int j = 0; j < k; ++j) total += __shfl_sync(0xffffffffu, p, j);
  }
  RouteSel sel;
  sel.id = idsel;
  sel.w = renorm ? p / total : p;
  sel.prec_req = (uint8_t)((p >= tau || lane < rank_high) ? 1 : 0);
  return sel;
}

template <class Row>
__device__ __forceinline__ RouteSel route_warp(const Row row, int E, int k, const float* bias, int renorm, float tau, int rank_high, int lane) {
  if (E <= 64) return route_warp_vpt<2>(row, E, k, bias, renorm, tau, rank_high, lane);
  if (E <= 128) return route_warp_vpt<4>(row, E, k, bias, renorm, tau, rank_high, lane);
  return route_warp_vpt<ROUTE_MAX_VPT>(row, E, k, bias, renorm, tau, rank_high, lane);
}

}  // namespace slicemoe
