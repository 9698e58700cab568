// Shared by the decode kernels: barrier, bulk copy and integer MMA instructions, and the fixed-point form of activations.
#pragma once

#include <stdint.h>

#include "common.cuh"

namespace slicemoe {

// Every device-side wait is bounded: by this many clock cycles (about 50 ms; a layer takes tens of microseconds)
// unless the workspace header carries another limit.
constexpr unsigned long long kWaitCycles = 100000000ull;

// ---- PTX helpers -------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// The CTA's wait limit sits 8 bytes behind its dead flag.
__device__ __forceinline__ unsigned long long wait_limit(volatile int* dead) {
  return *reinterpret_cast<volatile unsigned long long*>(dead + 2);
}
// Bounded wait.  Returns false (and raises the CTA's dead flag) when the limit is hit or another
// role of this CTA already gave up.
static __device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, volatile int* dead, unsigned* status) {
  const long long t0 = clock64();
  for (;;) {
    for (int i = 0; i < 256; ++i)
      if (mbar_try(bar, parity)) return true;
    if (*dead) return false;
    if ((unsigned long long)(clock64() - t0) > wait_limit(dead)) {
      *dead = 1;
      atomicOr(status, (unsigned)SLICEMOE_STATUS_WAIT_TIMEOUT);
      return false;
    }
  }
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* dead, unsigned* status) {
  if (mbar_try(bar, parity)) return true;
  return mbar_wait_slow(bar, parity, dead, status);
}
// Weights are used once per token: they go through L2 marked evict-first, so that the stream does not push out
// what every launch uses again (the kernel's own instructions, expert tables, h).
__device__ __forceinline__ uint64_t l2_evict_first_policy() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar, uint64_t pol) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(dst),
      "l"(src), "r"(bytes), "r"(bar), "l"(pol)
      : "memory");
}
__device__ __forceinline__ void mma_u8s8(int (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
  asm("mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// d = a * b (no accumulator input: the first step of a chain)
__device__ __forceinline__ void mma_u8s8_first(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                               uint32_t b0, uint32_t b1) {
  const int z = 0;
  asm("mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
      : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "r"(z));
}
// ---- fixed-point activations ---------------------------------------------------------------------
// Byte offset, inside a digit buffer, of digit t of the four values k..k+3 (k % 4 == 0): steps of 32
// columns, 3 digit rows of 32 bytes, and inside a row the order in which the B fragment of m16n8k32 wants
// them: (k % 16) / 4 selects the lane quad position, (k % 32) / 16 the register.
__device__ __forceinline__ int digit_offset(int k, int t) {
  return (k >> 5) * 96 + t * 32 + ((k >> 2) & 3) * 8 + ((k >> 4) & 1) * 4;
}

// Fixed point of four values of a 128-element block (lane L holds elements 4L..4L+3): X = rint(v * 2^e) with
// 2^e * max|v| < 2^22 over the block, split into balanced base-256 digits d0 + 256 d1 + 65536 d2 (each in int8 range; the
// low byte of X read as a signed byte is d0, and so on up), one digit of the four values per word; and 2^-e.
struct BlockDigits {
  uint32_t d0, d1, d2;
  float inv;
};
__device__ __forceinline__ BlockDigits block_digits(const float (&v)[4]) {
  unsigned mb = 0u;  // bit pattern of max |v|: non-negative floats order like their bit patterns
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const unsigned a = __float_as_uint(v[j]) & 0x7fffffffu;
    if (a <= 0x7f800000u) mb = max(mb, a);  // a NaN input gives an undefined result, never a fault
  }
  mb = __reduce_max_sync(0xffffffffu, mb);
  const int ex = (int)(mb >> 23) - 127;  // floor(log2 max) for normal numbers
  const int e = max(-100, min(100, 21 - ex));
  const float scale = __uint_as_float((unsigned)(127 + e) << 23);
  // Z = (X + 0x808080) ^ 0x808080 holds the three digits in its bytes: adding 128 to a byte and flipping its top
  // bit back leaves the byte read as a signed digit, and the carry into the next byte is exactly what remains
  // after taking that digit (X1 = (X + 128) >> 8, and so on up).
  uint32_t Z[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int X = max(-4194304, min(4194304, __float2int_rn(v[j] * scale)));
    Z[j] = (uint32_t)(X + 0x808080) ^ 0x808080u;
  }
  // byte i of each of the four values -> one word (value j in byte j)
  BlockDigits r;
  r.d0 = __byte_perm(__byte_perm(Z[0], Z[1], 0x0040), __byte_perm(Z[2], Z[3], 0x0040), 0x5410);
  r.d1 = __byte_perm(__byte_perm(Z[0], Z[1], 0x0051), __byte_perm(Z[2], Z[3], 0x0051), 0x5410);
  r.d2 = __byte_perm(__byte_perm(Z[0], Z[1], 0x0062), __byte_perm(Z[2], Z[3], 0x0062), 0x5410);
  r.inv = __uint_as_float((unsigned)(127 - e) << 23);
  return r;
}
// Sums of the three digits over the lane's group of G elements (G / 4 consecutive lanes).
template <int G>
__device__ __forceinline__ void group_digit_sums(const BlockDigits& b, int lane, int& s0, int& s1, int& s2) {
  constexpr int lanes_per_group = G / 4;  // 8, 16 or 32 consecutive lanes cover one group
  const unsigned gmask = lanes_per_group == 32 ? 0xffffffffu
                                               : ((1u << lanes_per_group) - 1u) << (lane & ~(lanes_per_group - 1));
  s0 = __reduce_add_sync(gmask, __dp4a((int)b.d0, 0x01010101, 0));  // sums of the signed bytes
  s1 = __reduce_add_sync(gmask, __dp4a((int)b.d1, 0x01010101, 0));
  s2 = __reduce_add_sync(gmask, __dp4a((int)b.d2, 0x01010101, 0));
}
__device__ __forceinline__ void store_digits(const BlockDigits& b, int k, uint8_t* dig) {
  *reinterpret_cast<uint32_t*>(dig + digit_offset(k, 0)) = b.d0;
  *reinterpret_cast<uint32_t*>(dig + digit_offset(k, 1)) = b.d1;
  *reinterpret_cast<uint32_t*>(dig + digit_offset(k, 2)) = b.d2;
}

}  // namespace slicemoe
