// slicemoe_pack: AMAT quantiser + MSB/LSB slice planes in the tiled layout, and the inverse hooks.
//
// One kernel per matrix, which reads W once.  A warp owns rows g and g + 8 of a 16-row block over 128 columns: lane l
// holds columns 4 l .. 4 l + 3 of both rows, which are the eight weights of one 32-bit word of each plane, and the
// groups are 8, 16 or 32 consecutive lanes, so that the range of a group is two warp reductions and the codes never
// leave the registers.  The eight warps of a block (g = 0 .. 7) fill whole 512-byte plane blocks.  Bound: HBM, 5
// bytes per weight.  Every integer is that of IEEE division and rint (a reciprocal only where it provably
// rounds to the same integer, see quantise_one), so the codes are bit-exact against a float32 CPU evaluation.
// Measured on a 1408 x 2048 matrix, G 128 (14.5 MB, 2.2 us at the copy rate): two kernels - range and meta first, then
// planes from a second read of W - 16 us; this one 5.8 us back to back (load latency, the chain of reductions and
// divides, and the hand-over from launch to launch; a larger matrix comes closer to the rate).
#include <cuda_fp16.h>

#include "common.cuh"

namespace slicemoe {

// clamp(rint(w / s) + z, 0, qmax) with the IEEE quotient.  w times the rounded reciprocal r is within 2^-22 of the
// quotient, relatively, so wherever the product is below 1024 in size and farther than 2^-10 from a half-integer its
// nearest integer is the quotient's; the others (one weight in five hundred, and whatever is not a number) divide.
__device__ __forceinline__ int quantise_one(float w, float s, float r, int z, int qmax) {
  const float t = w * r;
  const float big = t + 12582912.f;  // 1.5 x 2^23: the sum's unit is 1, so it is rounded to the nearest even integer
  const float frac = fabsf(t - (big - 12582912.f));
  int n = __float_as_int(big) - 0x4b400000;
  if (!(fabsf(t) < 1024.f && frac < 0.5f - 0.0009765625f)) {
    const float d = fminf(fmaxf(rintf(__fdiv_rn(w, s)), -1.0e9f), 1.0e9f);
    n = (int)d;
  }
  return min(max(n + z, 0), qmax);
}

// Smallest / largest of the float over the lanes of `mask` (which all call it); NaNs lose, as in fminf / fmaxf.
__device__ __forceinline__ float lanes_min(unsigned mask, float v) {
  float r;
  asm volatile("redux.sync.min.f32 %0, %1, %2;" : "=f"(r) : "f"(v), "r"(mask));
  return r;
}
__device__ __forceinline__ float lanes_max(unsigned mask, float v) {
  float r;
  asm volatile("redux.sync.max.f32 %0, %1, %2;" : "=f"(r) : "f"(v), "r"(mask));
  return r;
}

constexpr int kPackThreads = 256;  // eight warps: the row pairs (g, g + 8) of one 16-row block
constexpr int kPackBlocks = 2;     // 128-column blocks of a warp, their loads in flight together
template <int G>
__global__ void __launch_bounds__(kPackThreads) pack_kernel(const float* __restrict__ W, int K, int qmax, int shift,
                                                            uint32_t* __restrict__ msb, uint32_t* __restrict__ lsb,
                                                            uint16_t* __restrict__ scale, uint8_t* __restrict__ zp) {
  const int g = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int kblocks = K >> 7, per_row = (kblocks + kPackBlocks - 1) / kPackBlocks;
  const int rb = (int)(blockIdx.x / (unsigned)per_row), kb0 = (int)(blockIdx.x % (unsigned)per_row) * kPackBlocks;
  constexpr int kLanes = G / 4;  // lanes of a group
  const unsigned mask = kLanes == 32 ? 0xffffffffu : ((1u << (kLanes & 31)) - 1u) << (lane & ~(kLanes - 1));
  asm volatile("griddepcontrol.wait;" ::: "memory");  // W may be the work of the kernel before
  // The kernel behind is not let in early: the layer kernels stream the shared experts' planes ahead of their own wait.  (Three
  // matrices in a graph, us, let in on entry / not: 1408 x 2048 14.66 / 13.25, 2048 x 1408 14.65 / 14.88, 5632 x 2048 42.3 / 41.8,
  // 896 x 2688 18.5 / 18.6, 128 x 256 8.25 / 8.6.)
  float4 v[kPackBlocks][2];
#pragma unroll
  for (int i = 0; i < kPackBlocks; ++i)
#pragma unroll
    for (int hi = 0; hi < 2; ++hi)
    {
      v[i][hi] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (kb0 + i < kblocks)
        v[i][hi] = __ldcs(reinterpret_cast<const float4*>(W + (size_t)(rb * 16 + g + 8 * hi) * K + (kb0 + i) * 128) + lane);
    }
  // The range of every (block, row)'s group in all of its lanes; then lane l works out scale and zero-point for
  // combination l % 4 alone (every four consecutive lanes share a group), and the four take each other's results.
  static_assert(kPackBlocks == 2, "four combinations, one per lane of four");
  float lo_of = 0.f, top_of = 0.f;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const float4 w = v[c >> 1][c & 1];
    const float lo = lanes_min(mask, fminf(fminf(0.f, w.x), fminf(fminf(0.f, w.y), fminf(fminf(0.f, w.z), fminf(0.f, w.w)))));
    const float top = lanes_max(mask, fmaxf(fmaxf(0.f, w.x), fmaxf(fmaxf(0.f, w.y), fmaxf(fmaxf(0.f, w.z), fmaxf(0.f, w.w)))));
    if ((lane & 3) == c) {
      lo_of = lo;
      top_of = top;
    }
  }
  __half s16_of = __float2half_rn(__fdiv_rn(__fsub_rn(top_of, lo_of), (float)qmax));
  float s_of = __half2float(s16_of);
  int z_of = 0;
  if ((top_of == lo_of) || (s_of == 0.0f) || isinf(s_of) || isnan(s_of)) {  // degenerate
    s16_of = __float2half_rn(1.0f);
    s_of = 1.0f;
  } else {
    z_of = (int)fminf(fmaxf(rintf(__fdiv_rn(-lo_of, s_of)), 0.0f), (float)qmax);
  }
  const float r_of = __frcp_rn(s_of);
  if (lane % kLanes < 4) {
    const int c = lane & 3, kb = kb0 + (c >> 1);
    if (kb < kblocks) {
      const size_t idx = ((size_t)rb * (K / G) + kb * (128 / G) + lane / kLanes) * 16 + g + 8 * (c & 1);  // meta_index
      scale[idx] = __half_as_ushort(s16_of);
      zp[idx] = (uint8_t)z_of;
    }
  }
#pragma unroll
  for (int i = 0; i < kPackBlocks; ++i) {
    const int kb = kb0 + i;
    if (kb >= kblocks) break;
    uint32_t code[2];  // four codes of a row, one per byte
#pragma unroll
    for (int hi = 0; hi < 2; ++hi) {
      const int from = (lane & ~3) + 2 * i + hi;
      const float s = __shfl_sync(0xffffffffu, s_of, from), r = __shfl_sync(0xffffffffu, r_of, from);
      const int z = __shfl_sync(0xffffffffu, z_of, from);
      const float vals[4] = {v[i][hi].x, v[i][hi].y, v[i][hi].z, v[i][hi].w};
      uint32_t q[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) q[j] = (uint32_t)quantise_one(vals[j], s, r, z, qmax);
      code[hi] = q[0] | q[1] << 8 | q[2] << 16 | q[3] << 24;
    }
    // a slice narrower than 4 bits sits in the low bits of its nibble; the codes have no bits beyond theirs
    const uint32_t low = ((1u << shift) - 1u) * 0x01010101u;
    // column 4 lane of the 128 is tile lane / 16, word (lane / 4) % 4 of plane lane 4 g + lane % 4
    const size_t word = plane_word_index(K, rb, 2 * kb + (lane >> 4), 4 * g + (lane & 3), (lane >> 2) & 3);
    msb[word] = ((code[0] & ~low) >> shift) | ((code[1] & ~low) >> shift << 4);
    lsb[word] = (code[0] & low) | (code[1] & low) << 4;
  }
}

__global__ void unpack_plane_kernel(const uint32_t* __restrict__ plane, int N, int K,
                                    uint8_t* __restrict__ nibbles) {
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (size_t)N * K) return;
  const int n = (int)(idx / K), k = (int)(idx % K);
  size_t word;
  int pos;
  plane_locate(K, n, k, &word, &pos);
  nibbles[idx] = (uint8_t)((plane[word] >> (4 * pos)) & 15u);
}

__global__ void unpack_meta_kernel(const uint16_t* __restrict__ scale, const uint8_t* __restrict__ zp,
                                   int N, int ngroups, uint16_t* __restrict__ scale_rm,
                                   uint8_t* __restrict__ zp_rm) {
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (size_t)N * ngroups) return;
  const int n = (int)(idx / ngroups), g = (int)(idx % ngroups);
  const size_t mi = meta_index(ngroups, n, g);
  scale_rm[idx] = scale[mi];
  zp_rm[idx] = zp[mi];
}

// Dense storage of a slice narrower than a nibble: the plane's nibbles, in the order of its bytes (low nibble
// first), as a little-endian bit stream of `bits` bits each.  One thread per 32-bit plane word = 8 nibbles =
// `bits` bytes of the stream.
__global__ void compact_plane_kernel(const uint32_t* __restrict__ plane, size_t n_words, int bits,
                                     uint8_t* __restrict__ out) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_words) return;
  const uint32_t w = plane[i], mask = (1u << bits) - 1u;
  uint32_t packed = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) packed |= ((w >> (4 * j)) & mask) << (bits * j);
  for (int b = 0; b < bits; ++b) out[i * bits + b] = (uint8_t)(packed >> (8 * b));
}

__global__ void expand_plane_kernel(const uint8_t* __restrict__ in, size_t n_words, int bits,
                                    uint32_t* __restrict__ plane) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_words) return;
  uint32_t packed = 0;
  for (int b = 0; b < bits; ++b) packed |= (uint32_t)in[i * bits + b] << (8 * b);
  const uint32_t mask = (1u << bits) - 1u;
  uint32_t w = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) w |= ((packed >> (bits * j)) & mask) << (4 * j);
  plane[i] = w;
}

static int check_dims(int N, int K, int group) {
  if (N <= 0 || K <= 0 || (N % 16) != 0 || (K % 128) != 0) return SLICEMOE_E_INVALID_ARG;
  if (!valid_group(group)) return SLICEMOE_E_UNSUPPORTED;
  if ((K % group) != 0) return SLICEMOE_E_INVALID_ARG;
  return SLICEMOE_OK;
}

}  // namespace slicemoe

using namespace slicemoe;

extern "C" size_t slicemoe_plane_bytes(int N, int K) {
  if (N <= 0 || K <= 0) return 0;
  return (size_t)N * K / 2;
}

extern "C" size_t slicemoe_meta_count(int N, int K, int group) {
  if (N <= 0 || K <= 0 || group <= 0) return 0;
  return (size_t)N * (K / group);
}

extern "C" int slicemoe_pack(const float* W, int N, int K, int group, int b_high, int b_low, void* msb,
                             void* lsb, uint16_t* scale, uint8_t* zp, void* stream) {
  if (!W || !msb || !lsb || !scale || !zp) return SLICEMOE_E_INVALID_ARG;
  if (!valid_widths(b_high, b_low)) return SLICEMOE_E_UNSUPPORTED;
  const int qmax = (1 << b_high) - 1, shift = b_high - b_low;
  const int rc = check_dims(N, K, group);
  if (rc != SLICEMOE_OK) return rc;
  // four columns of W a load, a word of a plane a store: elsewhere the kernel would fault
  if ((reinterpret_cast<uintptr_t>(W) & 15) || ((reinterpret_cast<uintptr_t>(msb) | reinterpret_cast<uintptr_t>(lsb)) & 3) ||
      (reinterpret_cast<uintptr_t>(scale) & 1))
    return SLICEMOE_E_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const long long blocks = (long long)(N / 16) * ((K / 128 + kPackBlocks - 1) / kPackBlocks);
  if (blocks > 0x7fffffffll) return SLICEMOE_E_INVALID_ARG;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)blocks);
  cfg.blockDim = dim3(kPackThreads);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // the launch overlaps the end of the work ahead
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  auto* kernel = group == 128 ? pack_kernel<128> : group == 64 ? pack_kernel<64> : pack_kernel<32>;
  SM_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, W, K, qmax, shift, reinterpret_cast<uint32_t*>(msb),
                                 reinterpret_cast<uint32_t*>(lsb), scale, zp));
  return SLICEMOE_OK;
}

extern "C" int slicemoe_unpack_plane(const void* plane, int N, int K, uint8_t* nibbles, void* stream) {
  if (!plane || !nibbles) return SLICEMOE_E_INVALID_ARG;
  if (N <= 0 || K <= 0 || (N % 16) != 0 || (K % 128) != 0) return SLICEMOE_E_INVALID_ARG;
  const size_t total = (size_t)N * K;
  const int threads = 256;
  unpack_plane_kernel<<<(unsigned)((total + threads - 1) / threads), threads, 0, (cudaStream_t)stream>>>(
      reinterpret_cast<const uint32_t*>(plane), N, K, nibbles);
  SM_LAUNCH_CHECK();
  return SLICEMOE_OK;
}

extern "C" int slicemoe_unpack_meta(const uint16_t* scale, const uint8_t* zp, int N, int K, int group,
                                    uint16_t* scale_rm, uint8_t* zp_rm, void* stream) {
  if (!scale || !zp || !scale_rm || !zp_rm) return SLICEMOE_E_INVALID_ARG;
  const int rc = check_dims(N, K, group);
  if (rc != SLICEMOE_OK) return rc;
  const int ngroups = K / group;
  const size_t total = (size_t)N * ngroups;
  const int threads = 256;
  unpack_meta_kernel<<<(unsigned)((total + threads - 1) / threads), threads, 0, (cudaStream_t)stream>>>(
      scale, zp, N, ngroups, scale_rm, zp_rm);
  SM_LAUNCH_CHECK();
  return SLICEMOE_OK;
}

extern "C" size_t slicemoe_compact_bytes(int N, int K, int bits) {
  if (N <= 0 || K <= 0 || bits < 2 || bits > 4) return 0;
  return (size_t)N * K / 8 * bits;
}

static int compact_args(const void* a, const void* b, int N, int K, int bits) {
  if (!a || !b) return SLICEMOE_E_INVALID_ARG;
  if (N <= 0 || K <= 0 || (N % 16) != 0 || (K % 128) != 0) return SLICEMOE_E_INVALID_ARG;
  if (bits < 2 || bits > 4) return SLICEMOE_E_UNSUPPORTED;
  return SLICEMOE_OK;
}

extern "C" int slicemoe_compact_plane(const void* plane, int N, int K, int bits, void* compact, void* stream) {
  const int rc = compact_args(plane, compact, N, K, bits);
  if (rc != SLICEMOE_OK) return rc;
  const size_t n_words = (size_t)N * K / 8;
  const int threads = 256;
  compact_plane_kernel<<<(unsigned)((n_words + threads - 1) / threads), threads, 0, (cudaStream_t)stream>>>(
      reinterpret_cast<const uint32_t*>(plane), n_words, bits, reinterpret_cast<uint8_t*>(compact));
  SM_LAUNCH_CHECK();
  return SLICEMOE_OK;
}

extern "C" int slicemoe_expand_plane(const void* compact, int N, int K, int bits, void* plane, void* stream) {
  const int rc = compact_args(compact, plane, N, K, bits);
  if (rc != SLICEMOE_OK) return rc;
  const size_t n_words = (size_t)N * K / 8;
  const int threads = 256;
  expand_plane_kernel<<<(unsigned)((n_words + threads - 1) / threads), threads, 0, (cudaStream_t)stream>>>(
      reinterpret_cast<const uint8_t*>(compact), n_words, bits, reinterpret_cast<uint32_t*>(plane));
  SM_LAUNCH_CHECK();
  return SLICEMOE_OK;
}
