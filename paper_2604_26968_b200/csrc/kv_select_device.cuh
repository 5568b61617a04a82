// Device-side pieces shared by the selection kernels.
#pragma once
#include "kvtier_internal.cuh"

namespace kvt {

// 32-bit keys whose unsigned order is the order of the scores; NaNs (a caller's array may hold them)
// are ordered by their bits, below -inf or above +inf.  -0.0 orders with +0.0, so the key 0x7FFFFFFF
// (its own bit pattern's) never occurs and stands for an entry that is no candidate.
constexpr uint32_t kKeyExcluded = 0x7FFFFFFFu;
constexpr uint32_t kKeyNegInf = 0x007FFFFFu, kKeyPosInf = 0xFF800000u;

__device__ __forceinline__ uint32_t key_of_bits(uint32_t b) {
  return b ^ ((uint32_t)((int32_t)b >> 31) | 0x80000000u);
}
__device__ __forceinline__ uint32_t score_key(float s) {
  const uint32_t b = __float_as_uint(s);
  return key_of_bits(b == 0x80000000u ? 0u : b);
}
// The same, in fewer instructions, of a number or of a NaN that arithmetic gave.
__device__ __forceinline__ uint32_t number_key(float s) {
  return key_of_bits(__float_as_uint(__fadd_rn(s, 0.0f)));   // -0.0 + 0.0 = +0.0; every other value is itself
}

// The score with a given key (keys of -inf .. +inf).
__device__ __forceinline__ float key_score(uint32_t key) {
  return __uint_as_float((key & 0x80000000u) ? key & 0x7FFFFFFFu : ~key);
}

__device__ __forceinline__ uint32_t warp_scan_incl(uint32_t v, uint32_t lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, v, o);
    if (lane >= (uint32_t)o) v += y;
  }
  return v;
}

// Bit l of the low byte of x moves to bit 4*l.
__device__ __forceinline__ uint32_t spread8(uint32_t x) {
  x &= 0xFFu;
  x = (x | x << 12) & 0x000F000Fu;
  x = (x | x << 6) & 0x03030303u;
  return (x | x << 3) & 0x11111111u;
}

// Bit 4*l + q of the result is bit l of the q-th argument (low bytes).
__device__ __forceinline__ uint32_t interleave4(uint32_t x0, uint32_t x1, uint32_t x2, uint32_t x3) {
  return spread8(x0) | spread8(x1) << 1 | spread8(x2) << 2 | spread8(x3) << 3;
}

// Two neighbouring counters in one 64-bit atomic (neither sum reaches 2^32).
__device__ __forceinline__ void add_pair(uint32_t* counters, uint2 c) {
  if (c.x | c.y)
    atomicAdd(reinterpret_cast<unsigned long long*>(counters), (unsigned long long)c.y << 32 | c.x);
}

}  // namespace kvt
