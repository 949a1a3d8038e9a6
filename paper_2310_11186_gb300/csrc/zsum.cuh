// Z as an exact sum: the order in which units or groups finish changes no bit.
//
// A value is held as hi 2^-32 + lo 2^-96 (two 64-bit integers) and added to
// four words that hold 32 bits of it each, so the words' sums cannot pass 2^63
// below 2^31 values.  2^-96 is far below anything that FP32 keeps beside a
// kernel value of 1, and it keeps Z where every pair is far apart and Z is
// nothing but such values: an FP32 partial sum loses bits below 2^-72 only
// (pairs 7e10 apart), and one that is not 0 counts as 2^-96 at least, so Z is
// positive as long as any kernel value is.  (In multiples of 2^-32 a layout of
// 9,000 points 1e5 apart was 1 % off, one of 1,000 points 14 %, and both had a Z
// of 0, so no finite gradient, at 1e9.)
#pragma once

#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

namespace tsgne {

constexpr int kZWords = 4;  // weights 2^-96, 2^-64, 2^-32, 1

struct ZSum {
  unsigned long long hi = 0ull, lo = 0ull;
  __host__ __device__ __forceinline__ void add(ZSum v) {
    lo += v.lo;
    hi += v.hi + (lo < v.lo ? 1ull : 0ull);
  }
};

// A partial sum z, 0 <= z < 2^26 (NaN: the caller's check), in two parts: from
// kZWhole on an FP32 value has no bits below 2^-32, so lo is needed only below.
constexpr float kZWhole = 1.0f / 256.0f;
__device__ __forceinline__ unsigned long long z_hi(float z) { return __float2ull_rz(z * 4294967296.0f); }
__device__ __forceinline__ unsigned long long z_lo(float z) {
  const float rest = fmaf(__ull2float_rn(z_hi(z)), -1.0f / 4294967296.0f, z);  // exact: hi has at most 24 bits
  return __float2ull_ru(rest * 7.9228162514264338e28f);                        // 2^96
}
__device__ __forceinline__ ZSum z_fix(double z) {
  ZSum v;
  v.hi = __double2ull_rz(z * 4294967296.0);
  const double rest = fma(__ull2double_rn(v.hi), -1.0 / 4294967296.0, z);
  v.lo = __double2ull_ru(rest * 79228162514264337593543950336.0);  // 2^96
  return v;
}

// Sum over the warp's lanes, hi below 2^58, in every lane.
__device__ __forceinline__ ZSum z_warp_sum(ZSum v) {
  constexpr unsigned full = 0xffffffffu;
  const unsigned long long m = (1ull << 27) - 1;
  ZSum s;
  const unsigned long long a = __reduce_add_sync(full, (uint32_t)(v.hi & m));
  const unsigned long long b = __reduce_add_sync(full, (uint32_t)((v.hi >> 27) & m));
  const unsigned long long c = __reduce_add_sync(full, (uint32_t)(v.hi >> 54));
  s.hi = a + (b << 27) + (c << 54);
  if (__any_sync(full, v.lo != 0ull)) {
    const unsigned long long d = __reduce_add_sync(full, (uint32_t)(v.lo & m));
    const unsigned long long e = __reduce_add_sync(full, (uint32_t)((v.lo >> 27) & m));
    const unsigned long long f = __reduce_add_sync(full, (uint32_t)(v.lo >> 54));
    s.lo = d + (e << 27);
    s.add(ZSum{f >> 10, f << 54});
  }
  return s;
}

// v rounded down to 53 significant bits: what a double holds, so that a unit's
// value is the same bits through a double as without one.
__device__ __forceinline__ ZSum z_top53(ZSum v) {
  if (v.lo == 0ull && v.hi >> 53 == 0ull) return v;
  const int bits = v.hi ? 128 - __clzll((long long)v.hi) : 64 - __clzll((long long)v.lo);
  const int drop = bits - 53;
  if (drop >= 64) {
    v.lo = 0ull;
    v.hi &= ~0ull << (drop - 64);
  } else if (drop > 0) {
    v.lo &= ~0ull << drop;
  }
  return v;
}
// Exact for a value of 53 significant bits.
__device__ __forceinline__ double z_double(ZSum v) {
  return (double)v.hi * (1.0 / 4294967296.0) + (double)v.lo * (1.0 / 79228162514264337593543950336.0);
}

__host__ __device__ __forceinline__ unsigned long long z_word(ZSum v, int k) {
  const unsigned long long half = k < 2 ? v.lo : v.hi;
  return k & 1 ? half >> 32 : half & 0xffffffffull;
}

// Adds v to the words in global memory (one thread).
__device__ __forceinline__ void z_add(unsigned long long* words, ZSum v) {
#pragma unroll
  for (int k = 0; k < kZWords; ++k) {
    const unsigned long long w = z_word(v, k);
    if (w)
      asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(words + k), "l"(w) : "memory");
  }
}

// The sum in the words, less a whole number (NaN if a kernel value was NaN).
__host__ __device__ __forceinline__ double z_value(const unsigned long long* words, uint32_t bad, int less) {
  const unsigned long long w1 = words[1] + (words[0] >> 32), w2 = words[2] + (w1 >> 32), w3 = words[3] + (w2 >> 32);
  const unsigned long long low = (w1 << 32) | (words[0] & 0xffffffffull);
  double part = (double)(w2 & 0xffffffffull) * (1.0 / 4294967296.0);
  if (low) part += (double)low * (1.0 / 79228162514264337593543950336.0);
  return bad ? (double)NAN : (double)((long long)w3 - less) + part;
}

}  // namespace tsgne
