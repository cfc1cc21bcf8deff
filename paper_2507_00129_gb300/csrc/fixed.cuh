// Exact two-word fixed point shared by the pair kernels that sum runs in 32-bit
// shared-memory words (FP32 shared-memory reductions are emulated on this part
// and far slower).  v (|v| < B) is represented as (hi * 2^16 + lo) * 2^-k with
// q = v * 2^(k-16), hi = floor(q), lo = round((q - hi) * 2^16) in [0, 2^16];
// sc16 = 2^(k-16) is chosen per forest pair so that |q| < 2^21 for every run of
// in-grid pairs.  Sums of hi and of lo are kept in separate 32-bit words (no
// carries between them), which shared memory adds natively.  floor and round
// are FP32 adds of 1.5 * 2^23.
#pragma once

#include "lya_internal.cuh"

namespace lya {

constexpr uint32_t kM15Bits = 0x4B400000u;   // bits of 1.5 * 2^23
constexpr float kM15 = 12582912.0f;
constexpr double kM52 = 6755399441055744.0;  // 1.5 * 2^52

// Two FP32 values in one 64-bit register: one instruction does both lanes'
// fused multiply-adds, each rounded exactly as the scalar one.
using F2 = uint64_t;
__device__ __forceinline__ F2 f2(float lo, float hi) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 unf2(F2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ F2 fma2_rd(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rm.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// Per-pair scale sc16 = 2^(20 - e) with 2^e <= B < 2^(e+1): every |v| < B
// maps to |q| < 2^21.
__device__ __forceinline__ float fixed_scale(float B) {
  if (!(B > 0.f) || !(B < 1e37f)) return 1.f;
  const int e = static_cast<int>((__float_as_uint(B) >> 23) & 0xFFu) - 127;
  const int ex = 20 - e + 127;
  return __uint_as_float(static_cast<uint32_t>(min(max(ex, 1), 254)) << 23);
}

// Knuth's TwoSum: (hi, lo) += x with the rounding error of hi + x kept in lo.
__device__ __forceinline__ void two_sum_add(float& hi, float& lo, float x) {
  const float s = hi + x;
  const float bp = s - hi;
  lo += (hi - (s - bp)) + (x - bp);
  hi = s;
}

// Number of staged pixels whose key (the 32-bit word at `word` of each 16-byte
// record, ascending) lies strictly below v (0 for a NaN).
__device__ __forceinline__ int staged_below(const ulonglong2* a, int word, int n, float v) {
  int lo = 0, hi = n;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (reinterpret_cast<const float*>(a + mid)[word] < v) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// e of a scale 2^e
__device__ __forceinline__ int scale_exponent(float sc) {
  return static_cast<int>((__float_as_uint(sc) >> 23) & 0xFFu) - 127;
}

}  // namespace lya
