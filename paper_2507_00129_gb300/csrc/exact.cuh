// Exact 64-bit integer products and sums for the kernels that work to FP64
// accuracy, on a part with 1.7 FP64 multiply-adds per clock and SM.  Per forest,
// w delta and w become 55-bit integers V = round(v 2^s) = 2^28 H + L (H, L
// signed, at most 2^26 and 2^27); v_i v_j is 2^56 H_i H_j + 2^28 (H_i L_j + L_i H_j),
// three 32 x 32 + 64 bit multiply-adds without rounding (L_i L_j lies below the
// last bit kept).  A run of up to 256 products stays below 2^62.
#pragma once

#include "lya_internal.cuh"

namespace lya {

// 2^e
__device__ __forceinline__ double pow2(int e) {
  return (e < -1022 || e > 1023) ? scalbn(1.0, e) : __longlong_as_double(static_cast<long long>(e + 1023) << 52);
}

// H, L of round(v 2^s), |v| 2^s < 2^54: value = 2^28 H + L, L in [-2^27, 2^27)
__device__ __forceinline__ int2 split55(double v, double scale) {
  const long long q = __double2ll_rn(v * scale);
  const int lo = static_cast<int>(((q + (1ll << 27)) & ((1ll << 28) - 1)) - (1ll << 27));
  return make_int2(static_cast<int>((q - lo) >> 28), lo);
}

struct Sum64 {
  long long nh, nl, wh, wl;  // sums of H H and of H L + L H, of N and of W
};

// Adds the products of two pixels, each (H, L of w delta, H, L of w).
__device__ __forceinline__ void add_products(Sum64& s, const int4& a, const int4& b) {
  s.nh += static_cast<long long>(a.x) * b.x;
  s.nl += static_cast<long long>(a.x) * b.y;
  s.nl += static_cast<long long>(a.y) * b.x;
  s.wh += static_cast<long long>(a.z) * b.z;
  s.wl += static_cast<long long>(a.z) * b.w;
  s.wl += static_cast<long long>(a.w) * b.z;
}

// v / 2^shift to nearest, ties to even (rounding ties up would add a bias
// of 1e-14 to N, whose runs nearly cancel)
__device__ __forceinline__ long long round_shift(long long v, int shift) {
  return (v + ((1ll << (shift - 1)) - 1) + ((v >> shift) & 1)) >> shift;
}

// A run's sum in units of 2^(56 + shift).
__device__ __forceinline__ long long run_value(long long h, long long l, int shift) {
  return round_shift(h + ((l + (1ll << 27)) >> 28), shift);
}

// Sums of N and W in FP64, on the same records (the two FP64 values in place of
// the four integers): for values that lie too far apart for the integers.
struct SumF64 {
  double n, w;
};

__device__ __forceinline__ int4 pack_f64(double n, double w) {
  return make_int4(__double2loint(n), __double2hiint(n), __double2loint(w), __double2hiint(w));
}

__device__ __forceinline__ void add_products(SumF64& s, const int4& a, const int4& b) {
  s.n = fma(__hiloint2double(a.y, a.x), __hiloint2double(b.y, b.x), s.n);
  s.w = fma(__hiloint2double(a.w, a.z), __hiloint2double(b.w, b.z), s.w);
}

// Adds a run's sums to its bin (N, W at a shared-memory address), integers in
// units of 2^(56 + shift).
__device__ __forceinline__ void add_bin64(const Sum64& s, uint32_t addr, int shift) {
  const long long n = run_value(s.nh, s.nl, shift), w = run_value(s.wh, s.wl, shift);
  asm volatile("{\n\tred.shared.add.u64 [%0], %1;\n\tred.shared.add.u64 [%0+8], %2;\n\t}" ::"r"(addr), "l"(n), "l"(w));
}
__device__ __forceinline__ void add_bin64(const SumF64& s, uint32_t addr, int) {
  asm volatile("{\n\tred.shared.add.f64 [%0], %1;\n\tred.shared.add.f64 [%0+8], %2;\n\t}" ::"r"(addr), "d"(s.n), "d"(s.w));
}

}  // namespace lya
