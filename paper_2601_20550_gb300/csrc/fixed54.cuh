// FP64 products as integer sums: 54-bit fixed point against a common exponent, in limbs of
// 28 and 26 bits (q = hi 2^26 + lo), so that up to 64 products hi x hi and 128 products
// hi x lo sum without rounding in 64 bits.  GB300 issues 2 FP64 operations per clock and SM
// but 32 multiply-adds of 32 x 32 + 64 bits: three per product (lo x lo, at most 2^-58 of
// the largest product each, is dropped).  Errors are relative to the largest of the values
// that share the exponent.
#pragma once

#include <cuda_runtime.h>

namespace heom {

// x 2^(1076 - top) to the nearest integer below 2^54 in magnitude; top: the largest
// exponent field of the slice (at least 1)
__device__ __forceinline__ int2 fixed54(double x, int top) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int e = (int)(u >> 52) & 0x7ff, sh = min(top - max(e, 1), 63);
  const unsigned long long m = ((u & 0xfffffffffffffull) | (e ? 1ull << 52 : 0ull)) << 1;
  const long long r = (long long)((m + ((1ull << sh) >> 1)) >> sh), q = (long long)u < 0 ? -r : r;
  const int hi = (int)((q + (1 << 25)) >> 26);
  return make_int2(hi, (int)(q - ((long long)hi << 26)));
}

// re hi, re lo, im hi, im lo
__device__ __forceinline__ int4 fixed54(double2 z, int top) {
  const int2 a = fixed54(z.x, top), b = fixed54(z.y, top);
  return make_int4(a.x, a.y, b.x, b.y);
}

__device__ __forceinline__ int exponent(double2 z) {
  return max(__double2hiint(z.x) & 0x7ff00000, __double2hiint(z.y) & 0x7ff00000) >> 20;
}

__device__ __forceinline__ double pow2(int n) {   // 2^n, -1074 <= n <= 1023
  return n < -1022 ? __longlong_as_double(1ll << (n + 1074)) : __longlong_as_double((long long)(n + 1023) << 52);
}

// Sums in units of the two operands' fixed points, ea and eb their largest exponents.
struct Unit54 {
  double f1, f2;
  bool deep;
  __device__ __forceinline__ Unit54(int ea, int eb) {
    const int n = ea + eb - 2 * 1076 + 52;
    f1 = ea < 0x7ff && eb < 0x7ff ? pow2(n / 2) : __longlong_as_double(0x7ff8000000000000ll);
    f2 = pow2(n - n / 2);
    deep = n <= -1000 || n >= 900;
    if (!deep) f1 *= f2;
  }
  // s + (hh + hl 2^-26) units
  __device__ __forceinline__ double add(long long hh, long long hl, double s) const {
    const double v = __ll2double_rn(hh + ((hl + (1ll << 25)) >> 26));
    return deep ? fma(v * f1, f2, s) : fma(v, f1, s);
  }
};

}  // namespace heom
