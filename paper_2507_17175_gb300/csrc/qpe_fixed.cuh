// Integer arithmetic of the fixed-point epilogue. Internal; not part of the ABI.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

namespace qpe {

__host__ __device__ __forceinline__ int clz64(unsigned long long x) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)x);
#else
  return __builtin_clzll(x);
#endif
}
__host__ __device__ __forceinline__ double double_of_bits(unsigned long long x) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)x);
#else
  double v;
  memcpy(&v, &x, sizeof v);
  return v;
#endif
}

// A weight accumulator (bits u of an exact integer |acc| < 2^22 in FP32) plus 1.5 2^23
// in FP32 is exact and has the bits acc + M, M = 0x4B400000.
__host__ __device__ __forceinline__ uint32_t ot_acc_bits(uint32_t u) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(__fadd_rn(__uint_as_float(u), 12582912.0f));
#else
  float f;
  memcpy(&f, &u, sizeof f);
  f += 12582912.0f;
  memcpy(&u, &f, sizeof u);
  return u;
#endif
}

// The drain's fixed point W = floor(E / 2^9) of one T component from its
// seven weight sums, E = sum_w acc_w 2^(8 (6 - w)), T = 2^(tau + sigma - 62) E.
// With b_w = acc_w + M, the low part acc_5 2^8 + acc_6 = b_5 2^8 + b_6 - 257 M
// (exact in int32), and the rest sum_(w<5) b_w 2^(8 (6 - w) - 9) minus
// M sum_(w<5) 2^(8 (6 - w) - 9), modulo 2^64 (W itself fits).
constexpr int kOtFix = 9;  // W's unit in E's
__host__ __device__ __forceinline__ long long ot_weights_fix(uint32_t u0, uint32_t u1, uint32_t u2, uint32_t u3,
                                                             uint32_t u4, uint32_t u5, uint32_t u6) {
  constexpr unsigned long long kMW = 0xc5c5c5c5a0000000ull;  // M (2^39 + 2^31 + 2^23 + 2^15 + 2^7) mod 2^64
  const int r = (int)(ot_acc_bits(u5) * 256u + ot_acc_bits(u6) - 0x8b400000u) >> kOtFix;  // 257 M mod 2^32
  unsigned long long w = (unsigned long long)(long long)r - kMW;
  w += (unsigned long long)ot_acc_bits(u4) * 128u;
  w += (unsigned long long)ot_acc_bits(u3) * 32768u;
  w += (unsigned long long)ot_acc_bits(u2) * 8388608u;
  w += (unsigned long long)ot_acc_bits(u1) * 2147483648u;
  w += (unsigned long long)(ot_acc_bits(u0) * 128u) << 32;
  return (long long)w;
}

// Sums of squares of up to eight fixed-point X (|X| < 2^61.6): with X = A 2^32 + 2 b + its
// lowest bit, b in [-2^30, 2^30), (A 2^32 + 2 b)^2 = A^2 2^64 + A b 2^34 + b^2 4, each part summed
// by one 32 x 32 + 64-bit multiply-add without error (A^2 < 2^59.2 and |A b| < 2^59.6 stay below
// 2^63 over eight, b^2 reaches it). The lowest bit, half a unit of 2^-52 of the pencil's scale, is one
// the accumulators' sums carry for it: a split at bit 31 keeps it too, at four integer operations
// more a value, and takes the top level from 2.52 to 2.89 ms at Nmeas 24.
// GB300 issues FP64 at 2 lanes a clock and SM, so a conversion and an FP64 FMA for
// every value kept the FP64 pipe 76% busy and were what the top level waited
// for; here the FP64 work is one value per bin and drain thread.
struct OtSquares {
  unsigned long long hh = 0, ll = 0;
  long long hl = 0;
  __host__ __device__ __forceinline__ void add(long long x) {
    const uint32_t lo = (uint32_t)x;
    const int A = (int)(x >> 32) + (int)(lo >> 31);
    const int b = (int)lo >> 1;
    hh += (unsigned long long)((long long)A * A);
    hl += (long long)A * b;
    ll += (unsigned long long)((long long)b * b);
  }
  // the sum as a double, rounded to nearest, by integer operations: all drain warps reach
  // this at the end of a tile, and five FP64 operations a bin there took 10,000 clocks of
  // the SM during which no accumulator was read
  __host__ __device__ __forceinline__ double value() const {
    const unsigned long long mid = (unsigned long long)hl << 34, low = ll << 2;
    const unsigned long long lo = low + mid;
    const unsigned long long hi = hh + (unsigned long long)(hl >> 30) + (ll >> 62) + (lo < low ? 1 : 0);
    const unsigned long long top = hi ? hi : lo;
    if (top == 0) return 0.0;
    const int n = clz64(top);
    const unsigned long long frac = (hi && n) ? (hi << n) | (lo >> (64 - n)) : top << n;  // leading bit at 63
    const unsigned long long exp = (unsigned long long)(1023 + 63 + (hi ? 64 : 0) - n - 1);  // less the leading one
    return double_of_bits((exp << 52) + (frac >> 11) + ((frac >> 10) & 1));
  }
};

}  // namespace qpe
