// DFTs of up to 32 points in registers, shared by the level kernels and the
// QFT^-1 passes. Internal; not part of the ABI.
#pragma once

#include "qpe_internal.cuh"

namespace qpe {

// v exp(-2 pi i K / 32) for a compile-time K in 0 .. 15 after unrolling: nothing
// for 0, an exchange for 8, else a product and an FMA for each part. For 4 and 12
// (x +- y) cos(pi / 4) takes as many operations and rounds the sum before the product. In
// complex64 that is 2 to 4% more rms error of a DFT of 8 to 32 points, and it is not used;
// in complex128 the exact 0 of K = 8 gains more than it loses, and the FP64 units run it
// faster (QFT^-1 over 2^20 points of Nmat 6: 160 us with products and FMAs, 150 so).
template <typename C>
__host__ __device__ __forceinline__ C rot32(C v, int K) {
  using R_t = typename real_of<C>::type;
  constexpr double cs[9] = {1.0,
                            0.98078528040323044913,  // cos(pi k / 16)
                            0.92387953251128675613,
                            0.83146961230254523708,
                            0.70710678118654752440,
                            0.55557023301960222474,
                            0.38268343236508977173,
                            0.19509032201612826785,
                            0.0};
  if (K == 0) return v;
  if (K == 8) return mk(v.y, -v.x);
  if constexpr (sizeof(C) == 16) {
    const R_t c4 = (R_t)cs[4];
    if (K == 4) return mk((v.x + v.y) * c4, (v.y - v.x) * c4);
    if (K == 12) return mk((v.y - v.x) * c4, -((v.x + v.y) * c4));
  }
  const R_t c = (R_t)(K < 8 ? cs[K & 7] : -cs[(16 - K) & 7]), s = (R_t)(K < 8 ? cs[8 - (K & 7)] : cs[K & 7]);
  // s = sin(pi K / 16): cos(pi (8 - K) / 16) for K < 8, cos(pi (K - 8) / 16) above
  return mk(fma(v.x, c, v.y * s), fma(v.y, c, -(v.x * s)));
}

// X[k] = sum_n x[n] exp(-2 pi i n k / 2^K) of x[0 .. 2^K), natural order in and out
template <typename C, int K, int N>
__host__ __device__ __forceinline__ void dft_k(C (&x)[N]) {
  constexpr int R = 1 << K;
#pragma unroll
  for (int s = 0; s < K; ++s) {
    const int h = R >> (s + 1);
#pragma unroll
    for (int g = 0; g < R; g += 2 * h) {
#pragma unroll
      for (int p = 0; p < h; ++p) {
        const C u = x[g + p], v = x[g + p + h];
        x[g + p] = cadd(u, v);
        x[g + p + h] = rot32(csub(u, v), p * (32 / (2 * h)));
      }
    }
  }
#pragma unroll
  for (int i = 0; i < R; ++i) {
    int rv = 0;
#pragma unroll
    for (int b = 0; b < K; ++b) rv |= ((i >> b) & 1) << (K - 1 - b);
    if (rv > i) {
      const C t = x[i];
      x[i] = x[rv];
      x[rv] = t;
    }
  }
}

// A butterfly's difference times its twiddle, in a table-driven transform. complex64:
// the roundings are written out, so that they do not depend on how the surrounding code is
// compiled.
__device__ __forceinline__ float2 twiddled(float2 d, float2 w) {
  return mk(__fmaf_rn(d.x, w.x, -__fmul_rn(d.y, w.y)), __fmaf_rn(d.y, w.x, __fmul_rn(d.x, w.y)));
}
__device__ __forceinline__ double2 twiddled(double2 d, double2 w) { return cmul(d, w); }

// The same by radix-2 decimation-in-frequency stages whose twiddles tw(p, s) =
// w^(p 2^s) the caller supplies (stage s pairs points p and p + 2^(K - s - 1) of its
// blocks): as the first K stages of a longer transform, or its last ones.
template <int K, int N, typename Tw>
__device__ __forceinline__ void dft_stages(float2 (&x)[N], Tw tw) {
  using C = float2;
  constexpr int R = 1 << K;
#pragma unroll
  for (int s = 0; s < K; ++s) {
    const int h = R >> (s + 1);
#pragma unroll
    for (int p = 0; p < h; ++p) {
      const C w = tw(p, s);
#pragma unroll
      for (int g = 0; g < R; g += 2 * h) {
        const C u = x[g + p], v = x[g + p + h];
        x[g + p] = cadd(u, v);
        x[g + p + h] = twiddled(csub(u, v), w);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < R; ++i) {
    int rv = 0;
#pragma unroll
    for (int b = 0; b < K; ++b) rv |= ((i >> b) & 1) << (K - 1 - b);
    if (rv > i) {
      const C t = x[i];
      x[i] = x[rv];
      x[rv] = t;
    }
  }
}

}  // namespace qpe
