// FP64 pieces of the Helmholtz-kernel quadratures (assembly and fields): the
// FP64 pipe is the narrow one, so square roots, reciprocals and sincos are
// written for the ranges these kernels meet.
#pragma once

#include <cuda_runtime.h>

namespace mtf {

#define INV_FOUR_PI 0.079577471545947667884

// (cos x, sin x / x) series in x^2: coefficients of x^(2t)
static __constant__ double c_cos[13] = {1.0, -1.0 / 2, 1.0 / 24, -1.0 / 720, 1.0 / 40320, -1.0 / 3628800, 1.0 / 479001600,
                                 -1.0 / 87178291200.0, 1.0 / 20922789888000.0, -1.0 / 6402373705728000.0,
                                 1.0 / 2432902008176640000.0, -1.0 / 1124000727777607680000.0,
                                 1.0 / 620448401733239439360000.0};
static __constant__ double c_sin[13] = {1.0, -1.0 / 6, 1.0 / 120, -1.0 / 5040, 1.0 / 362880, -1.0 / 39916800,
                                 1.0 / 6227020800.0, -1.0 / 1307674368000.0, 1.0 / 355687428096000.0,
                                 -1.0 / 121645100408832000.0, 1.0 / 51090942171709440000.0,
                                 -1.0 / 25852016738884976640000.0, 1.0 / 15511210043330985984000000.0};

// terms beyond the first of the series above that carry |x| <= xmax to FP64
// rounding (next term below 1e-16); -1: too wide for them
__device__ __forceinline__ int series_degree(float xmax) {
  return xmax <= 0.25f ? 6 : xmax <= 0.5f ? 7 : xmax <= 1.f ? 9 : xmax <= 1.5f ? 10 : xmax <= 2.f ? 12 : -1;
}

// 1 / sqrt(d), d > 0: the hardware approximation refined by one step of the
// cubic Householder iteration y + y e (1/2 + 3/8 e), e = 1 - d y^2
__device__ __forceinline__ double rsqrt_h(double d) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
  const double e = fma(-(d * y), y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}

__device__ __forceinline__ double dot3(const double* a, const double* b) { return fma(a[0], b[0], fma(a[1], b[1], a[2] * b[2])); }
__device__ __forceinline__ void cross3(const double* a, const double* b, double* c) {
  c[0] = fma(a[1], b[2], -(a[2] * b[1]));
  c[1] = fma(a[2], b[0], -(a[0] * b[2]));
  c[2] = fma(a[0], b[1], -(a[1] * b[0]));
}

// sums of N values per lane over groups of 2 off lanes by recursive halving:
// the lane ends with values [base, base + count) of the sums in v[0 ..]
// (start with base = 0, count = N)
template <int N>
__device__ __forceinline__ void halve_sum(double* v, int lane, int off, int& base, int& count) {
  constexpr int H = (N + 1) / 2;
  const bool up = (lane & off) != 0;
#pragma unroll
  for (int i = 0; i < H; ++i) {
    const double lo = v[i], hi = H + i < N ? v[H + i] : 0.0;
    v[i] = (up ? hi : lo) + __shfl_xor_sync(0xffffffffu, up ? lo : hi, off);
  }
  if (up) {
    base += H;
    count = max(0, count - H);
  } else {
    count = min(count, H);
  }
  if constexpr (H > 1) {
    if (off > 1) halve_sum<H>(v, lane, off >> 1, base, count);
  } else {
    for (int o = off >> 1; o > 0; o >>= 1) {  // one value left: plain sums
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
      if (lane & o) count = 0;
    }
  }
}

}  // namespace mtf
