// Complex FFT of a short line held in registers (N = 2, 4, 8, 16 or 32 points,
// natural order in and out):  x[k] <- sum_n x[n] exp(SIGN 2 pi i n k / N).
//
// Radix-2 decimation in time.  The input permutation only renames registers.
// The twiddles 1 and i need no multiplication; every other one is applied as
// w v = f (p + i q) with p, q one fused multiply-add each (f the larger of
// cos and sin, the other as a ratio of at most 1) and f folded into the
// butterfly's sums, so a general butterfly is six fused operations.  A
// 16-point line takes 148 real operations (22 trivial butterflies of 4, 10
// general ones of 6); the plain form with separate complex products takes 168.
#pragma once
#include <cuda_runtime.h>

__host__ __device__ constexpr double fft_cos_first(int m) {   // cos(2 pi m / 32), m = 0..8
  return m == 0 ? 1.0
       : m == 1 ? 0.98078528040323044913
       : m == 2 ? 0.92387953251128675613
       : m == 3 ? 0.83146961230254523708
       : m == 4 ? 0.70710678118654752440
       : m == 5 ? 0.55557023301960222474
       : m == 6 ? 0.38268343236508977173
       : m == 7 ? 0.19509032201612826785
                : 0.0;
}
__host__ __device__ constexpr double fft_cos32(int m) { return m <= 8 ? fft_cos_first(m) : -fft_cos_first(16 - m); }
__host__ __device__ constexpr double fft_sin32(int m) { return fft_cos32(m > 8 ? m - 8 : 8 - m); }   // m = 0..16

// Real arithmetic of the two types; the float form sums complex values as
// packed pairs (one instruction for both components).
__device__ __forceinline__ double2 fft_add(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 fft_sub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 fft_axpy(double f, double2 p, double2 u) {
  return make_double2(fma(f, p.x, u.x), fma(f, p.y, u.y));
}
__device__ __forceinline__ float2 fft_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 fft_sub(float2 a, float2 b) { return __ffma2_rn(make_float2(-1.f, -1.f), b, a); }
__device__ __forceinline__ float2 fft_axpy(float f, float2 p, float2 u) {
  return __ffma2_rn(make_float2(f, f), p, u);
}

// (u, v) <- (u + w v, u - w v), w = exp(SIGN 2 pi i m / 32)
template <int SIGN, typename V> __device__ __forceinline__ void fft_butterfly(V& u, V& v, int m) {
  using T = decltype(u.x);
  const V a = u;
  if (m == 0) {
    u = fft_add(a, v);
    v = fft_sub(a, v);
  } else if (m == 8) {
    const V b = v;
    if (SIGN > 0) {
      u.x = a.x - b.y;
      u.y = a.y + b.x;
      v.x = a.x + b.y;
      v.y = a.y - b.x;
    } else {
      u.x = a.x + b.y;
      u.y = a.y - b.x;
      v.x = a.x - b.y;
      v.y = a.y + b.x;
    }
  } else {
    const double c = fft_cos32(m), s = SIGN * fft_sin32(m);
    const bool by_c = m <= 4 || m >= 12;   // |cos| >= |sin|
    const T r = (T)(by_c ? s / c : c / s), f = (T)(by_c ? c : s);
    V p;
    if (by_c) {
      p.x = fma(-r, v.y, v.x);
      p.y = fma(r, v.x, v.y);
    } else {
      p.x = fma(r, v.x, -v.y);
      p.y = fma(r, v.y, v.x);
    }
    u = fft_axpy(f, p, a);
    v = fft_axpy(-f, p, a);
  }
}

template <int N, int SIGN, typename V> __device__ __forceinline__ void fft_line(V (&x)[N]) {
  static_assert(N == 1 || N == 2 || N == 4 || N == 8 || N == 16 || N == 32, "line lengths 1 .. 32");
#pragma unroll
  for (int i = 0; i < N; ++i) {
    int j = 0;
#pragma unroll
    for (int b = 1, r = i; b < N; b <<= 1, r >>= 1) j = (j << 1) | (r & 1);
    if (j > i) {
      const V t = x[i];
      x[i] = x[j];
      x[j] = t;
    }
  }
#pragma unroll
  for (int len = 2; len <= N; len <<= 1)
#pragma unroll
    for (int i = 0; i < N; i += len)
#pragma unroll
      for (int k = 0; k < len / 2; ++k) fft_butterfly<SIGN>(x[i + k], x[i + k + len / 2], k * (32 / len));
}
