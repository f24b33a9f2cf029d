// Sums over a whole periodic grid line held in a thread's registers (the observation
// kernels of the 16^3 and 32^3 single-precision cells).
#pragma once
#include <cuda_runtime.h>

#include "tsbz_fft.cuh"
#include "tsbz_internal.h"
#include "tsbz_zmarch.cuh"

// Local current of the line, in correlation form:
//   sum_r Re(u* (-i grad) u) = 2 sum_m w_m Im sum_r u*(r) u(r + m),  m = 1 .. 4,
// which needs the forward neighbours only and does not depend on the point at which the
// line begins.  Runs of 16 points are summed in float, then the runs.
template <int N> __device__ __forceinline__ float line_current(const float2 (&u)[N], const float (&w)[TSBZ_MAX_ND + 1]) {
  constexpr int ND = ZM_ND, RUN = 16;
  float s = 0.f;
#pragma unroll
  for (int r0 = 0; r0 < N; r0 += RUN) {
    float2 cc[ND];
#pragma unroll
    for (int m = 0; m < ND; ++m) cc[m] = make_float2(0.f, 0.f);
#pragma unroll
    for (int r = r0; r < r0 + RUN; ++r) {
      const float2 t = make_float2(-u[r].y, u[r].x);   // Im(conj(u) v) = -u_i v_r + u_r v_i
#pragma unroll
      for (int m = 1; m <= ND; ++m) cc[m - 1] = __ffma2_rn(t, u[(r + m) & (N - 1)], cc[m - 1]);
    }
#pragma unroll
    for (int m = 1; m <= ND; ++m) s = __fmaf_rn(2.f * w[m], cc[m - 1].x + cc[m - 1].y, s);
  }
  return s;
}
