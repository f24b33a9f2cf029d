// Double precision on 16^3 grids: h applied to a band that stays in
// one CTA, for the whole time step (four Taylor stages, the projections of the
// current) or the whole Chebyshev filter of the ground-state solver in one launch.
//
// What bounds it: GB300's FP64 pipe (1.06 TFLOP/s measured, two operations a
// clock and SM), so everything here serves the number of FP64 operations per
// grid point; shared memory, launches and barriers cost nothing beside them.
//  - The kinetic operator -1/2 lap_FD - i q.grad_FD + |q|^2/2 is diagonal in
//    the discrete Fourier basis of the periodic grid, its symbol a sum of one
//    real number per axis (CellDev::ksym).  Six 16-point FFTs per line triple
//    and the scaling take 59 operations a point; the star stencil 108.
//  - The projectors factorise per axis.  Along z the phase e^{i q z} is common
//    to every atom, so one complex product per point leaves real sums per z
//    group (the minimum-image displacement jumps by one cell edge at one plane
//    per group: the running sums are turned by e^{i q L} there).  22 operations
//    a point for the sums (bra) and 20 for the ket with four groups; the box
//    and point forms took 111 and 84.
//  - The Taylor terms are kept as s_m = dt h^m psi; the rest of (-i dt)^m / m! enters only
//    the sum, psi's increment, which lives in shared memory (see tsbz_any.cu).
// One CTA per (unit, band), one thread per (x, y) column holding its N values
// along z in registers; the line transforms along x and y go through one
// shared buffer with the x index turned by y (no bank conflicts).  At 16^3 the
// two buffers take 128 KiB: one CTA per SM, whose 8 warps keep the FP64 pipe
// busy (a warp instruction occupies its quarter for 64 clocks).
// Measured, the whole time step: 512 k-points x 16 bands at 16^3, 79.8 -> 42.1 ms, FP64 pipe
// 82% busy at 132 operations per point and stage; 8 k-points x 16 bands 1.77 ->
// 0.83 ms.
#include <cuda_runtime.h>

#include "tsbz_fft.cuh"
#include "tsbz_internal.h"
#include "tsbz_launch.cuh"
#include "tsbz_symbol.cuh"

namespace {

constexpr int S64_NA = 8;        // atoms of a cell
constexpr int S64_GC = 4;        // z groups of one pass over a column

template <int N> struct S64Smem {
  static constexpr int NN = N * N, NP = N * N * N;
  double2 acc[NP];                          // Taylor sum, or the filter's previous block
  double2 buf[NP > 12 * NN ? NP : 12 * NN]; // line transforms; z sums of a projection pass
  double2 rs[S64_NA * 6 * N];               // x sums per (atom, k, w) and row
  double2 xf[S64_NA * N], yf[S64_NA * N];   // x and y factors g e^{i q d}
  double xd[S64_NA * N], yd[S64_NA * N];    // displacements
  double zw[3][S64_NA][N];                  // g, g d, g d^2 per z group
  double2 phi[N];                           // e^{i q z}
  double2 k0[S64_NA], kfin[S64_NA];         // phase of the group before / after its jump
  double2 turn[S64_NA];                     // k0 conj(k1)
  int zb[S64_NA];                           // plane of the jump (N: none)
  double2 gt[S64_NA * 3 * N];               // ket column tables
  double2 w[4 * S64_NA];                    // conj(k0) pn E P
  double2 mres[S64_NA * 10];                // monomial sums
  Symbol<double> lam[3][N];                 // kinetic symbol per axis, 1/N^3 folded in
  double lam3[N][NN];                       // and of line (k_x, k_z) at k_y
};

__device__ __forceinline__ double2 z_mul(double2 a, double2 b) {
  return make_double2(__fma_rn(a.x, b.x, -__dmul_rn(a.y, b.y)), __fma_rn(a.x, b.y, __dmul_rn(a.y, b.x)));
}
__device__ __forceinline__ double2 z_conj(double2 a) { return make_double2(a.x, -a.y); }

// monomial index of d_x^i d_y^j d_z^k (i + j + k <= 2): 000, 100, 010, 001, 200, 110, 101, 020, 011, 002
__device__ __forceinline__ int s64_mono(int i, int j, int k) {
  const int deg = i + j + k;
  if (deg == 0) return 0;
  if (deg == 1) return i ? 1 : (j ? 2 : 3);
  if (i == 2) return 4;
  if (i == 1) return j ? 5 : 6;
  if (j == 2) return 7;
  return j ? 8 : 9;
}

// Factor tables of one q (phase table ph of the unit); read after a barrier.
template <int N>
__device__ void s64_tables(S64Smem<N>& sm, const CellDev& c, const double2* ph, const double* q) {
  const int nm = c.nmax;
  for (int i = threadIdx.x; i < c.n_atoms * N; i += blockDim.x) {
    const int a = i / N, k = i - a * N, ix = a * 3 * nm + k, iy = ix + nm;
    const double gx = c.g1[ix], gy = c.g1[iy];
    const double2 px = ph[ix], py = ph[iy];
    sm.xf[i] = make_double2(gx * px.x, gx * px.y);
    sm.yf[i] = make_double2(gy * py.x, gy * py.y);
    sm.xd[i] = c.d1[ix];
    sm.yd[i] = c.d1[iy];
  }
  for (int i = threadIdx.x; i < c.n_zg * N; i += blockDim.x) {
    const int g = i / N, z = i - g * N, iz = (c.zg_rep[g] * 3 + 2) * nm + z;
    const double gz = c.g1[iz], dz = c.d1[iz];
    sm.zw[0][g][z] = gz;
    sm.zw[1][g][z] = gz * dz;
    sm.zw[2][g][z] = gz * dz * dz;
  }
  if (threadIdx.x < N) {
    double s, co;
    sincos(q[2] * (c.hz * (int)threadIdx.x), &s, &co);
    sm.phi[threadIdx.x] = make_double2(co, s);
  }
  if ((int)threadIdx.x < c.n_zg) {
    const int g = threadIdx.x;
    double s0, c0, s1, c1;
    sincos(q[2] * c.zg_k0[g], &s0, &c0);
    sincos(q[2] * (c.zg_k0[g] - c.hz * N), &s1, &c1);
    const double2 k0 = make_double2(c0, s0), k1 = make_double2(c1, s1);
    sm.zb[g] = c.zg_brk[g];
    sm.k0[g] = k0;
    sm.kfin[g] = c.zg_brk[g] < N ? k1 : k0;
    sm.turn[g] = z_mul(k0, z_conj(k1));
  }
}

// Kinetic symbol of the unit (barrier inside; lam3 is read by the thread that wrote it).
template <int N> __device__ void s64_symbol(S64Smem<N>& sm, const LaunchSet& L, int u) {
  if (threadIdx.x < 3 * N) sm.lam[threadIdx.x / N][threadIdx.x % N] = symbol_unit<double>(L, u)[threadIdx.x];
  __syncthreads();
  const Symbol<double> xz = symbol_add(sm.lam[0][threadIdx.x % N], sm.lam[2][threadIdx.x / N]);
#pragma unroll 4
  for (int y = 0; y < N; ++y) sm.lam3[y][threadIdx.x] = symbol_value(symbol_add(xz, sm.lam[1][y]));
}

// Monomial sums M_a(i, j, k) = sum_r F_x F_y F_z d_x^i d_y^j d_z^k t(r), i + j + k <= D,
// of every atom into mres[a NM + mono]; t is the thread's column.  Starts and
// ends with a barrier.  The D = 1 and D = 2 passes form the sums they share by
// the same rounded operations.
template <int N, int D>
__device__ void s64_project(S64Smem<N>& sm, const CellDev& c, const double2 (&t)[N]) {
  constexpr int NN = N * N, NM = D == 1 ? 4 : 10;
  const int tid = threadIdx.x, ix = tid % N, iy = tid / N;
  for (int g0 = 0; g0 < c.n_zg; g0 += S64_GC) {
    __syncthreads();
    double2 s[S64_GC][D + 1];
#pragma unroll
    for (int g = 0; g < S64_GC; ++g)
#pragma unroll
      for (int k = 0; k <= D; ++k) s[g][k] = make_double2(0.0, 0.0);
#pragma unroll
    for (int z = 0; z < N; ++z) {
      const double2 u = z_mul(sm.phi[z], t[z]);
#pragma unroll
      for (int g = 0; g < S64_GC; ++g) {
        if (g0 + g >= c.n_zg) break;
        if (z == sm.zb[g0 + g]) {
#pragma unroll
          for (int k = 0; k <= D; ++k) s[g][k] = z_mul(sm.turn[g0 + g], s[g][k]);
        }
#pragma unroll
        for (int k = 0; k <= D; ++k) {
          const double w = sm.zw[k][g0 + g][z];
          s[g][k].x = __fma_rn(w, u.x, s[g][k].x);
          s[g][k].y = __fma_rn(w, u.y, s[g][k].y);
        }
      }
    }
#pragma unroll
    for (int g = 0; g < S64_GC; ++g)
#pragma unroll
      for (int k = 0; k <= D; ++k) sm.buf[(g * (D + 1) + k) * NN + iy * N + (ix ^ iy)] = s[g][k];
    __syncthreads();
    // x sums of row (atom, k, iy): R_w = sum_x F_x d_x^w S_k, w <= D - k
    const int m0 = c.zg_off[g0], nmem = c.zg_off[min(g0 + S64_GC, c.n_zg)] - m0;
    for (int id = tid; id < nmem * (D + 1) * N; id += NN) {
      const int y = id % N, r = id / N, k = r / nmem, i = r - k * nmem;
      const int a = c.zg_mem[m0 + i], g = c.zg_of[a] - g0;
      const double2* row = sm.buf + (g * (D + 1) + k) * NN + y * N;
      double2 R[3];
#pragma unroll
      for (int w = 0; w < 3; ++w) R[w] = make_double2(0.0, 0.0);
#pragma unroll 4
      for (int j = 0; j < N; ++j) {
        double2 p = z_mul(sm.xf[a * N + j], row[j ^ y]);
        R[0].x = __dadd_rn(R[0].x, p.x);
        R[0].y = __dadd_rn(R[0].y, p.y);
        if (k < D) {
          const double d = sm.xd[a * N + j];
          R[1].x = __fma_rn(d, p.x, R[1].x);
          R[1].y = __fma_rn(d, p.y, R[1].y);
          if (D == 2 && k == 0) {
            R[2].x = __fma_rn(d * d, p.x, R[2].x);
            R[2].y = __fma_rn(d * d, p.y, R[2].y);
          }
        }
      }
      double2* o = sm.rs + (a * 6 + (k == 0 ? 0 : (k == 1 ? 3 : 5))) * N + y;
      o[0] = R[0];
      if (k < D) o[N] = R[1];
      if (D == 2 && k == 0) o[2 * N] = R[2];
    }
    __syncthreads();
    // y sums, and the group's phase
    for (int id = tid; id < nmem * NM; id += NN) {
      const int i = id / NM, mo = id - i * NM, a = c.zg_mem[m0 + i];
      int ex = 0, ey = 0, ez = 0;
      if (mo == 1 || mo == 5 || mo == 6) ex = 1;
      if (mo == 4) ex = 2;
      if (mo == 2 || mo == 5 || mo == 8) ey = 1;
      if (mo == 7) ey = 2;
      if (mo == 3 || mo == 6 || mo == 8) ez = 1;
      if (mo == 9) ez = 2;
      const double2* R = sm.rs + (a * 6 + (ez == 0 ? ex : (ez == 1 ? 3 + ex : 5))) * N;
      double2 M = make_double2(0.0, 0.0);
      for (int y = 0; y < N; ++y) {
        const double2 p = z_mul(sm.yf[a * N + y], R[y]);
        const double d = sm.yd[a * N + y], wy = ey == 0 ? 1.0 : (ey == 1 ? d : d * d);
        M.x = __fma_rn(wy, p.x, M.x);
        M.y = __fma_rn(wy, p.y, M.y);
      }
      sm.mres[a * NM + mo] = z_mul(sm.kfin[c.zg_of[a]], M);
    }
  }
  __syncthreads();
}

// Ket weights of the band from its projections P (nullptr: from mres of a
// first-order pass); ends with a barrier.
template <int N> __device__ void s64_weights(S64Smem<N>& sm, const CellDev& c, const double2* P) {
  for (int j = threadIdx.x; j < c.n_proj; j += blockDim.x) {
    const double sc = c.dv * c.pnorm[j], e = c.wkb[j];
    const double2 p = P ? P[j] : make_double2(sc * sm.mres[j].x, sc * sm.mres[j].y);
    sm.w[j] = z_mul(z_conj(sm.k0[c.zg_of[j >> 2]]), make_double2(e * p.x, e * p.y));
  }
  __syncthreads();
}

// f = h t for the thread's column t; the ket weights are in sm.w.
template <int N>
__device__ void s64_apply(S64Smem<N>& sm, const CellDev& c, const double* __restrict__ veff, const double2 (&t)[N],
                          double2 (&f)[N]) {
  constexpr int NN = N * N;
  const int tid = threadIdx.x, lo = tid % N, hi = tid / N;   // as a column: ix, iy
  double2* buf = sm.buf;
  const int cb = hi * N + (lo ^ hi);
#pragma unroll
  for (int z = 0; z < N; ++z) f[z] = t[z];
  fft_line<N, -1>(f);
#pragma unroll
  for (int z = 0; z < N; ++z) buf[z * NN + cb] = f[z];
  if (c.use_proj) {
    // ket column tables: G00 = conj(F_x) (W_s + d_x W_px), G10 = conj(F_x) W_py, G01 = conj(F_x) W_pz
    for (int i = tid; i < c.n_atoms * N; i += NN) {
      const int a = i / N, x = i - a * N;
      const double2 F = z_conj(sm.xf[i]);
      const double d = sm.xd[i];
      const double2 ws = sm.w[4 * a], wx = sm.w[4 * a + 1];
      sm.gt[(a * 3 + 0) * N + x] = z_mul(F, make_double2(fma(d, wx.x, ws.x), fma(d, wx.y, ws.y)));
      sm.gt[(a * 3 + 1) * N + x] = z_mul(F, sm.w[4 * a + 2]);
      sm.gt[(a * 3 + 2) * N + x] = z_mul(F, sm.w[4 * a + 3]);
    }
  }
  __syncthreads();
  {
    double2* row = buf + hi * NN + lo * N;   // row y = lo of plane hi
#pragma unroll
    for (int x = 0; x < N; ++x) f[x] = row[x ^ lo];
    fft_line<N, -1>(f);
#pragma unroll
    for (int x = 0; x < N; ++x) row[x ^ lo] = f[x];
  }
  __syncthreads();
  {
    double2* pl = buf + hi * NN;   // column x = lo of plane hi
#pragma unroll
    for (int y = 0; y < N; ++y) f[y] = pl[y * N + (lo ^ y)];
    fft_line<N, -1>(f);
#pragma unroll
    for (int y = 0; y < N; ++y) {
      const double l = sm.lam3[y][tid];
      f[y].x *= l;
      f[y].y *= l;
    }
    fft_line<N, 1>(f);
#pragma unroll
    for (int y = 0; y < N; ++y) pl[y * N + (lo ^ y)] = f[y];
  }
  __syncthreads();
  {
    double2* row = buf + hi * NN + lo * N;
#pragma unroll
    for (int x = 0; x < N; ++x) f[x] = row[x ^ lo];
    fft_line<N, 1>(f);
#pragma unroll
    for (int x = 0; x < N; ++x) row[x ^ lo] = f[x];
  }
  __syncthreads();
#pragma unroll
  for (int z = 0; z < N; ++z) f[z] = buf[z * NN + cb];
  fft_line<N, 1>(f);
#pragma unroll
  for (int z = 0; z < N; ++z) {
    const double v = veff[z * NN + tid];
    f[z].x = fma(v, t[z].x, f[z].x);
    f[z].y = fma(v, t[z].y, f[z].y);
  }
  if (!c.use_proj) return;
  for (int g0 = 0; g0 < c.n_zg; g0 += S64_GC) {
    // column coefficients of the pass's groups
    double2 c0[S64_GC], c1[S64_GC];
#pragma unroll
    for (int g = 0; g < S64_GC; ++g) {
      c0[g] = c1[g] = make_double2(0.0, 0.0);
      if (g0 + g >= c.n_zg) continue;
      for (int i = c.zg_off[g0 + g]; i < c.zg_off[g0 + g + 1]; ++i) {
        const int a = c.zg_mem[i];
        const double2 F = z_conj(sm.yf[a * N + hi]);
        const double d = sm.yd[a * N + hi];
        const double2 g00 = sm.gt[(a * 3 + 0) * N + lo], g10 = sm.gt[(a * 3 + 1) * N + lo];
        const double2 g01 = sm.gt[(a * 3 + 2) * N + lo];
        const double2 e = make_double2(fma(d, g10.x, g00.x), fma(d, g10.y, g00.y));
        c0[g].x = fma(F.x, e.x, fma(-F.y, e.y, c0[g].x));
        c0[g].y = fma(F.x, e.y, fma(F.y, e.x, c0[g].y));
        c1[g].x = fma(F.x, g01.x, fma(-F.y, g01.y, c1[g].x));
        c1[g].y = fma(F.x, g01.y, fma(F.y, g01.x, c1[g].y));
      }
    }
#pragma unroll
    for (int z = 0; z < N; ++z) {
      double2 x = make_double2(0.0, 0.0);
#pragma unroll
      for (int g = 0; g < S64_GC; ++g) {
        if (g0 + g >= c.n_zg) break;
        if (z == sm.zb[g0 + g]) {
          c0[g] = z_mul(sm.turn[g0 + g], c0[g]);
          c1[g] = z_mul(sm.turn[g0 + g], c1[g]);
        }
        const double w0 = sm.zw[0][g0 + g][z], w1 = sm.zw[1][g0 + g][z];
        x.x = fma(w0, c0[g].x, fma(w1, c1[g].x, x.x));
        x.y = fma(w0, c0[g].y, fma(w1, c1[g].y, x.y));
      }
      const double2 p = sm.phi[z];   // conj(phi) x
      f[z].x = fma(p.x, x.x, fma(p.y, x.y, f[z].x));
      f[z].y = fma(p.x, x.y, fma(-p.y, x.x, f[z].y));
    }
  }
}

// P of the current and of the next step from the second-order sums of t:
// rows (a, c_x, c_y, c_z) of projector j to Pa, and a to Pnext if given.
template <int N>
__device__ void s64_current(S64Smem<N>& sm, const CellDev& c, const double2 (&t)[N], double2* __restrict__ Pab,
                            double2* __restrict__ Pnext) {
  s64_project<N, 2>(sm, c, t);
  for (int o = threadIdx.x; o < 4 * c.n_proj; o += N * N) {
    const int j = o >> 2, s = o & 3, a = j >> 2, ty = j & 3;
    int e[3] = {ty == 1, ty == 2, ty == 3};
    if (s > 0) e[s - 1] += 1;
    const double sc = c.dv * c.pnorm[j];
    const double2 M = sm.mres[a * 10 + s64_mono(e[0], e[1], e[2])];
    const double2 v = make_double2(sc * M.x, sc * M.y);
    Pab[4 * j + s] = v;
    if (Pnext && s == 0) Pnext[j] = v;
  }
}

// One time step of every band, psi in and out of global memory once.
//   fresh_p: the projections of psi are formed here (else read from P);
//   want_pa: the projections of the current at q_obs, and with same_next (a
//     constant field: the next step's q is q_obs) those of the next step, too.
template <int N>
__global__ void __launch_bounds__(N* N, 1) k_step64(LaunchSet L, double2* __restrict__ psi, double2* __restrict__ P,
                                                    double2* __restrict__ Pa, int fresh_p, int want_pa,
                                                    int same_next) {
  step_enter();
  extern __shared__ __align__(16) unsigned char s64_raw[];
  S64Smem<N>& sm = *reinterpret_cast<S64Smem<N>*>(s64_raw);
  constexpr int NN = N * N;
  const CellDev& c = L.cell;
  const int b = blockIdx.x % c.n_bands;
  const int u = L.unit_ids[blockIdx.x / c.n_bands];
  if (!unit_active(L, u)) return;
  const UnitDev U = L.units[u];
  const SubDev S = L.subs[U.sub];
  const int tid = threadIdx.x;
  const double* veff = reinterpret_cast<const double*>(S.veff);
  double2* band = psi + U.psi_off + (long long)b * (N * NN) + tid;
  double2* Pu = P + U.p_off + (long long)b * c.n_proj;
  double2 t[N], f[N];
#pragma unroll
  for (int z = 0; z < N; ++z) t[z] = band[z * NN];
  s64_symbol<N>(sm, L, u);
  if (c.use_proj) s64_tables<N>(sm, c, (const double2*)L.ph_half + (long long)u * L.ph_stride, L.q_half + 3 * u);
  __syncthreads();
  if (c.use_proj) {
    if (fresh_p) s64_project<N, 1>(sm, c, t);
    s64_weights<N>(sm, c, fresh_p ? nullptr : Pu);
  }
  const double dt = S.dt * L.dt_scale;
  double coef = 1.0;
#pragma unroll 1
  for (int m = 1; m <= 4; ++m) {
    s64_apply<N>(sm, c, veff, t, f);
    // the increment of psi: (-i)^m coef s_m summed over m
    if (m == 1) {
#pragma unroll
      for (int z = 0; z < N; ++z) {
        t[z] = make_double2(dt * f[z].x, dt * f[z].y);
        sm.acc[z * NN + tid] = make_double2(t[z].y, -t[z].x);
      }
    } else {
      coef *= dt / (double)m;
      const double sx = m == 2 ? -coef : coef;
#pragma unroll
      for (int z = 0; z < N; ++z) {
        double2 a = sm.acc[z * NN + tid];
        if (m == 3) {
          a.x = fma(-coef, f[z].y, a.x);
          a.y = fma(coef, f[z].x, a.y);
        } else {
          a.x = fma(sx, f[z].x, a.x);
          a.y = fma(sx, f[z].y, a.y);
        }
        if (m < 4) {
          sm.acc[z * NN + tid] = a;
          t[z] = f[z];
        } else {
          const double2 u0 = band[z * NN];
          t[z] = make_double2(u0.x + a.x, u0.y + a.y);
          band[z * NN] = t[z];
        }
      }
    }
    if (m < 4 && c.use_proj) {
      s64_project<N, 1>(sm, c, t);
      s64_weights<N>(sm, c, nullptr);
    }
  }
  if (!c.use_proj || !want_pa) return;
  __syncthreads();
  if (!same_next) {
    s64_tables<N>(sm, c, (const double2*)L.ph_obs + (long long)u * L.ph_stride, L.q_obs + 3 * u);
  }
  s64_current<N>(sm, c, t, Pa + U.pa_off + 4LL * b * c.n_proj, same_next ? Pu : nullptr);
}

// Projections of the current outside a step (J(0-), J(0+), restored states).
template <int N>
__global__ void __launch_bounds__(N* N, 1) k_pa64(LaunchSet L, const double2* __restrict__ src,
                                                  double2* __restrict__ Pa) {
  extern __shared__ __align__(16) unsigned char s64_raw[];
  S64Smem<N>& sm = *reinterpret_cast<S64Smem<N>*>(s64_raw);
  constexpr int NN = N * N;
  const CellDev& c = L.cell;
  const int b = blockIdx.x % c.n_bands;
  const int u = L.unit_ids[blockIdx.x / c.n_bands];
  if (!unit_active(L, u)) return;
  const UnitDev U = L.units[u];
  const double2* band = src + U.psi_off + (long long)b * (N * NN) + threadIdx.x;
  double2 t[N];
#pragma unroll
  for (int z = 0; z < N; ++z) t[z] = band[z * NN];
  s64_tables<N>(sm, c, (const double2*)L.ph_obs + (long long)u * L.ph_stride, L.q_obs + 3 * u);
  s64_current<N>(sm, c, t, Pa + U.pa_off + 4LL * b * c.n_proj, nullptr);
}

// The ground-state solver's filter: Y_1 = fa0 h Y_0 + fa1 Y_0, then
// Y_{j+1} = fb0 h Y_j + fb1 Y_j + fb2 Y_{j-1} up to Y_degree (coefficients per
// unit); degree 1 applies h alone.  Bands are independent and h is fixed, so
// the whole recurrence of a band runs in its CTA (in and out may be the same block).
template <int N>
__global__ void __launch_bounds__(N* N, 1) k_filter64(LaunchSet L, const double2* in, double2* out, const double* __restrict__ fa,
                                                      const double* __restrict__ fb, int degree) {
  extern __shared__ __align__(16) unsigned char s64_raw[];
  S64Smem<N>& sm = *reinterpret_cast<S64Smem<N>*>(s64_raw);
  constexpr int NN = N * N;
  const CellDev& c = L.cell;
  const int b = blockIdx.x % c.n_bands;
  const int u = L.unit_ids[blockIdx.x / c.n_bands];
  if (!unit_active(L, u)) return;
  const UnitDev U = L.units[u];
  const SubDev S = L.subs[U.sub];
  const int tid = threadIdx.x;
  const double* veff = reinterpret_cast<const double*>(S.veff);
  const long long off = U.psi_off + (long long)b * (N * NN) + tid;
  double2 t[N], f[N];
#pragma unroll
  for (int z = 0; z < N; ++z) t[z] = in[off + z * NN];
  s64_symbol<N>(sm, L, u);
  if (c.use_proj) s64_tables<N>(sm, c, (const double2*)L.ph_half + (long long)u * L.ph_stride, L.q_half + 3 * u);
  __syncthreads();
#pragma unroll 1
  for (int j = 0; j < degree; ++j) {
    if (c.use_proj) {
      s64_project<N, 1>(sm, c, t);
      s64_weights<N>(sm, c, nullptr);
    }
    s64_apply<N>(sm, c, veff, t, f);
    const double* fc = j == 0 ? fa : fb;
    const double f0 = fc[3 * u], f1 = fc[3 * u + 1], f2 = j == 0 ? 0.0 : fc[3 * u + 2];
#pragma unroll
    for (int z = 0; z < N; ++z) {
      double2 y = make_double2(fma(f0, f[z].x, f1 * t[z].x), fma(f0, f[z].y, f1 * t[z].y));
      if (j > 0) {
        const double2 p = sm.acc[z * NN + tid];
        y.x = fma(f2, p.x, y.x);
        y.y = fma(f2, p.y, y.y);
      }
      sm.acc[z * NN + tid] = t[z];
      t[z] = y;
    }
    if (!c.use_proj) __syncthreads();   // the line buffer is written again
  }
#pragma unroll
  for (int z = 0; z < N; ++z) out[off + z * NN] = t[z];
}

template <typename K> void s64_attr(K* k, size_t bytes) {
  cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

}  // namespace

static bool step64_supported(const CellDev& c) {
  return c.n1 == 16 && c.n2 == 16 && c.n3 == 16 && c.n_atoms <= S64_NA;
}

// Variant 0 of such cells, where it is the quicker form.  One CTA holds a band, so up to 152
// orbitals cost what one does, while the point-parallel sequence spreads few bands of
// many k-points over every SM: its projections cost by the bands of a unit (a CTA takes
// up to 8), its stages by the rounds of 32 point tiles per unit and the bands.  Both sides
// as fitted to times of a whole step (us; 1 .. 64 k-points times 1 .. 16 bands, no, 1, 2, 4 and 8
// atoms in 1 .. 8 z groups, within 8%; sequence against one launch):
// 8 atoms on 4 planes: 8 x 1 433 / 772, 8 x 4 714 / 782, 8 x 6 947 / 787, 16 x 1 676 / 778,
// 16 x 2 810 / 783, 24 x 1 989 / 782, 1 x 6 762 / 772, 1 x 8 913 / 775; 8 atoms on 8 planes: 8 x 6
// 973 / 1003, 1 x 16 1211 / 994; without projectors: 1 x 8 219 / 489, 8 x 16 640 / 527, 64 x 1 343 / 511.
// The filter of the ground-state solver is chosen alike (an application of h, 2 atoms, 1 x 4
// 84 / 154, 24 x 2 130 / 154, 1 x 16 194 / 154).
static bool step64_quicker(const CellDev& c, int n_units) {
  const long long b = c.n_bands, n = (32LL * n_units + 151) / 152, waves = (n_units * b + 151) / 152;
  if (!c.use_proj) return 60 + 2 * n + 18 * n * b >= 50 + 440 * waves;
  const long long whole =
      440 + 138 + 38 * (c.n_zg - 1) + 8 * (c.n_atoms - c.n_zg) + (c.n_zg > S64_GC ? 65 : 0);
  return 146 + n * (2 + 12 * c.n_atoms) + 64 * (b < 8 ? b : 8) + 35 * n * b / 2 >= 50 + whole * waves;
}
static bool step64_taken(const LaunchSet& L) {
  return L.variant == 0 && step64_supported(L.cell) && step64_quicker(L.cell, L.n_units);
}

bool launch_step64(const LaunchSet& L, void* psi, void* P, void* Pa, int fresh_p, int want_pa, int same_next,
                   void* stream) {
  if (L.n_units == 0 || !step64_taken(L)) return false;
  s64_attr(k_step64<16>, sizeof(S64Smem<16>));
  step_launch(k_step64<16>, (unsigned)L.n_units * L.cell.n_bands, 256, sizeof(S64Smem<16>), stream, L, (double2*)psi,
              (double2*)P, (double2*)Pa, fresh_p, want_pa, same_next);
  return true;
}

bool launch_pa64(const LaunchSet& L, const void* src, void* Pa, void* stream) {
  if (L.n_units == 0 || !step64_taken(L) || !L.cell.use_proj) return false;
  s64_attr(k_pa64<16>, sizeof(S64Smem<16>));
  k_pa64<16><<<(unsigned)L.n_units * L.cell.n_bands, 256, sizeof(S64Smem<16>), (cudaStream_t)stream>>>(
      L, (const double2*)src, (double2*)Pa);
  return true;
}

bool launch_filter64(const LaunchSet& L, const void* in, void* out, const double* fa, const double* fb, int degree,
                     void* stream) {
  if (L.n_units == 0 || !step64_supported(L.cell) || !step64_quicker(L.cell, L.n_units)) return false;
  s64_attr(k_filter64<16>, sizeof(S64Smem<16>));
  k_filter64<16><<<(unsigned)L.n_units * L.cell.n_bands, 256, sizeof(S64Smem<16>), (cudaStream_t)stream>>>(
      L, (const double2*)in, (double2*)out, fa, fb, degree);
  return true;
}
