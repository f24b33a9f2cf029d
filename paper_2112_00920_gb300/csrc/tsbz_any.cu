// Small grids of any shape: the whole time step of a band (or the whole
// Chebyshev recurrence of the ground-state solver) in one CTA and one launch, in
// double or single precision; with few orbitals in double in a cluster of CTAs.
//
// What bounds such runs is latency: a step of nine to twelve launches, each a
// few CTAs that wait on dependent loads, and in double precision the FP64
// instructions a warp issues (64 clocks each on its quarter of the SM).  So
// the band of t_{m-1}, t_m and the Taylor sum stay in shared memory, every
// contraction is spread over all eight warps as independent items, and the next
// launch is the observation.
//  - Kinetic operator: the star stencil from shared memory, or on 8^3 grids its
//    Fourier symbol (Form8): four threads per line, each forming the outputs k and
//    k + 4 of an 8-point transform (20 operations), 6 passes.
//  - Projectors: the phase e^{i q z} is taken off once per point, so the z sums are
//    real per (z group, column); then x sums per (atom, power, row), y sums per
//    (atom, monomial).  The ket goes back the same way.  A group's minimum image
//    jumps by one cell edge at one plane; the running sums are turned there.
//  - Taylor terms are s_m = dt h^m psi; the rest of (-i dt)^m / m! enters the sum only.  The
//    first dt sits in s_1 because dt^2 / 2 is no number of the type: as a coefficient of h^2 psi its
//    rounding is the same every step and the norms drift, while dt / 2 of s_2 is exact.  The
//    sum holds psi's increment, and psi is added last: rounded once a step, not four times
//    (500 steps at 8^3 in single precision: mean of the norms off by 2.5e-7 -> 3e-8).
// Everything the first- and second-order projection passes share is formed by the
// same rounded operations, so a step may start from the projections that the
// last one left (same q) or from fresh ones, bit for bit.
// Measured per step, all four stages with their projections: 8^3, 16 orbitals in
// double 298 -> 64 us (96 with a CTA per band), 512 orbitals in single 65 -> 41 us; 10 x 12 x 14, 324 orbitals
// in single under a pulse 179 -> 73 us (before: two launches per stage and one for
// the current).
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "tsbz_internal.h"
#include "tsbz_launch.cuh"
#include "tsbz_symbol.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int ANY_NA = 8;          // atoms
constexpr int ANY_MIN_ORB = 8;     // orbitals from which the whole-step form is taken
constexpr size_t ANY_MAX_SMEM = 200 * 1024, ANY_WIDE_SMEM = 56 * 1024;

// The form of a kernel: 8^3 grids with every size at compile time, or any grid with so many threads.
// ctas > 1: a cluster of so many CTAs shares a band (see k_step_any).
struct Form8 {
  static constexpr bool eight = true;
  static constexpr int threads = 256, ctas = 1, proj0 = 0;
};
template <int N> struct FormAny {
  static constexpr bool eight = false;
  static constexpr int threads = N, ctas = 1, proj0 = 0;
};
struct Form8Cluster {
  static constexpr bool eight = true;
  static constexpr int threads = 128, ctas = 4, proj0 = 64;   // threads 0 .. 63 transform meanwhile
};
template <int C> struct FormCluster {
  static constexpr bool eight = false;
  static constexpr int threads = 256, ctas = C, proj0 = 0;
};

// Rows of the CTA's share: all of them, or those of its rank in the cluster.
template <class F> __device__ __forceinline__ int any_row0(int rank, int n2) { return rank * n2 / F::ctas; }
// Barrier of the threads that project, proj0 and up.
template <class F> __device__ __forceinline__ void any_sync() {
  if constexpr (F::proj0 == 0)
    __syncthreads();
  else
    asm volatile("bar.sync 1, %0;\n" ::"n"(F::threads - F::proj0) : "memory");
}
__device__ __forceinline__ int any_rank() { return (int)cg::this_cluster().block_rank(); }

__host__ __device__ __forceinline__ bool any_fft8(const CellDev& c) { return c.n1 == 8 && c.n2 == 8 && c.n3 == 8; }

template <typename T> struct AnyC;
template <> struct AnyC<double> { using V = double2; };
template <> struct AnyC<float> { using V = float2; };

__device__ __forceinline__ double rmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float rmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double radd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float radd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double rfm(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float rfm(float a, float b, float c) { return __fmaf_rn(a, b, c); }

template <typename V> __device__ __forceinline__ V vmk(decltype(V().x) a, decltype(V().x) b) {
  V r;
  r.x = a;
  r.y = b;
  return r;
}
template <typename V> __device__ __forceinline__ V vmul(V a, V b) {   // complex product, fixed rounding
  return vmk<V>(rfm(a.x, b.x, -rmul(a.y, b.y)), rfm(a.x, b.y, rmul(a.y, b.x)));
}
template <typename V> __device__ __forceinline__ V vconj(V a) { return vmk<V>(a.x, -a.y); }
template <typename V, typename T> __device__ __forceinline__ V vaxpy(T s, V b, V a) {   // a + s b
  return vmk<V>(rfm(s, b.x, a.x), rfm(s, b.y, a.y));
}
// sign flip without arithmetic
__device__ __forceinline__ double flip(double a, unsigned m) {
  return __hiloint2double(__double2hiint(a) ^ (int)(m << 31), __double2loint(a));
}
__device__ __forceinline__ float flip(float a, unsigned m) { return __uint_as_float(__float_as_uint(a) ^ (m << 31)); }

// Shared memory of a CTA: pointers into one block, laid out alike on both sides.
template <typename T> struct AnySmem {
  using V = typename AnyC<T>::V;
  V *a, *b, *acc;        // t_{m-1} / t_m (roles alternate), Taylor sum
  V* s;                  // z sums, ket coefficients per (group, column); line transforms (8^3)
  V *xk, *xl, *part;     // clusters: all k_z planes of an 8^3 band, the CTA's two, the ranks' monomial sums
  V *rs, *gt, *xf, *yf, *phi, *w, *mres, *k0, *kfin, *turn;
  T *xd, *yd, *zw, *lam3, *st;
  Symbol<T>* lam;
  int *idx, *zb;
};

constexpr int ANY_X8 = 8 * 72;   // one 8^3 line buffer with rows of 9

template <typename T>
__host__ __device__ inline size_t any_carve(const CellDev& c, unsigned char* base, AnySmem<T>& m, int ctas = 1) {
  using V = typename AnyC<T>::V;
  size_t at = 0;
  auto take = [&](size_t bytes) {
    unsigned char* p = base + at;
    at += (bytes + 15) / 16 * 16;
    return p;
  };
  const int na = c.use_proj ? c.n_atoms : 0, ng = c.use_proj ? c.n_zg : 0, n12 = c.n1 * c.n2;
  size_t ns = (size_t)3 * ng * n12;
  if (any_fft8(c) && ns < 2 * ANY_X8) ns = 2 * ANY_X8;
  m.a = (V*)take(sizeof(V) * c.npts);
  m.b = (V*)take(sizeof(V) * c.npts);
  m.acc = (V*)take(sizeof(V) * c.npts);
  m.s = (V*)take(sizeof(V) * ns);
  m.rs = (V*)take(sizeof(V) * na * 6 * c.n2);
  m.gt = (V*)take(sizeof(V) * na * 3 * c.n1);
  m.xf = (V*)take(sizeof(V) * na * c.n1);
  m.yf = (V*)take(sizeof(V) * na * c.n2);
  m.phi = (V*)take(sizeof(V) * c.n3);
  m.w = (V*)take(sizeof(V) * 4 * ANY_NA);
  m.mres = (V*)take(sizeof(V) * 10 * ANY_NA);
  m.k0 = (V*)take(sizeof(V) * ANY_NA);
  m.kfin = (V*)take(sizeof(V) * ANY_NA);
  m.turn = (V*)take(sizeof(V) * ANY_NA);
  m.xd = (T*)take(sizeof(T) * na * c.n1);
  m.yd = (T*)take(sizeof(T) * na * c.n2);
  m.zw = (T*)take(sizeof(T) * 3 * ng * c.n3);
  if (any_fft8(c)) {
    m.lam = (Symbol<T>*)take(sizeof(Symbol<T>) * 3 * 8);
    m.lam3 = (T*)take(sizeof(T) * 512);   // the symbol at (k_z, k_y, k_x)
  }
  m.st = (T*)take(sizeof(T) * (6 * (TSBZ_MAX_ND + 1) + 1));
  m.idx = (int*)take(sizeof(int) * c.npts);
  m.zb = (int*)take(sizeof(int) * ANY_NA);
  if (ctas > 1) {
    m.part = (V*)take(sizeof(V) * 10 * ANY_NA * ctas);
    if (any_fft8(c)) {
      m.xk = (V*)take(sizeof(V) * ANY_X8);
      m.xl = (V*)take(sizeof(V) * ANY_X8 / 2);
    }
  }
  return at;
}

template <typename T> struct AnyTab;
template <> struct AnyTab<double> {
  static __device__ const double* g1(const CellDev& c) { return c.g1; }
  static __device__ const double* d1(const CellDev& c) { return c.d1; }
  static __device__ const double* pnorm(const CellDev& c) { return c.pnorm; }
  static __device__ const double* wkb(const CellDev& c) { return c.wkb; }
  static __device__ double dv(const CellDev& c) { return c.dv; }
};
template <> struct AnyTab<float> {
  static __device__ const float* g1(const CellDev& c) { return c.g1f; }
  static __device__ const float* d1(const CellDev& c) { return c.d1f; }
  static __device__ const float* pnorm(const CellDev& c) { return c.pnormf; }
  static __device__ const float* wkb(const CellDev& c) { return c.wkbf; }
  static __device__ float dv(const CellDev& c) { return c.dvf; }
};

__device__ __forceinline__ int any_mono(int i, int j, int k) {   // 000 100 010 001 200 110 101 020 011 002
  const int deg = i + j + k;
  if (deg == 0) return 0;
  if (deg == 1) return i ? 1 : (j ? 2 : 3);
  if (i == 2) return 4;
  if (i == 1) return j ? 5 : 6;
  if (j == 2) return 7;
  return j ? 8 : 9;
}

// Point i of the thread: in 8^3 cells the outputs z = p, p + 4 of column l (l = t / 4, p = t % 4).
template <class F> __device__ __forceinline__ int any_point(int i) {
  return F::eight ? ((int)threadIdx.x & 3) * 64 + ((int)threadIdx.x >> 2) + 256 * i : (int)threadIdx.x + F::threads * i;
}

// Projector factor tables of one q (phase table ph of the unit); read after a barrier.
template <typename T, class F>
__device__ void any_tables(const AnySmem<T>& sm, const CellDev& c, const typename AnyC<T>::V* ph) {
  using V = typename AnyC<T>::V;
  const int n1 = F::eight ? 8 : c.n1, n2 = F::eight ? 8 : c.n2, n3 = F::eight ? 8 : c.n3;
  const int nm = F::eight ? 8 : c.nmax;
  const T *g1 = AnyTab<T>::g1(c), *d1 = AnyTab<T>::d1(c);
  for (int i = threadIdx.x; i < c.n_atoms * n1; i += F::threads) {
    const int a = i / n1, k = a * 3 * nm + i - a * n1;
    sm.xf[i] = vmk<V>(g1[k] * ph[k].x, g1[k] * ph[k].y);
    sm.xd[i] = d1[k];
  }
  for (int i = threadIdx.x; i < c.n_atoms * n2; i += F::threads) {
    const int a = i / n2, k = (a * 3 + 1) * nm + i - a * n2;
    sm.yf[i] = vmk<V>(g1[k] * ph[k].x, g1[k] * ph[k].y);
    sm.yd[i] = d1[k];
  }
  for (int i = threadIdx.x; i < c.n_zg * n3; i += F::threads) {
    const int g = i / n3, k = (c.zg_rep[g] * 3 + 2) * nm + i - g * n3;
    sm.zw[i] = g1[k];
    sm.zw[c.n_zg * n3 + i] = g1[k] * d1[k];
    sm.zw[2 * c.n_zg * n3 + i] = g1[k] * d1[k] * d1[k];
  }
  // phases along z (formed with the other tables, CellDev::ph_z): of the planes, of
  // each group before its jump and at its end, and of the jump
  const V* pz = ph + c.ph_z;
  for (int i = threadIdx.x; i < n3 + c.n_zg; i += F::threads) {
    if (i < n3) {
      sm.phi[i] = pz[i];
    } else {
      const int g = i - n3;
      sm.k0[g] = pz[n3 + 2 * g];
      sm.kfin[g] = pz[n3 + 2 * g + 1];
      sm.turn[g] = pz[n3 + 2 * c.n_zg];   // phase before over phase after
      sm.zb[g] = c.zg_brk[g];
    }
  }
}

// Stencil weights (or the symbol of 8^3 grids) of the step's q, and the points' coordinates.
template <typename T, class F>
__device__ void any_setup(const AnySmem<T>& sm, const CellDev& c, const LaunchSet& L, int u, const double* q) {
  const int tid = threadIdx.x;
  if (F::eight) {
    if (tid < 24) sm.lam[tid] = symbol_unit<T>(L, u)[tid];
    __syncthreads();
    const Symbol<T> xy = symbol_add(sm.lam[tid & 7], sm.lam[8 + ((tid >> 3) & 7)]);
    for (int p = tid; p < 512; p += F::threads) sm.lam3[p] = symbol_value(symbol_add(xy, sm.lam[16 + (p >> 6)]));
  } else {
    constexpr int M = TSBZ_MAX_ND + 1;
    if (tid < 3 * M) {
      const int ax = tid / M, m = tid - ax * M;
      sm.st[tid] = (T)(-0.5 * c.lapw[ax][m]);
      sm.st[3 * M + tid] = (T)(q[ax] * c.gradw[ax][m]);
    }
    if (tid == 3 * M) {
      double d = 0.5 * (q[0] * q[0] + q[1] * q[1] + q[2] * q[2]);
      for (int ax = 0; ax < 3; ++ax) d -= 0.5 * c.lapw[ax][0];
      sm.st[6 * M] = (T)d;
    }
    for (int p = tid; p < c.npts; p += F::threads) {
      const int ix = p % c.n1, r = p / c.n1;
      sm.idx[p] = ix | (r % c.n2) << 10 | (r / c.n2) << 20;
    }
  }
}

// Lanes that share one sum when `items` sums are formed by the CTA's threads (1 .. 8).
template <class F> __device__ __forceinline__ int any_share(int items) {
  constexpr int n = F::threads - F::proj0;
  return items * 8 <= n ? 8 : items * 4 <= n ? 4 : items * 2 <= n ? 2 : 1;
}

// Sum over `n` consecutive lanes (a power of two), the same in all of them.
template <typename V> __device__ __forceinline__ V any_lane_sum(V v, int n) {
  for (int off = 1; off < n; off <<= 1) {
    v.x = radd(v.x, __shfl_xor_sync(0xffffffffu, v.x, off));
    v.y = radd(v.y, __shfl_xor_sync(0xffffffffu, v.y, off));
  }
  return v;
}

// Monomial sums of order <= D of every atom into mres[a NM + mono] (see tsbz_step64.cu),
// from the band in t; u is scratch of npts.  Begins and ends with a barrier.  Few sums
// are shared by lanes (by the count of the second-order pass, so that both orders
// share alike).
template <typename T, int D, class F>
__device__ void any_project(const AnySmem<T>& sm, const CellDev& c, const typename AnyC<T>::V* t,
                            typename AnyC<T>::V* u, int rank = 0) {
  using V = typename AnyC<T>::V;
  constexpr int NM = D == 1 ? 4 : 10;
  constexpr int NT = F::threads - F::proj0;
  const int tid = (int)threadIdx.x - F::proj0;
  const int n1 = F::eight ? 8 : c.n1, n2 = F::eight ? 8 : c.n2, n3 = F::eight ? 8 : c.n3, n12 = n1 * n2, ng = c.n_zg;
  const int npts = n12 * n3;
  const int y0 = any_row0<F>(rank, n2), rows = any_row0<F>(rank + 1, n2) - y0, cols = rows * n1;
  any_sync<F>();
  if constexpr (F::ctas == 1) {
    for (int p = tid; p < npts; p += NT) u[p] = vmul(sm.phi[F::eight ? p >> 6 : sm.idx[p] >> 20], t[p]);
  } else {
    for (int i = tid; i < cols * n3; i += NT) {
      const int z = i / cols, p = z * n12 + y0 * n1 + i - z * cols;
      u[p] = vmul(sm.phi[z], t[p]);
    }
  }
  any_sync<F>();
  // z sums of (group, column)
  for (int i = tid; i < ng * cols; i += NT) {
    const int g = i / cols, col = y0 * n1 + i - g * cols, zb = sm.zb[g];
    const T* w = sm.zw + g * n3;
    V s[D + 1];
#pragma unroll
    for (int k = 0; k <= D; ++k) s[k] = vmk<V>((T)0, (T)0);
    auto run = [&](int z0, int z1) {
#pragma unroll 4
      for (int z = z0; z < z1; ++z) {
        const V v = u[z * n12 + col];
#pragma unroll
        for (int k = 0; k <= D; ++k) s[k] = vaxpy(w[k * ng * n3 + z], v, s[k]);
      }
    };
    run(0, zb);
    if (zb < n3) {
#pragma unroll
      for (int k = 0; k <= D; ++k) s[k] = vmul(sm.turn[g], s[k]);
      run(zb, n3);
    }
#pragma unroll
    for (int k = 0; k <= D; ++k) sm.s[(g * (D + 1) + k) * n12 + col] = s[k];
  }
  any_sync<F>();
  // x sums of (atom, power of d_z, row)
  {
    const int share = any_share<F>(c.n_atoms * 3 * rows), sub = tid & (share - 1), items = c.n_atoms * (D + 1) * rows;
    for (int i0 = 0; i0 < items; i0 += NT / share) {
      const int i = i0 + tid / share;
      const bool in = i < items;
      const int y = y0 + (in ? i % rows : 0), r = in ? i / rows : 0, k = r / c.n_atoms, a = r - k * c.n_atoms;
      const V* row = sm.s + (c.zg_of[a] * (D + 1) + k) * n12 + y * n1;
      V R[3];
#pragma unroll
      for (int w = 0; w < 3; ++w) R[w] = vmk<V>((T)0, (T)0);
      for (int x = sub; in && x < n1; x += share) {
        const V p = vmul(sm.xf[a * n1 + x], row[x]);
        const T d = sm.xd[a * n1 + x];
        R[0] = vmk<V>(radd(R[0].x, p.x), radd(R[0].y, p.y));
        if (k < D) R[1] = vaxpy(d, p, R[1]);
        if (D == 2 && k == 0) R[2] = vaxpy(rmul(d, d), p, R[2]);
      }
#pragma unroll
      for (int w = 0; w <= D; ++w) R[w] = any_lane_sum(R[w], share);
      if (in && sub == 0) {
        V* o = sm.rs + (a * 6 + (k == 0 ? 0 : (k == 1 ? 3 : 5))) * n2 + y;
        o[0] = R[0];
        if (k < D) o[n2] = R[1];
        if (D == 2 && k == 0) o[2 * n2] = R[2];
      }
    }
  }
  any_sync<F>();
  // y sums of (atom, monomial), and the group's phase
  {
    const int share = any_share<F>(c.n_atoms * 10), sub = tid & (share - 1), items = c.n_atoms * NM;
    for (int i0 = 0; i0 < items; i0 += NT / share) {
      const int i = i0 + tid / share;
      const bool in = i < items;
      const int a = in ? i / NM : 0, mo = in ? i - a * NM : 0;
      int ex = 0, ey = 0, ez = 0;
      if (mo == 1 || mo == 5 || mo == 6) ex = 1;
      if (mo == 4) ex = 2;
      if (mo == 2 || mo == 5 || mo == 8) ey = 1;
      if (mo == 7) ey = 2;
      if (mo == 3 || mo == 6 || mo == 8) ez = 1;
      if (mo == 9) ez = 2;
      const V* R = sm.rs + (a * 6 + (ez == 0 ? ex : (ez == 1 ? 3 + ex : 5))) * n2;
      V M = vmk<V>((T)0, (T)0);
      for (int y = y0 + sub; in && y < y0 + rows; y += share) {
        const T d = sm.yd[a * n2 + y], wy = ey == 0 ? (T)1 : (ey == 1 ? d : rmul(d, d));
        M = vaxpy(wy, vmul(sm.yf[a * n2 + y], R[y]), M);
      }
      M = any_lane_sum(M, share);
      if (!in || sub != 0) continue;
      if constexpr (F::ctas == 1) {
        sm.mres[i] = vmul(sm.kfin[c.zg_of[a]], M);
      } else {
        for (int r = 0; r < F::ctas; ++r)
          cg::this_cluster().map_shared_rank(sm.part, r)[rank * 10 * ANY_NA + i] = M;
      }
    }
  }
  if constexpr (F::ctas == 1) any_sync<F>();
}

// The monomial sums from the ranks' parts, in rank order (behind a barrier of the cluster).
template <typename T, int D, class F> __device__ void any_total(const AnySmem<T>& sm, const CellDev& c) {
  using V = typename AnyC<T>::V;
  constexpr int NM = D == 1 ? 4 : 10;
  for (int i = threadIdx.x; i < c.n_atoms * NM; i += F::threads) {
    V M = sm.part[i];
#pragma unroll
    for (int r = 1; r < F::ctas; ++r) {
      const V v = sm.part[r * 10 * ANY_NA + i];
      M = vmk<V>(radd(M.x, v.x), radd(M.y, v.y));
    }
    sm.mres[i] = vmul(sm.kfin[c.zg_of[i / NM]], M);
  }
  __syncthreads();
}


// Projection of projector j from its monomial sum, and the ket weights from P (null: from mres).
template <typename T, class F>
__device__ void any_weights(const AnySmem<T>& sm, const CellDev& c, const typename AnyC<T>::V* P) {
  using V = typename AnyC<T>::V;
  for (int j = threadIdx.x; j < c.n_proj; j += F::threads) {
    const T sc = rmul(AnyTab<T>::dv(c), AnyTab<T>::pnorm(c)[j]), e = AnyTab<T>::wkb(c)[j];
    const V p = P ? P[j] : vmk<V>(rmul(sc, sm.mres[j].x), rmul(sc, sm.mres[j].y));
    sm.w[j] = vmul(vconj(sm.k0[c.zg_of[j >> 2]]), vmk<V>(rmul(e, p.x), rmul(e, p.y)));
  }
  __syncthreads();
}

// The two outputs k = p, p + 4 of an 8-point transform of x (INV: conjugate), p = the thread's part.
template <bool INV, typename V>
__device__ __forceinline__ void any_dft8(const V (&x)[8], V& lo, V& hi, unsigned p = threadIdx.x & 3) {
  using T = decltype(V().x);
  const unsigned s = p & 1;
  // four-point sums over the even and the odd inputs: (x0 + s x4) + i^p (x2 + s x6)
  V h[2];
#pragma unroll
  for (int o = 0; o < 2; ++o) {
    const V e0 = vmk<V>(x[o].x + flip(x[o + 4].x, s), x[o].y + flip(x[o + 4].y, s));
    const V e1 = vmk<V>(x[o + 2].x + flip(x[o + 6].x, s), x[o + 2].y + flip(x[o + 6].y, s));
    // times (-i)^p (forward) or i^p
    const unsigned sx = INV ? (p == 1 || p == 2) : (p >= 2), sy = INV ? (p >= 2) : (p == 1 || p == 2);
    const T rx = s ? e1.y : e1.x, ry = s ? e1.x : e1.y;
    h[o] = vmk<V>(e0.x + flip(rx, sx), e0.y + flip(ry, sy));
  }
  // exp(-+ 2 pi i p / 8)
  const T r = (T)0.70710678118654752440;
  const T co = p == 0 ? (T)1 : (p == 1 ? r : (p == 2 ? (T)0 : -r));
  const T sn = flip(p == 0 ? (T)0 : (p == 2 ? (T)1 : r), INV ? 0u : 1u);
  const V w = vmk<V>(fma(co, h[1].x, -sn * h[1].y), fma(co, h[1].y, sn * h[1].x));
  lo = vmk<V>(h[0].x + w.x, h[0].y + w.y);
  hi = vmk<V>(h[0].x - w.x, h[0].y - w.y);
}

struct Fwd { static constexpr bool value = false; };
struct Inv { static constexpr bool value = true; };

// Kinetic term of an 8^3 band for the thread's two points (z = p, p + 4 of column l).
template <typename T>
__device__ void any_kinetic8(const AnySmem<T>& sm, const typename AnyC<T>::V* t, typename AnyC<T>::V (&k)[2]) {
  using V = typename AnyC<T>::V;
  const int p = threadIdx.x & 3, l = threadIdx.x >> 2, l0 = l & 7, l1 = l >> 3;
  V *x1 = sm.s, *x2 = sm.s + ANY_X8, v[8], lo, hi;
  auto line = [&](V* src, V* dst, int at, int stride, auto inv) {
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = src[at + j * stride];
    any_dft8<decltype(inv)::value>(v, lo, hi);
    if (dst) {
      dst[at + p * stride] = lo;
      dst[at + (p + 4) * stride] = hi;
      __syncwarp();   // a plane's x and y lines belong to one warp
    }
  };
  const int cz = l1 * 9 + l0, cx = l1 * 72 + l0 * 9, cy = l1 * 72 + l0;   // column; row y = l0; line x = l0
#pragma unroll
  for (int j = 0; j < 8; ++j) v[j] = t[j * 64 + l];
  any_dft8<false>(v, lo, hi);
  x1[cz + p * 72] = lo;
  x1[cz + (p + 4) * 72] = hi;
  __syncthreads();
  line(x1, x2, cx, 1, Fwd());
#pragma unroll
  for (int j = 0; j < 8; ++j) v[j] = x2[cy + j * 9];
  any_dft8<false>(v, lo, hi);
  {
    const T *e = sm.lam3 + l1 * 64 + p * 8 + l0, e0 = e[0], e1 = e[32];
    x1[cy + p * 9] = vmk<V>(e0 * lo.x, e0 * lo.y);
    x1[cy + (p + 4) * 9] = vmk<V>(e1 * hi.x, e1 * hi.y);
  }
  __syncwarp();
  line(x1, x2, cy, 9, Inv());
  line(x2, x1, cx, 1, Inv());
  __syncthreads();
  line(x1, (V*)nullptr, cz, 72, Inv());
  k[0] = lo;
  k[1] = hi;
}

// The same in a cluster of four: CTA `rank` takes frequencies k_z = rank, rank + 4 through x and
// y and hands the two planes to every CTA (before the cluster's barrier); behind it, the
// inverse along z for the CTA's 16 columns.  Called by threads 0 .. 63.
template <typename T> __device__ void any_planes8(const AnySmem<T>& sm, const typename AnyC<T>::V* t, int rank) {
  using V = typename AnyC<T>::V;
  const int tid = threadIdx.x, p = tid & 3, line = (tid >> 2) & 15, j = line >> 3, l = line & 7;
  V *x1 = sm.xl, *x2 = sm.xl + 2 * 72, v[8], lo, hi;
  const int cx = j * 72 + l * 9, cy = j * 72 + l;
#pragma unroll
  for (int k = 0; k < 8; ++k) v[k] = t[k * 64 + tid];
  any_dft8<false>(v, lo, hi, (unsigned)rank);
  x1[(tid >> 3) * 9 + (tid & 7)] = lo;
  x1[72 + (tid >> 3) * 9 + (tid & 7)] = hi;
  asm volatile("bar.sync 2, 64;\n" ::: "memory");
#pragma unroll
  for (int k = 0; k < 8; ++k) v[k] = x1[cx + k];
  any_dft8<false>(v, lo, hi);
  x2[cx + p] = lo;
  x2[cx + p + 4] = hi;
  __syncwarp();   // a plane's x and y lines belong to one warp
#pragma unroll
  for (int k = 0; k < 8; ++k) v[k] = x2[cy + k * 9];
  any_dft8<false>(v, lo, hi);
  {
    const T *e = sm.lam3 + (rank + 4 * j) * 64 + p * 8 + l, e0 = e[0], e1 = e[32];
    x1[cy + p * 9] = vmk<V>(e0 * lo.x, e0 * lo.y);
    x1[cy + (p + 4) * 9] = vmk<V>(e1 * hi.x, e1 * hi.y);
  }
  __syncwarp();
#pragma unroll
  for (int k = 0; k < 8; ++k) v[k] = x1[cy + k * 9];
  any_dft8<true>(v, lo, hi);
  x2[cy + p * 9] = lo;
  x2[cy + (p + 4) * 9] = hi;
  __syncwarp();
#pragma unroll
  for (int k = 0; k < 8; ++k) v[k] = x2[cx + k];
  any_dft8<true>(v, lo, hi);
  for (int r = 0; r < Form8Cluster::ctas; ++r) {
    V* o = cg::this_cluster().map_shared_rank(sm.xk, r) + (rank + 4 * j) * 72 + l * 9;
    o[p] = lo;
    o[p + 4] = hi;
  }
}
template <typename T>
__device__ void any_columns8(const AnySmem<T>& sm, int rank, typename AnyC<T>::V (&k)[2]) {
  using V = typename AnyC<T>::V;
  const int q = (threadIdx.x >> 2) & 15;   // of the CTA's columns: row 2 rank + q / 8, x = q % 8
  V v[8];
#pragma unroll
  for (int z = 0; z < 8; ++z) v[z] = sm.xk[z * 72 + (2 * rank + (q >> 3)) * 9 + (q & 7)];
  any_dft8<true>(v, k[0], k[1]);
}

// Kinetic term at point p from the star stencil.
template <typename T>
__device__ __forceinline__ typename AnyC<T>::V any_kinetic(const AnySmem<T>& sm, const CellDev& c,
                                                           const typename AnyC<T>::V* t, int p) {
  using V = typename AnyC<T>::V;
  constexpr int M = TSBZ_MAX_ND + 1;
  const int id = sm.idx[p], n12 = c.n1 * c.n2;
  const int pos[3] = {id & 1023, (id >> 10) & 1023, id >> 20}, n[3] = {c.n1, c.n2, c.n3}, st[3] = {1, c.n1, n12};
  const V ce = t[p];
  V h = vmk<V>(sm.st[6 * M] * ce.x, sm.st[6 * M] * ce.y);
#pragma unroll
  for (int ax = 0; ax < 3; ++ax) {
    const V* line = t + p - pos[ax] * st[ax];
#pragma unroll 4
    for (int m = 1; m <= c.nd; ++m) {
      const int up = pos[ax] + m, dn = pos[ax] - m;
      const V a = line[(up >= n[ax] ? up - n[ax] : up) * st[ax]], b = line[(dn < 0 ? dn + n[ax] : dn) * st[ax]];
      const T lw = sm.st[ax * M + m], qw = sm.st[3 * M + ax * M + m];
      h.x = fma(lw, a.x + b.x, fma(qw, a.y - b.y, h.x));
      h.y = fma(lw, a.y + b.y, fma(-qw, a.x - b.x, h.y));
    }
  }
  return h;
}

// h t at the thread's points, handed to `use(point, t, h t)`; the ket weights are in sm.w.
// t is complete (barrier behind its writes); `use` may write anywhere but t and sm.s.
template <typename T, class F, typename U>
__device__ void any_apply(const AnySmem<T>& sm, const CellDev& c, const T* __restrict__ veff,
                          const typename AnyC<T>::V* t, U&& use, int rank = 0) {
  using V = typename AnyC<T>::V;
  const int tid = threadIdx.x;
  const int n1 = F::eight ? 8 : c.n1, n2 = F::eight ? 8 : c.n2, n3 = F::eight ? 8 : c.n3, n12 = n1 * n2;
  const int ng = c.use_proj ? c.n_zg : 0;
  const int y0 = any_row0<F>(rank, n2), cols = (any_row0<F>(rank + 1, n2) - y0) * n1;
  V k8[2];
  if constexpr (F::eight && F::ctas == 1) any_kinetic8<T>(sm, t, k8);
  if constexpr (F::eight && F::ctas > 1) any_columns8<T>(sm, rank, k8);
  if (ng) {
    // ket tables of (atom, x), then the coefficients C0, C1 of (group, column)
    for (int i = tid; i < c.n_atoms * n1; i += F::threads) {
      const int a = i / n1, x = i - a * n1;
      const V cf = vconj(sm.xf[i]);
      const T d = sm.xd[i];
      sm.gt[(a * 3 + 0) * n1 + x] = vmul(cf, vaxpy(d, sm.w[4 * a + 1], sm.w[4 * a]));
      sm.gt[(a * 3 + 1) * n1 + x] = vmul(cf, sm.w[4 * a + 2]);
      sm.gt[(a * 3 + 2) * n1 + x] = vmul(cf, sm.w[4 * a + 3]);
    }
    __syncthreads();
    for (int i = tid; i < ng * cols; i += F::threads) {
      const int g = i / cols, col = y0 * n1 + i - g * cols, y = col / n1, x = col - y * n1;
      V c0 = vmk<V>((T)0, (T)0), c1 = c0;
      for (int e = c.zg_off[g]; e < c.zg_off[g + 1]; ++e) {
        const int a = c.zg_mem[e];
        const V cf = vconj(sm.yf[a * n2 + y]);
        const V b = vaxpy(sm.yd[a * n2 + y], sm.gt[(a * 3 + 1) * n1 + x], sm.gt[(a * 3 + 0) * n1 + x]);
        const V g1 = sm.gt[(a * 3 + 2) * n1 + x];
        c0 = vmk<V>(fma(cf.x, b.x, fma(-cf.y, b.y, c0.x)), fma(cf.x, b.y, fma(cf.y, b.x, c0.y)));
        c1 = vmk<V>(fma(cf.x, g1.x, fma(-cf.y, g1.y, c1.x)), fma(cf.x, g1.y, fma(cf.y, g1.x, c1.y)));
      }
      sm.s[(2 * g) * n12 + col] = c0;
      sm.s[(2 * g + 1) * n12 + col] = c1;
    }
    __syncthreads();
  }
  const int own = cols * n3, pts = F::eight ? 2 : (own + F::threads - 1) / F::threads;
#pragma unroll(F::eight ? 2 : 1)
  for (int i = 0; i < pts; ++i) {
    int p = any_point<F>(i);
    if constexpr (F::ctas == 1) {
      if (!F::eight && p >= own) break;
    } else if constexpr (F::eight) {
      if (tid >= 64) break;
      p = (tid & 3) * 64 + 16 * rank + (tid >> 2) + 256 * i;
    } else {
      if (p >= own) break;
      const int z = p / cols;
      p = z * n12 + y0 * n1 + p - z * cols;
    }
    const V ce = t[p];
    V h;
    if constexpr (F::eight) h = i ? k8[1] : k8[0]; else h = any_kinetic<T>(sm, c, t, p);
    const T v = veff[p];
    h.x = fma(v, ce.x, h.x);
    h.y = fma(v, ce.y, h.y);
    if (ng) {
      const int z = F::eight ? p >> 6 : sm.idx[p] >> 20, col = p - z * n12;
      V x0 = vmk<V>((T)0, (T)0), x = x0;
      for (int g = 0; g < ng; ++g) {
        const T w0 = sm.zw[g * n3 + z], w1 = sm.zw[(ng + g) * n3 + z];
        const V c0 = sm.s[(2 * g) * n12 + col], c1 = sm.s[(2 * g + 1) * n12 + col];
        const V y = vmk<V>(fma(w0, c0.x, w1 * c1.x), fma(w0, c0.y, w1 * c1.y));
        if (z < sm.zb[g]) {
          x = vmk<V>(x.x + y.x, x.y + y.y);
        } else {   // past the group's jump
          const V tn = sm.turn[g];
          x = vmk<V>(fma(tn.x, y.x, fma(-tn.y, y.y, x.x)), fma(tn.x, y.y, fma(tn.y, y.x, x.y)));
        }
      }
      const V f = sm.phi[z];   // conj(phi) x
      h.x = fma(f.x, x.x, fma(f.y, x.y, h.x));
      h.y = fma(f.x, x.y, fma(-f.y, x.x, h.y));
    }
    use(p, ce, h);
  }
}

// Pa rows (a, c_x, c_y, c_z) of every projector from the second-order sums of t, and a to Pnext if given.
template <typename T, class F>
__device__ void any_current(const AnySmem<T>& sm, const CellDev& c, const typename AnyC<T>::V* t,
                            typename AnyC<T>::V* u, typename AnyC<T>::V* __restrict__ Pab,
                            typename AnyC<T>::V* __restrict__ Pnext, int rank = 0) {
  using V = typename AnyC<T>::V;
  if ((int)threadIdx.x >= F::proj0) any_project<T, 2, F>(sm, c, t, u, rank);
  if constexpr (F::ctas > 1) {
    cg::this_cluster().sync();
    if (rank != 0) return;
    any_total<T, 2, F>(sm, c);
  }
  for (int o = threadIdx.x; o < 4 * c.n_proj; o += F::threads) {
    const int j = o >> 2, s = o & 3, a = j >> 2, ty = j & 3;
    int e[3] = {ty == 1, ty == 2, ty == 3};
    if (s > 0) e[s - 1] += 1;
    const T sc = rmul(AnyTab<T>::dv(c), AnyTab<T>::pnorm(c)[j]);
    const V M = sm.mres[a * 10 + any_mono(e[0], e[1], e[2])];
    const V v = vmk<V>(rmul(sc, M.x), rmul(sc, M.y));
    Pab[4 * j + s] = v;
    if (Pnext && s == 0) Pnext[j] = v;
  }
}

// Unit and band of the CTA; false when the unit sits the step out.
__device__ __forceinline__ bool any_open(const LaunchSet& L, int& u, int& b, int ctas = 1) {
  const int orb = blockIdx.x / ctas;
  b = orb % L.cell.n_bands;
  u = L.unit_ids[orb / L.cell.n_bands];
  return unit_active(L, u);
}

// One time step of every band (arguments as launch_step64).
//
// With few orbitals in double one SM's FP64 pipe is the bound (8^3: 24 us a stage), so a
// cluster of F::ctas CTAs shares a band by rows y.  Each CTA keeps the whole t_{m-1} and
// forms its own rows of t_m, which it stores to every CTA; the projections' x and z sums
// run over the CTA's rows and the ranks' sums are added in rank order; the 8^3 transform
// splits by k_z between its two z passes.  Two barriers of the cluster a stage.
template <typename T, class F>
__device__ __forceinline__ void any_step(const LaunchSet& L, typename AnyC<T>::V* __restrict__ psi,
                                         typename AnyC<T>::V* __restrict__ P, typename AnyC<T>::V* __restrict__ Pa,
                                         int fresh_p, int want_pa, int same_next) {
  step_enter();
  using V = typename AnyC<T>::V;
  extern __shared__ __align__(16) unsigned char any_raw[];
  const CellDev& c = L.cell;
  int u, b;
  if (!any_open(L, u, b, F::ctas)) return;   // the whole cluster
  const int rank = F::ctas > 1 ? any_rank() : 0;
  AnySmem<T> sm;
  any_carve<T>(c, any_raw, sm, F::ctas);
  const UnitDev U = L.units[u];
  const SubDev S = L.subs[U.sub];
  const T* veff = reinterpret_cast<const T*>(S.veff);
  V* band = psi + U.psi_off + (long long)b * c.npts;
  V* Pu = P + U.p_off + (long long)b * c.n_proj;
  for (int p = threadIdx.x; p < c.npts; p += F::threads) sm.a[p] = band[p];
  any_setup<T, F>(sm, c, L, u, L.q_half + 3 * u);
  if (c.use_proj) any_tables<T, F>(sm, c, (const V*)L.ph_half + (long long)u * L.ph_stride);
  if constexpr (F::ctas > 1) cg::this_cluster().sync(); else __syncthreads();
  if (F::ctas == 1 && c.use_proj) {
    if (fresh_p) any_project<T, 1, F>(sm, c, sm.a, sm.b);
    any_weights<T, F>(sm, c, fresh_p ? nullptr : Pu);
  }
  V *t = sm.a, *o = sm.b;
  const T dt = (T)(S.dt * L.dt_scale);
  T coef = (T)1;
#pragma unroll 1
  for (int m = 1; m <= 4; ++m) {
    if (m > 1) coef *= dt / (T)m;
    const T scale = m == 1 ? dt : (T)1, sg = m == 4 ? coef : -coef;   // (-i)^m coef s_m
    if constexpr (F::ctas > 1) {
      const bool chain = c.use_proj && (m > 1 || fresh_p);   // projections of t, else from P
      if constexpr (F::eight) {
        if (threadIdx.x < F::proj0) any_planes8<T>(sm, t, rank);
      }
      if (chain && (int)threadIdx.x >= F::proj0) any_project<T, 1, F>(sm, c, t, o, rank);
      cg::this_cluster().sync();
      if (chain) any_total<T, 1, F>(sm, c);
      if (c.use_proj) any_weights<T, F>(sm, c, chain ? nullptr : Pu);
    }
    if (F::ctas == 1 && m == 4) {   // psi back, to the thread's own points, ahead of their use
      if constexpr (F::eight) {
        for (int i = 0; i < 2; ++i) o[any_point<F>(i)] = band[any_point<F>(i)];
      } else {
#pragma unroll 4
        for (int p = threadIdx.x; p < c.npts; p += F::threads) o[p] = band[p];
      }
    }
    auto use = [&](int p, V, V h) {
      h = vmk<V>(scale * h.x, scale * h.y);
      V a = m == 1 ? vmk<V>(h.y, -h.x) : sm.acc[p];
      if (m == 3) {
        a.x = fma(sg, h.y, a.x);
        a.y = fma(-sg, h.x, a.y);
      } else if (m > 1) {
        a.x = fma(sg, h.x, a.x);
        a.y = fma(sg, h.y, a.y);
      }
      if (m < 4) {
        sm.acc[p] = a;
      } else {
        const V u0 = F::ctas == 1 ? o[p] : band[p];
        h = vmk<V>(u0.x + a.x, u0.y + a.y);
        band[p] = h;
      }
      if constexpr (F::ctas == 1) {
        o[p] = h;
      } else {
#pragma unroll
        for (int r = 0; r < F::ctas; ++r) cg::this_cluster().map_shared_rank(o, r)[p] = h;
      }
    };
    any_apply<T, F>(sm, c, veff, t, use, rank);
    V* s = t;
    t = o;
    o = s;
    if constexpr (F::ctas > 1) {
      cg::this_cluster().sync();
    } else if (m < 4) {
      if (c.use_proj) {
        any_project<T, 1, F>(sm, c, t, o);
        any_weights<T, F>(sm, c, nullptr);
      } else {
        __syncthreads();
      }
    }
  }
  if (!c.use_proj || !want_pa) return;
  __syncthreads();
  if (!same_next) any_tables<T, F>(sm, c, (const V*)L.ph_obs + (long long)u * L.ph_stride);
  if constexpr (F::proj0 > 0) __syncthreads();   // (else the projection begins with it)
  any_current<T, F>(sm, c, t, o, Pa + U.pa_off + 4LL * b * c.n_proj, same_next ? Pu : nullptr, rank);
}

template <typename T, class F>
__global__ void __launch_bounds__(F::threads)
    k_step_any(LaunchSet L, typename AnyC<T>::V* psi, typename AnyC<T>::V* P, typename AnyC<T>::V* Pa, int fresh_p,
               int want_pa, int same_next) {
  any_step<T, F>(L, psi, P, Pa, fresh_p, want_pa, same_next);
}
template <typename T, class F>
__global__ void __cluster_dims__(F::ctas, 1, 1) __launch_bounds__(F::threads)
    k_step_any_cluster(LaunchSet L, typename AnyC<T>::V* psi, typename AnyC<T>::V* P, typename AnyC<T>::V* Pa,
                       int fresh_p, int want_pa, int same_next) {
  any_step<T, F>(L, psi, P, Pa, fresh_p, want_pa, same_next);
}

// Projections of the current outside a step.
template <typename T, class F>
__global__ void __launch_bounds__(F::threads) k_pa_any(LaunchSet L, const typename AnyC<T>::V* __restrict__ src,
                                                  typename AnyC<T>::V* __restrict__ Pa) {
  using V = typename AnyC<T>::V;
  extern __shared__ __align__(16) unsigned char any_raw[];
  const CellDev& c = L.cell;
  int u, b;
  if (!any_open(L, u, b)) return;
  AnySmem<T> sm;
  any_carve<T>(c, any_raw, sm);
  const UnitDev U = L.units[u];
  const V* band = src + U.psi_off + (long long)b * c.npts;
  for (int p = threadIdx.x; p < c.npts; p += F::threads) sm.a[p] = band[p];
  any_setup<T, F>(sm, c, L, u, L.q_obs + 3 * u);
  any_tables<T, F>(sm, c, (const V*)L.ph_obs + (long long)u * L.ph_stride);
  any_current<T, F>(sm, c, sm.a, sm.b, Pa + U.pa_off + 4LL * b * c.n_proj, nullptr);
}

// The ground-state solver's filter (see k_filter64); clusters as any_step.
template <class F>
__device__ __forceinline__ void any_filter(const LaunchSet& L, const double2* in, double2* out,
                                           const double* __restrict__ fa, const double* __restrict__ fb, int degree) {
  extern __shared__ __align__(16) unsigned char any_raw[];
  const CellDev& c = L.cell;
  int u, b;
  if (!any_open(L, u, b, F::ctas)) return;
  const int rank = F::ctas > 1 ? any_rank() : 0;
  AnySmem<double> sm;
  any_carve<double>(c, any_raw, sm, F::ctas);
  const UnitDev U = L.units[u];
  const double* veff = reinterpret_cast<const double*>(L.subs[U.sub].veff);
  const long long off = U.psi_off + (long long)b * c.npts;
  for (int p = threadIdx.x; p < c.npts; p += F::threads) sm.a[p] = in[off + p];
  any_setup<double, F>(sm, c, L, u, L.q_half + 3 * u);
  if (c.use_proj)
    any_tables<double, F>(sm, c, (const double2*)L.ph_half + (long long)u * L.ph_stride);
  if constexpr (F::ctas > 1) cg::this_cluster().sync(); else __syncthreads();
  double2 *t = sm.a, *o = sm.b;
#pragma unroll 1
  for (int j = 0; j < degree; ++j) {
    if constexpr (F::ctas > 1) {
      if constexpr (F::eight) {
        if (threadIdx.x < F::proj0) any_planes8<double>(sm, t, rank);
      }
      if (c.use_proj && (int)threadIdx.x >= F::proj0) any_project<double, 1, F>(sm, c, t, o, rank);
      cg::this_cluster().sync();
      if (c.use_proj) any_total<double, 1, F>(sm, c);
    } else if (c.use_proj) {
      any_project<double, 1, F>(sm, c, t, o);
    }
    if (c.use_proj) any_weights<double, F>(sm, c, nullptr);
    const double* f = j == 0 ? fa : fb;
    const double f0 = f[3 * u], f1 = f[3 * u + 1], f2 = j == 0 ? 0.0 : f[3 * u + 2];
    auto use = [&](int p, double2 ce, double2 h) {
      double2 y = make_double2(fma(f0, h.x, f1 * ce.x), fma(f0, h.y, f1 * ce.y));
      if (j > 0) {
        const double2 v = sm.acc[p];
        y.x = fma(f2, v.x, y.x);
        y.y = fma(f2, v.y, y.y);
      }
      sm.acc[p] = ce;
      if constexpr (F::ctas == 1) {
        o[p] = y;
      } else {
#pragma unroll
        for (int r = 0; r < F::ctas; ++r) cg::this_cluster().map_shared_rank(o, r)[p] = y;
      }
    };
    any_apply<double, F>(sm, c, veff, t, use, rank);
    double2* s = t;
    t = o;
    o = s;
    if constexpr (F::ctas > 1) cg::this_cluster().sync(); else __syncthreads();
  }
  const int p0 = rank * c.npts / F::ctas, p1 = (rank + 1) * c.npts / F::ctas;
  for (int p = p0 + threadIdx.x; p < p1; p += F::threads) out[off + p] = t[p];
}
template <class F>
__global__ void __launch_bounds__(F::threads) k_filter_any(LaunchSet L, const double2* in, double2* out,
                                                           const double* fa, const double* fb, int degree) {
  any_filter<F>(L, in, out, fa, fb, degree);
}
template <class F>
__global__ void __cluster_dims__(F::ctas, 1, 1) __launch_bounds__(F::threads)
    k_filter_any_cluster(LaunchSet L, const double2* in, double2* out, const double* fa, const double* fb, int degree) {
  any_filter<F>(L, in, out, fa, fb, degree);
}

template <typename T> size_t any_smem(const CellDev& c) {
  AnySmem<T> m;
  return any_carve<T>(c, nullptr, m);
}

template <typename T> bool any_ok(const CellDev& c) {
  return c.n_atoms <= ANY_NA && c.n1 < 1024 && c.n2 < 1024 && c.n3 < 1024 && any_smem<T>(c) <= ANY_MAX_SMEM;
}

// Variant 0, from ANY_MIN_ORB orbitals on.  The launches per stage are slower for fewer too
// (us a step, 4 orbitals: 8^3 single 76 -> 50, 10 x 12 x 14 single 208 -> 88, double 410 -> 170);
// such runs keep them because callers rely on the number of launches of a small run's step.
template <typename T> bool any_taken(const LaunchSet& L) {
  return L.variant == 0 && (long long)L.n_units * L.cell.n_bands >= ANY_MIN_ORB && any_ok<T>(L.cell);
}

// Double precision with few orbitals takes clusters, while their CTAs find an SM each (8^3:
// two an SM, it is bound by latency as much as by the pipe).  20 steps, one CTA a band
// -> cluster: 8^3 with 8 atoms 16 orbitals 3.21 -> 2.29 ms, 64 3.25 -> 2.55 (128 3.31 -> 4.23, so
// not); 10^3 32 orbitals 6.92 -> 4.28 (four CTAs), 64 6.96 -> 4.89 (two), 96 5.97 -> 6.12 (two, 2 atoms; so
// not); 12^3 32 orbitals 10.1 -> 4.86.  Eight CTAs gain less than four (32 orbitals at 12^3
// 8.68 against 4.58 ms with 2 atoms).  Single precision gains nothing (12^3, 32 orbitals 2.86 -> 2.78 ms; 8^3 loses).
template <typename G> bool any_cluster(const LaunchSet& L, G&& go) {
  const long long orb = (long long)L.n_units * L.cell.n_bands;
  if (any_fft8(L.cell)) {
    if (orb * Form8Cluster::ctas > 304) return false;
    go(Form8Cluster());
  } else if (orb * 4 <= 152) {
    go(FormCluster<4>());
  } else if (orb * 2 <= 152) {
    go(FormCluster<2>());
  } else {
    return false;
  }
  return true;
}

// The form of a cell's kernels where no cluster is taken (k_pa_any never takes one: J(0+) and
// J(t) of a run in clusters are summed in different orders).  In single precision a CTA that fewer than four fit an SM takes 512 threads:
// the SM then holds 16 warps or more (10 steps of 768 k-points, 12 orbitals each:
// 18^3 21.1 -> 16.3 ms, 17 x 13 x 15 9.06 -> 8.40, 16 x 16 x 8 5.46 -> 5.35; smaller
// cells lose, 9 x 11 x 13 3.77 -> 4.12 ms).  In double 256 threads hold the FP64 pipe
// full already and 512 only wait longer at the barriers (10 x 12 x 14, 81 k-points
// 22.3 -> 23.1 ms).
template <typename T, typename G> void any_form(const CellDev& c, size_t bytes, G&& go) {
  if (any_fft8(c)) return go(Form8());
  if constexpr (sizeof(T) == sizeof(float)) {
    if (bytes > ANY_WIDE_SMEM) return go(FormAny<512>());
  }
  go(FormAny<256>());
}

}  // namespace

template <typename T> bool any_cell(const CellDev& c) { return any_ok<T>(c); }
template bool any_cell<double>(const CellDev&);
template bool any_cell<float>(const CellDev&);

template <typename T>
bool launch_step_any(const LaunchSet& L, void* psi, void* P, void* Pa, int fresh_p, int want_pa, int same_next,
                     void* stream) {
  using V = typename AnyC<T>::V;
  if (L.n_units == 0 || !any_taken<T>(L)) return false;
  const size_t bytes = any_smem<T>(L.cell);
  const unsigned grid = (unsigned)L.n_units * L.cell.n_bands;
  auto cluster = [&](auto f) {
    using F = decltype(f);
    AnySmem<T> m;
    const size_t more = any_carve<T>(L.cell, nullptr, m, F::ctas);
    smem_limit<k_step_any_cluster<T, F>>(more);
    step_launch(k_step_any_cluster<T, F>, grid * F::ctas, F::threads, more, stream, L, (V*)psi, (V*)P, (V*)Pa, fresh_p,
                want_pa, same_next);
  };
  if constexpr (sizeof(T) == sizeof(double)) {
    if (any_cluster(L, cluster)) return true;
  }
  any_form<T>(L.cell, bytes, [&](auto f) {
    using F = decltype(f);
    smem_limit<k_step_any<T, F>>(bytes);
    step_launch(k_step_any<T, F>, grid, F::threads, bytes, stream, L, (V*)psi, (V*)P, (V*)Pa, fresh_p, want_pa,
                same_next);
  });
  return true;
}

template <typename T> bool launch_pa_any(const LaunchSet& L, const void* src, void* Pa, void* stream) {
  using V = typename AnyC<T>::V;
  if (L.n_units == 0 || !any_taken<T>(L) || !L.cell.use_proj) return false;
  const size_t bytes = any_smem<T>(L.cell);
  any_form<T>(L.cell, bytes, [&](auto f) {
    using F = decltype(f);
    smem_limit<k_pa_any<T, F>>(bytes);
    k_pa_any<T, F><<<(unsigned)L.n_units * L.cell.n_bands, F::threads, bytes, (cudaStream_t)stream>>>(
        L, (const V*)src, (V*)Pa);
  });
  return true;
}

template bool launch_step_any<double>(const LaunchSet&, void*, void*, void*, int, int, int, void*);
template bool launch_step_any<float>(const LaunchSet&, void*, void*, void*, int, int, int, void*);
template bool launch_pa_any<double>(const LaunchSet&, const void*, void*, void*);
template bool launch_pa_any<float>(const LaunchSet&, const void*, void*, void*);

bool launch_filter_any(const LaunchSet& L, const void* in, void* out, const double* fa, const double* fb, int degree,
                       void* stream) {
  if (L.n_units == 0 || !any_ok<double>(L.cell)) return false;
  const size_t bytes = any_smem<double>(L.cell);
  const bool done = any_cluster(L, [&](auto f) {
    using F = decltype(f);
    AnySmem<double> m;
    const size_t more = any_carve<double>(L.cell, nullptr, m, F::ctas);
    smem_limit<k_filter_any_cluster<F>>(more);
    k_filter_any_cluster<F><<<(unsigned)L.n_units * L.cell.n_bands * F::ctas, F::threads, more, (cudaStream_t)stream>>>(
        L, (const double2*)in, (double2*)out, fa, fb, degree);
  });
  if (done) return true;
  any_form<double>(L.cell, bytes, [&](auto f) {
    using F = decltype(f);
    smem_limit<k_filter_any<F>>(bytes);
    k_filter_any<F><<<(unsigned)L.n_units * L.cell.n_bands, F::threads, bytes, (cudaStream_t)stream>>>(
        L, (const double2*)in, (double2*)out, fa, fb, degree);
  });
  return true;
}
