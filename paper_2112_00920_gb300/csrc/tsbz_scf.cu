// Kernels of the ground-state solver (FP64): Chebyshev-filtered subspace
// iteration for the n_bands lowest eigenvectors of h_k[v_eff] at A = 0, per
// k-point.  The filter steps run in the point-parallel stage kernel (m = 0);
// the kernels here orthonormalise the filtered block and bound its spectrum.
//
// The filtered block is very ill-conditioned (the filter amplifies the lowest
// occupied states by many orders of magnitude more than the highest), so it
// is orthonormalised by shifted CholeskyQR3 (Fukaya, Kannan, Nakatsukasa,
// Zhang, Yamamoto, SIAM J. Sci. Comput. 42 (2020)): one Cholesky-QR pass of
// the Gram matrix plus a small multiple of its trace on the diagonal, then two
// plain Cholesky-QR passes of the rotated block.  The bound of the block's
// spectrum (the largest Ritz value) comes from h applied to the final
// orthonormal block Q: carried through the ill-conditioned passes by
// congruence, C^H (Y^H h Y) C loses every digit in the directions that the
// filter left small.
//
// Per unit (k-point) with the block Y (n_b columns); the n_b x n_b matrices of
// unit i (row-major, pitch n_b) start at i n_b^2 in each buffer:
//   S = dV Y^H Y (and Hs = dV Y^H (h Y) when h Y is given)
//                                             (k_scf_gram, k_scf_gram_sum)
//   S + s I = L L^H,  C = L^{-H}  (orthonormalisation pass), or
//   S = L L^H,  lam = largest eigenvalue of L^{-1} Hs L^{-H}  (bound pass)
//                                             (k_scf_ortho, one CTA per unit)
//   Y' = Y C                                  (k_scf_rotate, out of place)
#include <cuda_runtime.h>

#include "tsbz_internal.h"
#include "tsbz_launch.cuh"

#define SCF_MAXB 256   // bands a unit may have in the ground-state solver
#define SCF_T 16       // band tile edge of the Gram kernel
#define SCF_CH 16      // points per staged chunk of the Gram kernel
#define SCF_RB 16      // output bands per CTA of the rotation
#define SCF_OT 256     // threads of the factorisation kernel (>= SCF_MAXB)

namespace {

__device__ __forceinline__ double2 zmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 zconj(double2 a) { return make_double2(a.x, -a.y); }
__device__ __forceinline__ double2 zadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 zsub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }

// One 16 x 16 tile (rows t1, columns t2 <= t1) of S (and Hs when WH) of one unit over
// one chunk of points: CTA (unit, tile, chunk), one entry per thread.  Bands t1 of Y and
// bands t2 of Y and HY are staged SCF_CH points at a time.  Bound by FP64
// operations, four per entry and point: S and Hs are Hermitian, so only the lower
// triangle's tiles are formed, and the points are split into chunks until the CTAs
// fill the GPU (k_scf_gram_sum adds them in order).  8 units of 16 bands at 8^3:
// 887 -> 19 us (one 32 x 32 tile over all points per unit before).
template <bool WH>
__global__ void __launch_bounds__(256) k_scf_gram(LaunchSet L, const double2* __restrict__ Y,
                                                  const double2* __restrict__ HY, double2* __restrict__ G,
                                                  int tiles, int chunk) {
  __shared__ double2 y1[SCF_T][SCF_CH + 1];
  __shared__ double2 y2[SCF_T][SCF_CH + 1];
  __shared__ double2 h2[SCF_T][SCF_CH + 1];
  const CellDev& c = L.cell;
  const int u = L.unit_ids[blockIdx.x];
  const UnitDev U = L.units[u];
  const int nb = c.n_bands;
  int t1 = 0, t2 = blockIdx.y;   // tile index t1 (t1 + 1) / 2 + t2
  while (t2 > t1) t2 -= ++t1;
  const double2* yb = Y + U.psi_off;
  const double2* hb = HY + U.psi_off;
  const int col = threadIdx.x & (SCF_T - 1), row = threadIdx.x / SCF_T;
  const double2 z = make_double2(0.0, 0.0);
  double2 sacc = z, hacc = z;
  const int p_end = min(c.npts, ((int)blockIdx.z + 1) * chunk);
  for (int p0 = blockIdx.z * chunk; p0 < p_end; p0 += SCF_CH) {
    __syncthreads();
    for (int i = threadIdx.x; i < SCF_T * SCF_CH; i += 256) {
      const int b = i / SCF_CH, k = i % SCF_CH, p = p0 + k;
      const int g1 = t1 * SCF_T + b, g2 = t2 * SCF_T + b;
      const bool in = p < p_end;
      y1[b][k] = in && g1 < nb ? yb[(long long)g1 * c.npts + p] : z;
      y2[b][k] = in && g2 < nb ? yb[(long long)g2 * c.npts + p] : z;
      if (WH) h2[b][k] = in && g2 < nb ? hb[(long long)g2 * c.npts + p] : z;
    }
    __syncthreads();
#pragma unroll 4
    for (int k = 0; k < SCF_CH; ++k) {
      const double2 a1 = y1[row][k], a2 = y2[col][k];   // conj(a1) a2
      sacc.x = fma(a1.x, a2.x, fma(a1.y, a2.y, sacc.x));
      sacc.y = fma(a1.x, a2.y, fma(-a1.y, a2.x, sacc.y));
      if (WH) {
        const double2 g2 = h2[col][k];
        hacc.x = fma(a1.x, g2.x, fma(a1.y, g2.y, hacc.x));
        hacc.y = fma(a1.x, g2.y, fma(-a1.y, g2.x, hacc.y));
      }
    }
  }
  double2* g = G + (((long long)blockIdx.x * gridDim.z + blockIdx.z) * tiles + blockIdx.y) * 2 * 256 + threadIdx.x;
  g[0] = sacc;
  if (WH) g[256] = hacc;
}

// S (and Hs) of one unit from the chunks' tiles, added in chunk order; the upper triangle mirrored.
template <bool WH>
__global__ void __launch_bounds__(256) k_scf_gram_sum(int nb, double dv, const double2* __restrict__ G,
                                                      double2* __restrict__ Sout, double2* __restrict__ Hout,
                                                      int tiles, int chunks) {
  int t1 = 0, t2 = blockIdx.y;
  while (t2 > t1) t2 -= ++t1;
  const int i = t1 * SCF_T + threadIdx.x / SCF_T, j = t2 * SCF_T + (threadIdx.x & (SCF_T - 1));
  if (i >= nb || j >= nb || j > i) return;
  const double2* g = G + ((long long)blockIdx.x * chunks * tiles + blockIdx.y) * 2 * 256 + threadIdx.x;
  const long long o = (long long)blockIdx.x * nb * nb;
#pragma unroll
  for (int w = 0; w < (WH ? 2 : 1); ++w) {
    double2 s = make_double2(0.0, 0.0);
    for (int k = 0; k < chunks; ++k) s = zadd(s, g[(long long)k * tiles * 2 * 256 + w * 256]);
    s = make_double2(dv * s.x, dv * s.y);
    double2* M = (w ? Hout : Sout) + o;
    if (i == j) s.y = 0.0;
    M[(long long)i * nb + j] = s;
    if (i != j) M[(long long)j * nb + i] = zconj(s);
  }
}

// One CTA per unit (blockIdx.x): Cholesky S + s I = L L^H (right-looking, in
// W1; s = shift_coef tr S), Li = L^{-1} (one column per thread, in W2) and
// C = L^{-H}; when want_lam is set, also A = L^{-1} Hs L^{-H} over Hs (T =
// Hs L^{-H} in W1 first) and its largest eigenvalue by power iteration on
// A + shift (Gershgorin shift, and a little more, so that A + shift is positive definite: a
// multiple of the identity, as one band has, would leave a zero matrix to iterate with).
// The matrices live in global memory (they stay in L2); every sum runs in a
// fixed order.  status bit 4: S + s I not positive definite.
__global__ void __launch_bounds__(SCF_OT) k_scf_ortho(int nb, double shift_coef, int want_lam,
                                                      const double2* __restrict__ Sg, double2* __restrict__ Hg,
                                                      double2* __restrict__ Cg, double2* __restrict__ W1g,
                                                      double2* __restrict__ W2g, double* __restrict__ lam,
                                                      int* __restrict__ bad) {
  __shared__ double2 v[SCF_MAXB], w[SCF_MAXB];
  __shared__ double red[1][SCF_OT];
  __shared__ double sc[3];
  __shared__ int okf;
  const long long o = (long long)blockIdx.x * nb * nb;
  const double2* S = Sg + o;
  double2* A = Hg + o;   // Hs on entry, L^{-1} Hs L^{-H} on exit (want_lam)
  double2* C = Cg + o;
  double2* Lm = W1g + o;
  double2* Li = W2g + o;
  const int tid = threadIdx.x, nt = blockDim.x, n2 = nb * nb;
  const double2 z = make_double2(0.0, 0.0);
  for (int i = tid; i < n2; i += nt) Lm[i] = S[i];
  if (tid == 0) {
    okf = 1;
    double tr = 0.0;
    for (int i = 0; i < nb; ++i) tr += S[i * nb + i].x;
    sc[0] = shift_coef * tr;
  }
  __syncthreads();
  for (int i = tid; i < nb; i += nt) Lm[i * nb + i].x += sc[0];
  __syncthreads();
  // Cholesky, lower triangle of Lm; column j is final after step j
  for (int j = 0; j < nb; ++j) {
    const double d = Lm[j * nb + j].x;
    const double ljj = sqrt(d > 0.0 ? d : 1e-300);
    for (int i = j + 1 + tid; i < nb; i += nt) {
      const double2 x = Lm[i * nb + j];
      Lm[i * nb + j] = make_double2(x.x / ljj, x.y / ljj);
    }
    __syncthreads();
    if (tid == 0) {
      Lm[j * nb + j] = make_double2(ljj, 0.0);
      if (!(d > 0.0)) okf = 0;
    }
    const int m = nb - j - 1;
    for (int idx = tid; idx < m * m; idx += nt) {
      const int i = j + 1 + idx / m, k = j + 1 + idx % m;
      if (k <= i) Lm[i * nb + k] = zsub(Lm[i * nb + k], zmul(Lm[i * nb + j], zconj(Lm[k * nb + j])));
    }
    __syncthreads();
  }
  // Li = L^{-1}: column jj by forward substitution
  for (int jj = tid; jj < nb; jj += nt) {
    for (int i = 0; i < jj; ++i) Li[i * nb + jj] = z;
    Li[jj * nb + jj] = make_double2(1.0 / Lm[jj * nb + jj].x, 0.0);
    for (int i = jj + 1; i < nb; ++i) {
      double2 s = z;
      for (int k = jj; k < i; ++k) s = zadd(s, zmul(Lm[i * nb + k], Li[k * nb + jj]));
      const double lii = Lm[i * nb + i].x;
      Li[i * nb + jj] = make_double2(-s.x / lii, -s.y / lii);
    }
  }
  __syncthreads();
  // C = L^{-H} (upper triangular)
  for (int idx = tid; idx < n2; idx += nt) C[idx] = zconj(Li[(idx % nb) * nb + idx / nb]);
  if (!want_lam) {
    if (tid == 0 && !okf) atomicOr(bad, 4);
    return;
  }
  // T = Hs L^{-H} into Lm (Hs is in A)
  for (int idx = tid; idx < n2; idx += nt) {
    const int i = idx / nb, j = idx % nb;
    double2 s = z;
    for (int k = 0; k <= j; ++k) s = zadd(s, zmul(A[i * nb + k], zconj(Li[j * nb + k])));
    Lm[idx] = s;
  }
  __syncthreads();
  // A = L^{-1} T (Hs was last read in the previous loop)
  for (int idx = tid; idx < n2; idx += nt) {
    const int i = idx / nb, j = idx % nb;
    double2 s = z;
    for (int k = 0; k <= i; ++k) s = zadd(s, zmul(Li[i * nb + k], Lm[k * nb + j]));
    A[idx] = s;
  }
  __syncthreads();
  // Gershgorin lower bound of the Hermitian A
  double gl = 1e300;
  for (int i = tid; i < nb; i += nt) {
    double r = 0.0;
    for (int j = 0; j < nb; ++j)
      if (j != i) r += sqrt(A[i * nb + j].x * A[i * nb + j].x + A[i * nb + j].y * A[i * nb + j].y);
    gl = fmin(gl, A[i * nb + i].x - r);
  }
  red[0][tid] = gl;
  for (int i = tid; i < nb; i += nt) v[i] = make_double2(1.0 + 0.01 * i, 0.0);
  __syncthreads();
  if (tid == 0) {
    double lo = red[0][0];
    for (int i = 1; i < min(nb, nt); ++i) lo = fmin(lo, red[0][i]);
    sc[0] = -lo + 1e-6 * (1.0 + fabs(lo));
  }
  __syncthreads();
  const double shift = sc[0];
  // 200 steps of power iteration on A + shift.  FP64 instructions on the chain are
  // what it costs: the rows are shared by `parts` threads each, small matrices
  // are squared three times first (25 steps of the eighth power), and the vector is
  // normalised every eighth step only.
  double2* M = Lm;       // A + shift, and its squares
  double2* M2 = Li;
  for (int i = tid; i < n2; i += nt) {
    M[i] = A[i];
    if (i / nb == i % nb) M[i].x += shift;
  }
  __syncthreads();
  int steps = 200;
  if (nb <= 32)
    for (int q = 0; q < 3; ++q) {
      steps /= 2;
      if (tid == 0) {
        double tr = 0.0;
        for (int i = 0; i < nb; ++i) tr += M[i * nb + i].x;
        sc[1] = tr > 0.0 ? 1.0 / tr : 1.0;   // eigenvalues of M / tr M are at most 1
      }
      __syncthreads();
      const double f = sc[1] * sc[1];
      for (int idx = tid; idx < n2; idx += nt) {
        const int i = idx / nb, j = idx % nb;
        double2 s = z;
        for (int k = 0; k < nb; ++k) s = zadd(s, zmul(M[i * nb + k], M[k * nb + j]));
        M2[idx] = make_double2(f * s.x, f * s.y);
      }
      __syncthreads();
      double2* t = M;
      M = M2;
      M2 = t;
    }
  int parts = 1;
  while (parts < 32 && 2 * parts * nb <= nt) parts *= 2;
  const int part = tid & (parts - 1);
  // w = B v for all rows (row tid / parts, ...); ends with a barrier
  auto apply = [&](const double2* B) {
    for (int i0 = 0; i0 < nb; i0 += nt / parts) {
      const int i = i0 + tid / parts;
      double2 s = z;
      if (i < nb)
        for (int j = part; j < nb; j += parts) s = zadd(s, zmul(B[i * nb + j], v[j]));
      for (int off = parts / 2; off > 0; off /= 2) {
        s.x += __shfl_xor_sync(0xffffffffu, s.x, off);
        s.y += __shfl_xor_sync(0xffffffffu, s.y, off);
      }
      if (i < nb && part == 0) w[i] = s;
    }
    __syncthreads();
  };
  // sums over the rows of |v|^2 and Re(conj(v) w), and of |w|^2, by warp 0 (fixed order)
  auto sums = [&]() {
    if (tid < 32) {
      double a = 0.0, b = 0.0, d = 0.0;
      for (int i = tid; i < nb; i += 32) {
        a = fma(v[i].x, v[i].x, fma(v[i].y, v[i].y, a));
        b = fma(v[i].x, w[i].x, fma(v[i].y, w[i].y, b));
        d = fma(w[i].x, w[i].x, fma(w[i].y, w[i].y, d));
      }
      for (int off = 16; off > 0; off >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, off);
        b += __shfl_xor_sync(0xffffffffu, b, off);
        d += __shfl_xor_sync(0xffffffffu, d, off);
      }
      if (tid == 0) {
        sc[0] = a;
        sc[1] = b;
        sc[2] = d;
      }
    }
    __syncthreads();
  };
  for (int it = 0; it < steps; ++it) {
    apply(M);
    double f = 1.0;
    if (it % 8 == 7) {
      sums();
      f = rsqrt(sc[2]);
    }
    for (int i = tid; i < nb; i += nt) v[i] = make_double2(f * w[i].x, f * w[i].y);
    __syncthreads();
  }
  apply(A);
  sums();
  if (tid == 0) {
    lam[blockIdx.x] = sc[1] / sc[0];
    if (!okf) atomicOr(bad, 4);
  }
}

// Y'[:, b] = sum_{k <= b} Y[:, k] C[k][b] for the SCF_RB bands of blockIdx.y,
// one point per thread (blockIdx.z selects the point block), out of place.
// The rows of C that the tile needs are staged in shared memory.
__global__ void __launch_bounds__(128) k_scf_rotate(LaunchSet L, const double2* __restrict__ Y,
                                                    const double2* __restrict__ Cg, double2* __restrict__ Yout) {
  extern __shared__ double2 cs[];   // [k][SCF_RB], k < kend
  const CellDev& c = L.cell;
  const int u = L.unit_ids[blockIdx.x];
  const UnitDev U = L.units[u];
  const int nb = c.n_bands, b0 = blockIdx.y * SCF_RB, nbt = min(SCF_RB, nb - b0), kend = b0 + nbt;
  const double2* C = Cg + (long long)blockIdx.x * nb * nb;
  for (int i = threadIdx.x; i < kend * SCF_RB; i += blockDim.x) {
    const int k = i / SCF_RB, j = i % SCF_RB;
    cs[i] = j < nbt ? C[(long long)k * nb + b0 + j] : make_double2(0.0, 0.0);
  }
  __syncthreads();
  const int p = blockIdx.z * blockDim.x + threadIdx.x;
  if (p >= c.npts) return;
  const double2* yb = Y + U.psi_off + p;
  double2 s[SCF_RB];
#pragma unroll
  for (int j = 0; j < SCF_RB; ++j) s[j] = make_double2(0.0, 0.0);
  // C is upper triangular with exact zeros below the diagonal, so the sum
  // over all k < kend adds only zeros beyond k = b
  for (int k = 0; k < kend; ++k) {
    const double2 y = yb[(long long)k * c.npts];
#pragma unroll
    for (int j = 0; j < SCF_RB; ++j) s[j] = zadd(s[j], zmul(y, cs[k * SCF_RB + j]));
  }
  double2* ob = Yout + U.psi_off + p;
#pragma unroll
  for (int j = 0; j < SCF_RB; ++j)
    if (j < nbt) ob[(long long)(b0 + j) * c.npts] = s[j];
}

}  // namespace

int scf_max_bands() { return SCF_MAXB; }

// Lower-triangle tiles of a unit, and the point chunks that fill the GPU (about two CTAs per SM).
static int gram_tiles(const CellDev& c) {
  const int nt = (c.n_bands + SCF_T - 1) / SCF_T;
  return nt * (nt + 1) / 2;
}
static int gram_chunk(const CellDev& c, int n_units) {
  const long long have = (long long)n_units * gram_tiles(c);
  long long chunks = have >= 304 ? 1 : (304 + have - 1) / have;
  const long long most = (c.npts + 2 * SCF_CH - 1) / (2 * SCF_CH);
  if (chunks > most) chunks = most;
  const int chunk = (int)((c.npts + chunks - 1) / chunks);
  return (chunk + SCF_CH - 1) / SCF_CH * SCF_CH;
}

size_t scf_gram_scratch(const CellDev& c, int n_units) {
  if (n_units == 0) return 0;
  const int chunk = gram_chunk(c, n_units);
  return sizeof(double2) * 2 * 256 * (size_t)gram_tiles(c) * n_units * ((c.npts + chunk - 1) / chunk);
}

void launch_scf_gram(const LaunchSet& L, const void* Y, const void* HY, void* S, void* H, void* G, void* stream) {
  if (L.n_units == 0) return;
  const int tiles = gram_tiles(L.cell), chunk = gram_chunk(L.cell, L.n_units);
  const int chunks = (L.cell.npts + chunk - 1) / chunk, nb = L.cell.n_bands;
  const dim3 grid(L.n_units, tiles, chunks), gs(L.n_units, tiles);
  cudaStream_t st = (cudaStream_t)stream;
  if (HY) {
    k_scf_gram<true><<<grid, 256, 0, st>>>(L, (const double2*)Y, (const double2*)HY, (double2*)G, tiles, chunk);
    k_scf_gram_sum<true><<<gs, 256, 0, st>>>(nb, L.cell.dv, (const double2*)G, (double2*)S, (double2*)H, tiles,
                                             chunks);
  } else {
    k_scf_gram<false><<<grid, 256, 0, st>>>(L, (const double2*)Y, nullptr, (double2*)G, tiles, chunk);
    k_scf_gram_sum<false><<<gs, 256, 0, st>>>(nb, L.cell.dv, (const double2*)G, (double2*)S, nullptr, tiles, chunks);
  }
}

void launch_scf_ortho(int n_units, int nb, double shift_coef, int want_lam, const void* S, void* H, void* C,
                      void* W1, void* W2, double* lam, int* bad, void* stream) {
  if (n_units == 0) return;
  k_scf_ortho<<<n_units, SCF_OT, 0, (cudaStream_t)stream>>>(nb, shift_coef, want_lam, (const double2*)S,
                                                            (double2*)H, (double2*)C, (double2*)W1, (double2*)W2,
                                                            lam, bad);
}

void launch_scf_rotate(const LaunchSet& L, const void* Y, const void* C, void* Yout, void* stream) {
  if (L.n_units == 0) return;
  const int nb = L.cell.n_bands;
  const size_t smem = sizeof(double2) * (size_t)nb * SCF_RB;
  smem_limit<k_scf_rotate>(smem);
  dim3 grid(L.n_units, (nb + SCF_RB - 1) / SCF_RB, (L.cell.npts + 127) / 128);
  k_scf_rotate<<<grid, 128, smem, (cudaStream_t)stream>>>(L, (const double2*)Y, (const double2*)C, (double2*)Yout);
}
