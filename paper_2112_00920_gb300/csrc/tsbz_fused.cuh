// Taylor stage on 16^3 grids with the factorised projector contractions on
// tensor cores (three-product TF32 mma.sync, FP32 accumulate).
//
// Per (unit, band) CTA, with C_{a,t}(r) = pn F^a_x F^a_y F^a_z w_t as in the
// header of the z-march kernels:
//   ket   conj(V_NL t)(col, z) = sum_q A[col][q] Z_q(z): the z dependence is a
//         GEMM over q = (atom, {F_z, d_z F_z}) with the column coefficients
//         A[col][(a,0)] = F_y (G00 + d_y G10), A[col][(a,1)] = F_y G01,
//         G00 = F_x (conj W_s + d_x conj W_px), G10 = F_x conj W_py,
//         G01 = F_x conj W_pz, W = pn E P (x tables first, then y).
//   bra   monomial sums M_a(i,j,k) = sum_r F_x F_y F_z d_x^i d_y^j d_z^k u(r)
//         in three contractions: z as a GEMM S[col][(a,k)] = sum_z u Z_{a,k},
//         then x per (a, k, iy) row, then y per (a, i, j, k) output.
//         P_{a,t} = dV pn M_a(w_t) with w_t = 000, 100, 010, 001 (s, p_x, p_y,
//         p_z); the current needs the second-order sums as well.
// Three-product TF32: x = x_hi + x_lo with x_hi = tf32(x), x_lo = tf32(x -
// x_hi) (round to nearest); A B ~ A_lo B_hi + A_hi B_lo + A_hi B_hi, an
// error of order 2^-21 relative per product, accumulated in FP32.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "tsbz_fft.cuh"
#include "tsbz_line.cuh"
#include "tsbz_sep.cuh"

#define FS_N 16
#define FS_NP 256          // columns (threads)
#define FS_NPTS 4096
#define FS_PU 260          // plane pitch of ubuf in float2 (bank-conflict-free fragment stores)
#define FS_BKP 36          // row pitch of the ket B matrix in uint2

__device__ __forceinline__ uint32_t fs_tf32(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;\n" : "=r"(r) : "f"(x));
  return r;
}

__device__ __forceinline__ void fs_split(float x, uint32_t& hi, uint32_t& lo) {
  hi = fs_tf32(x);
  lo = fs_tf32(x - __uint_as_float(hi));
}

__device__ __forceinline__ uint2 fs_split2(float x) {
  uint2 r;
  fs_split(x, r.x, r.y);
  return r;
}

__device__ __forceinline__ void fs_mma(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// d += A B, A = ah + al, B = (b.x hi, b.y lo) for the two B registers
__device__ __forceinline__ void fs_mma3(float (&d)[4], const uint32_t (&ah)[4], const uint32_t (&al)[4], uint2 b0,
                                        uint2 b1) {
  fs_mma(d, al, b0.x, b1.x);
  fs_mma(d, ah, b0.y, b1.y);
  fs_mma(d, ah, b0.x, b1.x);
}

struct FsSmem {
  // two plane buffers of pitch FS_PU: the band of t_{m-1}, and V_NL per plane
  // (ket) overwritten by t_m; the projection passes use them as scratch
  float2 xb[FS_N * FS_PU];
  float2 yb[FS_N * FS_PU];
  uint2 bk[32 * FS_BKP];             // ket B matrix (hi, lo)
  float4 zt[SEP_NA * FS_N];          // (Re F_z, Im F_z, d_z, 0) per atom and plane
  float4 colt[SEP_NA * 2 * FS_N];    // x and y factors (Re F, Im F, d, 0)
  float4 xpk[SEP_NA * FS_N * 3];     // x factors times d^w, w = 0..2, as (Re, Re, Im, Im) pairs
  float2 gt[SEP_NA * 3 * FS_N];      // ket column tables G00, G10, G01 per atom and ix
  float2 wt[SEP_NP];                 // pn E P of the band
  float2 mres[SEP_NA * 10];          // monomial sums of one projection pass
  float vbuf[FS_NPTS];               // v_eff of the sub-simulation (stage kernel)
  int zg[SEP_NA];                    // z group of atom a
  int zrep[4];                       // first atom of group g
  int zmem[4][2];                    // the (at most two) atoms of group g
  int zcnt[4];
  unsigned long long mbar;
};

// z group tables of the cell into shared memory (grouped kernels; read after
// the next barrier)
template <int NZU> __device__ __forceinline__ void fz_load(FsSmem& sm, const CellDev& c) {
  if constexpr (NZU != SEP_NA) {
    const int t = threadIdx.x;
    if (t < SEP_NA) sm.zg[t] = c.zg_of[t];
    if (t < 4) {
      const int lo = c.zg_off[t], n = c.zg_off[t + 1] - lo;
      sm.zrep[t] = c.zg_rep[t];
      sm.zcnt[t] = n;
      sm.zmem[t][0] = n > 0 ? c.zg_mem[lo] : 0;
      sm.zmem[t][1] = n > 1 ? c.zg_mem[lo + 1] : 0;
    }
  }
}

// z factors of one phase table
__device__ __forceinline__ void fs_load_z(float4* zt, const CellDev& c, const float2* ph) {
  const int nm = c.nmax;
  for (int i = threadIdx.x; i < SEP_NA * FS_N; i += blockDim.x) {
    const int a = i / FS_N, z = i - a * FS_N;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (a < c.n_atoms) {
      const int idx = (a * 3 + 2) * nm + z;
      const float g = c.g1f[idx];
      const float2 p = ph[idx];
      v = make_float4(g * p.x, g * p.y, c.d1f[idx], 0.f);
    }
    zt[i] = v;
  }
}

// Factor tables of one phase table: colt (x and y rows, as the column loader
// of the other kernels) and, for the x contraction of the projection passes,
// d_x^w F_x for w = 0..2 in the (Re, Re, Im, Im) form of the packed products.
__device__ __forceinline__ void fs_load_cols(FsSmem& sm, const CellDev& c, const float2* ph) {
  const int nm = c.nmax;
  for (int i = threadIdx.x; i < SEP_NA * 2 * FS_N; i += blockDim.x) {
    const int a = i / (2 * FS_N), r = i - a * 2 * FS_N, ax = r / FS_N, ii = r - ax * FS_N;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (a < c.n_atoms && ii < (ax == 0 ? c.n1 : c.n2)) {
      const int idx = (a * 3 + ax) * nm + ii;
      const float g = c.g1f[idx];
      const float2 p = ph[idx];
      v = make_float4(g * p.x, g * p.y, c.d1f[idx], 0.f);
    }
    sm.colt[i] = v;
    if (ax == 0) {
      float fr = v.x, fi = v.y;
#pragma unroll
      for (int w = 0; w < 3; ++w) {
        sm.xpk[(a * FS_N + ii) * 3 + w] = make_float4(fr, fr, fi, fi);
        fr = __fmul_rn(v.z, fr);
        fi = __fmul_rn(v.z, fi);
      }
    }
  }
}

// complex product with explicit round-to-nearest operations (never contracted)
__device__ __forceinline__ float2 fs_cmul_rn(float2 a, float2 b) {
  return make_float2(__fsub_rn(__fmul_rn(a.x, b.x), __fmul_rn(a.y, b.y)),
                     __fadd_rn(__fmul_rn(a.x, b.y), __fmul_rn(a.y, b.x)));
}

// monomial index of d_x^i d_y^j d_z^k (i + j + k <= 2) in the order
// 000, 100, 010, 001, 200, 110, 101, 020, 011, 002
__device__ __forceinline__ int fs_mono(int i, int j, int k) {
  const int deg = i + j + k;
  if (deg == 0) return 0;
  if (deg == 1) return i ? 1 : (j ? 2 : 3);
  if (i == 2) return 4;
  if (i == 1) return j ? 5 : 6;
  if (j == 2) return 7;
  return j ? 8 : 9;
}

// z groups (atoms with identical z factor tables, see CellDev): with NZU =
// SEP_NA every atom is its own group; with NZU < SEP_NA the cell's groups
// (at most NZU of them) are used and every z contraction runs per group.
template <int NZU> __device__ __forceinline__ int fz_grp(const FsSmem& sm, int a) {
  if constexpr (NZU == SEP_NA) return a; else return sm.zg[a];
}
template <int NZU> __device__ __forceinline__ float4 fz_table(const FsSmem& sm, const CellDev& c, int g, int z) {
  if constexpr (NZU == SEP_NA) {
    return sm.zt[g * FS_N + z];
  } else {
    return g < c.n_zg ? sm.zt[sm.zrep[g] * FS_N + z] : make_float4(0.f, 0.f, 0.f, 0.f);
  }
}

// ----------------------------------------------------------------------------
// ket: ubuf[z][col] = conj(V_NL t)(col, z) for the warp's 32 columns.  The z
// dependence is a GEMM over q = (z group, {F_z, d_z F_z}): column coefficient
// A[col][q] = sum over the group's atoms of F_y (G00 + d_y G10) or F_y G01.
// ----------------------------------------------------------------------------
template <int NZU>
__device__ __forceinline__ void fs_ket(FsSmem& sm, const CellDev& c, float2* vout, bool build_b) {
  constexpr int Q = 2 * NZU;   // complex columns of the GEMM
  constexpr int KS = Q / 4;    // k steps of 8 over the 2 Q real rows (Re rows, then Im rows)
  constexpr int NI = Q / 4;    // q values per thread: t4 + 4 i
  const int tid = threadIdx.x;
  // column tables G00, G10, G01 (conj W) and the B matrix B[k][n], k < 16: Re rows,
  // k >= 16: Im rows of q = (a, w); n = 2 z + c
  for (int i = tid; i < SEP_NA * FS_N; i += blockDim.x) {
    const int a = i / FS_N, ix = i - a * FS_N;
    const float4 fx = sm.colt[(2 * a) * FS_N + ix];
    const float2 F = make_float2(fx.x, fx.y);
    const float2 ws = sm.wt[4 * a], wx = sm.wt[4 * a + 1], wy = sm.wt[4 * a + 2], wz = sm.wt[4 * a + 3];
    const float2 q0 = make_float2(ws.x + fx.z * wx.x, -(ws.y + fx.z * wx.y));
    sm.gt[(a * 3 + 0) * FS_N + ix] = sep_cmul(F, q0);
    sm.gt[(a * 3 + 1) * FS_N + ix] = sep_cmul(F, make_float2(wy.x, -wy.y));
    sm.gt[(a * 3 + 2) * FS_N + ix] = sep_cmul(F, make_float2(wz.x, -wz.y));
  }
  for (int i = tid; build_b && i < 2 * Q * 2 * FS_N; i += blockDim.x) {
    const int k = i / (2 * FS_N), n = i - k * 2 * FS_N;
    const bool rrow = k < Q;
    const int q = rrow ? k : k - Q, z = n >> 1, cc = n & 1;
    const float4 f = fz_table<NZU>(sm, c, q >> 1, z);
    const float s = (q & 1) ? f.z : 1.f;
    const float zr = s * f.x, zi = s * f.y;
    const float v = rrow ? (cc ? zi : zr) : (cc ? zr : -zi);
    sm.bk[k * FS_BKP + n] = fs_split2(v);
  }
  __syncthreads();
  const int lane = tid & 31, warp = tid >> 5, g = lane >> 2, t4 = lane & 3;
  // A fragments of both m-tiles: rows = columns 32 warp + 16 mt + g (+8), k = 8 ks + t4 (+4)
  uint32_t ah[2][KS][4], al[2][KS][4];
#pragma unroll
  for (int mt = 0; mt < 2; ++mt) {
    const int iyc = 2 * warp + mt;
    float re[2][NI], im[2][NI];   // [column A/B][q index i: q = t4 + 4 i]
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      const int q = t4 + 4 * i, gq = q >> 1;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int ixc = g + 8 * h;
        float2 v = make_float2(0.f, 0.f);
        auto add_atom = [&](int a) {
          const float4 fy = sm.colt[(2 * a + 1) * FS_N + iyc];
          const float2 F = make_float2(fy.x, fy.y);
          float2 w;
          if (q & 1) {
            w = sep_cmul(F, sm.gt[(a * 3 + 2) * FS_N + ixc]);
          } else {
            const float2 g0 = sm.gt[(a * 3 + 0) * FS_N + ixc], g1 = sm.gt[(a * 3 + 1) * FS_N + ixc];
            w = sep_cmul(F, make_float2(g0.x + fy.z * g1.x, g0.y + fy.z * g1.y));
          }
          v.x += w.x;
          v.y += w.y;
        };
        if constexpr (NZU == SEP_NA) {
          add_atom(gq);
        } else {
          const int cnt = sm.zcnt[gq];
#pragma unroll
          for (int j = 0; j < 2; ++j)
            if (j < cnt) add_atom(sm.zmem[gq][j]);
        }
        re[h][i] = v.x;
        im[h][i] = v.y;
      }
    }
    // the first KS/2 k steps: Re of q = t4 + 8 ks (+4); the others: Im
#pragma unroll
    for (int ks = 0; ks < KS; ++ks) {
      const bool rpart = ks < KS / 2;
      const int i0 = 2 * (rpart ? ks : ks - KS / 2);
      const float(&src)[2][NI] = rpart ? re : im;
      fs_split(src[0][i0], ah[mt][ks][0], al[mt][ks][0]);
      fs_split(src[1][i0], ah[mt][ks][1], al[mt][ks][1]);
      fs_split(src[0][i0 + 1], ah[mt][ks][2], al[mt][ks][2]);
      fs_split(src[1][i0 + 1], ah[mt][ks][3], al[mt][ks][3]);
    }
  }
#pragma unroll
  for (int nt = 0; nt < (2 * FS_N) / 8; ++nt) {
    float d[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
    for (int ks = 0; ks < KS; ++ks) {
      const uint2 b0 = sm.bk[(8 * ks + t4) * FS_BKP + 8 * nt + g];
      const uint2 b1 = sm.bk[(8 * ks + t4 + 4) * FS_BKP + 8 * nt + g];
      fs_mma3(d[0], ah[0][ks], al[0][ks], b0, b1);
      fs_mma3(d[1], ah[1][ks], al[1][ks], b0, b1);
    }
    const int z = 4 * nt + t4;
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) {
      const int cA = 32 * warp + 16 * mt + g;
      vout[z * FS_PU + cA] = make_float2(d[mt][0], d[mt][1]);
      vout[z * FS_PU + cA + 8] = make_float2(d[mt][2], d[mt][3]);
    }
  }
}

// x and y contractions of a projection pass, from the z sums
// sbuf[q'][iy][ix ^ iy] of the pass's z weights q' = q0 .. q0 + NQ - 1 (read
// after a barrier): leaves mres[(a - a0) * NM + mono] and ends with a barrier.
template <int D, int NQ, int NAP, int NZU>
__device__ __forceinline__ void fs_xy_contract(FsSmem& sm, const CellDev& c, int q0, int a0, const float2* sbuf) {
  constexpr int NM = D == 1 ? 4 : 10;
  const int tid = threadIdx.x;
  // x contraction per row (q', iy): R_i = sum_ix F_x d_x^i S, i <= D - k; then the
  // y contraction M_a(i, j, k) = sum_iy F_y d_y^j R_i over the 16 lanes of the
  // half-warp that holds the rows iy = 0..15 of one q' (fixed-order shuffles).
  constexpr int NR = (D + 1) * NAP * FS_N;
  for (int r0 = 0; r0 < NR; r0 += FS_NP) {
    const int r = r0 + tid;
    const bool live = r < NR;
    const int ql = live ? (r >> 4) : 0, iyr = r & 15;
    const int al_ = ql / (D + 1), kz = ql - al_ * (D + 1), a = a0 + al_;
    const int sq = (D + 1) * fz_grp<NZU>(sm, a) + kz - q0;   // z sums of the atom's group
    // packed FP32x2 products: for w = 0..D - k, A_w accumulates d^w Re F_x (s_re, s_im)
    // and B_w d^w Im F_x (s_re, s_im); R_w = sum d^w F_x s = (A_w.x - B_w.y, A_w.y + B_w.x).
    // Every row runs every w of the pass (no divergence); the D = 1 and D = 2 passes
    // share the operations of w = 0, 1, so their common sums agree bit for bit.
    const float2 zero2 = make_float2(0.f, 0.f);
    float2 A0 = zero2, B0 = zero2, A1 = zero2, B1 = zero2, A2 = zero2, B2 = zero2;
    if (live) {
      const float4* xw = sm.xpk + a * FS_N * 3;
      const float2* sr = sbuf + sq * FS_NP + iyr * FS_N;
#pragma unroll 4
      for (int ixr = 0; ixr < FS_N; ++ixr) {
        const float2 sv = sr[ixr ^ iyr];
        const float4 p0 = xw[ixr * 3 + 0], p1 = xw[ixr * 3 + 1];
        A0 = __ffma2_rn(make_float2(p0.x, p0.y), sv, A0);
        B0 = __ffma2_rn(make_float2(p0.z, p0.w), sv, B0);
        A1 = __ffma2_rn(make_float2(p1.x, p1.y), sv, A1);
        B1 = __ffma2_rn(make_float2(p1.z, p1.w), sv, B1);
        if (D == 2) {
          const float4 p2 = xw[ixr * 3 + 2];
          A2 = __ffma2_rn(make_float2(p2.x, p2.y), sv, A2);
          B2 = __ffma2_rn(make_float2(p2.z, p2.w), sv, B2);
        }
      }
    }
    const float2 R0 = make_float2(__fsub_rn(A0.x, B0.y), __fadd_rn(A0.y, B0.x));
    const float2 R1 = make_float2(__fsub_rn(A1.x, B1.y), __fadd_rn(A1.y, B1.x));
    const float2 R2 = make_float2(__fsub_rn(A2.x, B2.y), __fadd_rn(A2.y, B2.x));
    // y weights of this row: F_y d_y^j
    const float4 fy = sm.colt[(2 * a + 1) * FS_N + iyr];
    const float2 Fy = make_float2(fy.x, fy.y), Fyd = make_float2(__fmul_rn(fy.z, fy.x), __fmul_rn(fy.z, fy.y));
    // contributions, in the order of the monomials this row feeds:
    //   D = 1, k = 0: 000 (F R0), 100 (F R1), 010 (F d R0);  k = 1: 001 (F R0)
    //   D = 2, k = 0: 000, 100, 010, 200 (F R2), 110 (F d R1), 020 (F d^2 R0)
    //          k = 1: 001, 101 (F R1), 011 (F d R0);  k = 2: 002
    constexpr int NC = D == 1 ? 3 : 6;
    float2 v[NC];
    v[0] = fs_cmul_rn(Fy, R0);
    v[1] = fs_cmul_rn(Fy, R1);
    v[2] = fs_cmul_rn(Fyd, R0);
    if (D == 2) {
      v[3 % NC] = fs_cmul_rn(Fy, R2);
      v[4 % NC] = fs_cmul_rn(Fyd, R1);
      v[5 % NC] = fs_cmul_rn(make_float2(__fmul_rn(fy.z, Fyd.x), __fmul_rn(fy.z, Fyd.y)), R0);
    }
#pragma unroll
    for (int off = 1; off < 16; off <<= 1)
#pragma unroll
      for (int e = 0; e < NC; ++e) {
        v[e].x = __fadd_rn(v[e].x, __shfl_xor_sync(0xffffffffu, v[e].x, off));
        v[e].y = __fadd_rn(v[e].y, __shfl_xor_sync(0xffffffffu, v[e].y, off));
      }
    if (live && iyr == 0) {
      float2* M = sm.mres + al_ * NM;
      if (D == 1) {
        if (kz == 0) {
          M[0] = v[0];
          M[1] = v[1];
          M[2] = v[2];
        } else {
          M[3] = v[0];
        }
      } else {
        if (kz == 0) {
          M[0] = v[0];
          M[1] = v[1];
          M[2] = v[2];
          M[4] = v[3 % NC];
          M[5] = v[4 % NC];
          M[7] = v[5 % NC];
        } else if (kz == 1) {
          M[3] = v[0];
          M[6] = v[1];
          M[8] = v[2];
        } else {
          M[9] = v[0];
        }
      }
    }
  }
  __syncthreads();
}



// ----------------------------------------------------------------------------
// Projection pass: monomial sums up to degree D of the atoms a0 .. a0 + NAP - 1,
// from the split A fragments of u (ah/al) and the tables zt / colt of the
// pass.  The z contraction covers the z weights q' = q0 .. q0 + NQ - 1 with
// q' = (D + 1) g + k (g the z group, k the power of d_z); the x and y
// contractions run per atom on the z sums of its group.  Leaves
// mres[(a - a0) * NM + mono] (NM = 4 for D = 1, 10 for D = 2).
// ----------------------------------------------------------------------------
template <int D, int NQ, int NAP, int NZU>
__device__ __forceinline__ void fs_project_pass(FsSmem& sm, const CellDev& c, int q0, int a0,
                                                const uint32_t (&ah)[2][4][4], const uint32_t (&al)[2][4][4],
                                                uint2* bz, float2* sbuf) {
  // bz: B_z (32 x (2 NQ + 4) uint2); sbuf: the z sums [q'][iy][ix ^ iy] (NQ x 256 float2)
  constexpr int NPR = 2 * NQ;          // real n of the pass
  constexpr int BZP = NPR + 4;         // B_z row pitch (uint2)
  constexpr int NM = D == 1 ? 4 : 10;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t4 = lane & 3;
  // B_z[k][n], k = 2 z + c (component of u), n = 2 q' + c' (component of S)
  for (int i = tid; i < 32 * NPR; i += blockDim.x) {
    const int k = i / NPR, n = i - k * NPR;
    const int z = k >> 1, cu = k & 1, qq = q0 + (n >> 1), cs = n & 1;
    const int gz = qq / (D + 1), kz = qq - gz * (D + 1);
    const float4 f = fz_table<NZU>(sm, c, gz, z);
    const float s = kz == 0 ? 1.f : (kz == 1 ? f.z : f.z * f.z);
    const float zr = s * f.x, zi = s * f.y;
    const float v = cs == 0 ? (cu == 0 ? zr : -zi) : (cu == 0 ? zi : zr);
    bz[k * BZP + n] = fs_split2(v);
  }
  __syncthreads();
  // z contraction on tensor cores: S[col][q'] for the warp's columns
#pragma unroll
  for (int nt = 0; nt < NPR / 8; ++nt) {
    float d[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
      const uint2 b0 = bz[(8 * ks + t4) * BZP + 8 * nt + g];
      const uint2 b1 = bz[(8 * ks + t4 + 4) * BZP + 8 * nt + g];
      fs_mma3(d[0], ah[0][ks], al[0][ks], b0, b1);
      fs_mma3(d[1], ah[1][ks], al[1][ks], b0, b1);
    }
    const int ql = 4 * nt + t4;
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) {
      const int iyc = 2 * warp + mt;
      sbuf[ql * FS_NP + iyc * FS_N + (g ^ iyc)] = make_float2(d[mt][0], d[mt][1]);
      sbuf[ql * FS_NP + iyc * FS_N + ((g + 8) ^ iyc)] = make_float2(d[mt][2], d[mt][3]);
    }
  }
  __syncthreads();
  fs_xy_contract<D, NQ, NAP, NZU>(sm, c, q0, a0, sbuf);
}

// A fragments (split) of u = ubuf[z][col] for the warp's columns, k = 2 z + c
__device__ __forceinline__ void fs_load_u(const float2* src, uint32_t (&ah)[2][4][4], uint32_t (&al)[2][4][4]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t4 = lane & 3;
  const float* ub = reinterpret_cast<const float*>(src);
#pragma unroll
  for (int mt = 0; mt < 2; ++mt) {
    const int cA = 32 * warp + 16 * mt + g;
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
      const int k0 = 8 * ks + t4, k1 = k0 + 4;
      const int z0 = k0 >> 1, c0 = k0 & 1, z1 = k1 >> 1, c1 = k1 & 1;
      fs_split(ub[2 * (z0 * FS_PU + cA) + c0], ah[mt][ks][0], al[mt][ks][0]);
      fs_split(ub[2 * (z0 * FS_PU + cA + 8) + c0], ah[mt][ks][1], al[mt][ks][1]);
      fs_split(ub[2 * (z1 * FS_PU + cA) + c1], ah[mt][ks][2], al[mt][ks][2]);
      fs_split(ub[2 * (z1 * FS_PU + cA + 8) + c1], ah[mt][ks][3], al[mt][ks][3]);
    }
  }
}

// ----------------------------------------------------------------------------
// Pieces shared by the per-stage and the whole-step kernels.
// ----------------------------------------------------------------------------
// One band (16 planes of 256 complex values) into a buffer of plane pitch FS_PU.
__device__ __forceinline__ void fs_copy_band(float2* dst, const float2* src, uint32_t bar) {
#pragma unroll 1
  for (int z = 0; z < FS_N; ++z)
    bk_copy_g2s(bk_smem(dst + z * FS_PU), src + z * FS_NP, FS_NP * (uint32_t)sizeof(float2), bar);
}

// Factor tables of the unit (q of the step) and W = E P of the band.
__device__ __forceinline__ void fs_unit_tables(FsSmem& sm, const CellDev& c, const float2* ph, const float2* Pu) {
  fs_load_z(sm.zt, c, ph);
  fs_load_cols(sm, c, ph);
  for (int j = threadIdx.x; j < SEP_NP; j += blockDim.x) {
    float2 w = make_float2(0.f, 0.f);
    if (j < c.n_proj) {
      const float2 p = Pu[j];
      const float e = c.wkbf[j];
      w = make_float2(e * p.x, e * p.y);
    }
    sm.wt[j] = w;
  }
}

// z-march of Taylor stage m over the band held in `tin`: t_m = (-i dt/m) h t_{m-1}
// with h t = -1/2 lap t - i q.grad t + (|q|^2/2 + v_eff) t + V_NL t.  `vio`
// holds conj(V_NL t_{m-1}) per plane on entry and receives, column by column,
// t_m (m < 4) or psi(t_{n+1}) (m = 4).
//   STEP = false (one launch per stage): psi in global memory, `acc` holds the
//     psi column (m >= 2), t_m goes to tout (m < 4);
//   STEP = true (the whole step in one launch): psi accumulates in `acc`
//     (acc = t_0 + t_1 at m = 1) and is written once, at m = 4.
template <bool STEP>
__device__ __forceinline__ void fs_march(const FsSmem& sm, const CellDev& c, const float2* tin, float2* vio, int m,
                                         float hdt, float q0, float q1, float q2, float dg0, float2 (&acc)[FS_N],
                                         float2* __restrict__ tout, float2* __restrict__ psi, long long base) {
  constexpr int ND = ZM_ND, N = FS_N, NP = FS_NP;
  const int col = threadIdx.x, ix = col & (N - 1), iy = col / N;
  const float2 zero = make_float2(0.f, 0.f);
  const float2* cz = tin + col;
  const float2* xp[ND];
  const float2* xm[ND];
  const float2* yp[ND];
  const float2* ym[ND];
#pragma unroll
  for (int mm = 1; mm <= ND; ++mm) {
    xp[mm - 1] = tin + iy * N + ((ix + mm) & (N - 1));
    xm[mm - 1] = tin + iy * N + ((ix - mm) & (N - 1));
    yp[mm - 1] = tin + ((iy + mm) & (N - 1)) * N + ix;
    ym[mm - 1] = tin + ((iy - mm) & (N - 1)) * N + ix;
  }
  const float2 neg1 = make_float2(-1.f, -1.f);
  float2 qv[N + 2 * ND];
#pragma unroll
  for (int k = 0; k < 2 * ND; ++k) qv[k] = cz[((k - ND + N) & (N - 1)) * FS_PU];
#pragma unroll
  for (int z = 0; z < N; ++z) {
    qv[z + 2 * ND] = cz[((z + ND) & (N - 1)) * FS_PU];
    const float2 ce = qv[z + ND];
    const float dg = dg0 + sm.vbuf[z * NP + col];
    float2 h = __fmul2_rn(make_float2(dg, dg), ce);
    float2 gx = zero, gy = zero, gz = zero;
#pragma unroll
    for (int mm = 1; mm <= ND; ++mm) {
      const float2 xu = xp[mm - 1][z * FS_PU], xd = xm[mm - 1][z * FS_PU];
      const float2 yu = yp[mm - 1][z * FS_PU], yd = ym[mm - 1][z * FS_PU];
      const float2 zu = qv[z + ND + mm], zd = qv[z + ND - mm];
      h = f2fma(c.hlap2[0][mm], __fadd2_rn(xu, xd), h);
      h = f2fma(c.hlap2[1][mm], __fadd2_rn(yu, yd), h);
      h = f2fma(c.hlap2[2][mm], __fadd2_rn(zu, zd), h);
      gx = f2fma(c.gradw2[0][mm], f2fma(neg1, xd, xu), gx);
      gy = f2fma(c.gradw2[1][mm], f2fma(neg1, yd, yu), gy);
      gz = f2fma(c.gradw2[2][mm], f2fma(neg1, zd, zu), gz);
    }
    float2 qg = __fmul2_rn(make_float2(q0, q0), gx);
    qg = f2fma(make_float2(q1, q1), gy, qg);
    qg = f2fma(make_float2(q2, q2), gz, qg);
    const float2 vq = vio[z * FS_PU + col];   // conj(V_NL t)
    const float hr = h.x + qg.y + vq.x;
    const float hi = h.y - qg.x - vq.y;
    const float2 t = make_float2(hdt * hi, -hdt * hr);
    const long long idx = base + (long long)z * NP + col;
    float2 uo = t;
    if constexpr (STEP) {
      if (m == 1) {
        acc[z] = __fadd2_rn(ce, t);
      } else if (m < 4) {
        acc[z] = __fadd2_rn(acc[z], t);
      } else {
        uo = __fadd2_rn(acc[z], t);   // psi(t_{n+1})
        psi[idx] = uo;
      }
    } else {
      if (m < 4) tout[idx] = t;
      if (m == 2) {
        psi[idx] = __fadd2_rn(acc[z], __fadd2_rn(ce, t));
      } else if (m == 3) {
        psi[idx] = __fadd2_rn(acc[z], t);
      } else if (m == 4) {
        uo = __fadd2_rn(acc[z], t);   // psi(t_{n+1})
        psi[idx] = uo;
      }
    }
    vio[z * FS_PU + col] = uo;
  }
}

// P_j = dV pn_j M_j of a degree-1 pass (float, as stored in P).
__device__ __forceinline__ float2 fs_proj_value(const FsSmem& sm, const CellDev& c, int j) {
  const float2 M = sm.mres[(j >> 2) * 4 + (j & 3)];
  const double sc = c.dv * (double)c.pnormf[j];
  return make_float2((float)(sc * M.x), (float)(sc * M.y));
}

// Stage 4 after the march: projections of psi(t_{n+1}) (split fragments ah/al)
// for the next step (P, q of the next step) and for the current (Pa, q at
// t_{n+1}).  With a constant field both use the same q, and the first-order
// sums of the current's pass are those of the next step's (same z sums, rows
// and order).  bz / sbuf: scratch (B_z, z sums), both buffers free.
template <int NZU>
__device__ __forceinline__ void fs_stage4_projections(FsSmem& sm, const LaunchSet& L, const CellDev& c, int u,
                                                      const UnitDev& U, int b, float2* __restrict__ Pu,
                                                      float2* __restrict__ Pa, int same_next,
                                                      const uint32_t (&ah)[2][4][4], const uint32_t (&al)[2][4][4],
                                                      uint2* bz, float2* sbuf) {
  const int tid = threadIdx.x;
  const float2* phn = (const float2*)L.ph_next + (long long)u * L.ph_stride;
  const float2* pho = (const float2*)L.ph_obs + (long long)u * L.ph_stride;
  if (!same_next) {
    fs_load_z(sm.zt, c, phn);
    fs_load_cols(sm, c, phn);
    __syncthreads();
    fs_project_pass<1, 2 * NZU, SEP_NA, NZU>(sm, c, 0, 0, ah, al, bz, sbuf);
    if (tid < c.n_proj) Pu[tid] = fs_proj_value(sm, c, tid);
  }
  fs_load_z(sm.zt, c, pho);
  fs_load_cols(sm, c, pho);
  __syncthreads();
  float2* Pab = Pa + U.pa_off + 4LL * b * c.n_proj;
  // the second-order sums of every atom in one pass when the z groups halve
  // the z weights (12 of them), else in two passes of 4 atoms
  constexpr int NPASS = NZU == SEP_NA ? 2 : 1, NAP = SEP_NA / NPASS;
#pragma unroll 1
  for (int half = 0; half < NPASS; ++half) {
    fs_project_pass<2, 3 * NZU / NPASS, NAP, NZU>(sm, c, half * (3 * NZU / NPASS), half * NAP, ah, al, bz, sbuf);
    // rows (a, c_x, c_y, c_z) of projector type t: monomials w_t and w_t + e_alpha
    const int o = tid;
    if (o < 4 * 4 * NAP) {
      const int al_ = o >> 4, t = (o >> 2) & 3, s = o & 3;
      const int a = half * NAP + al_;
      const int j = 4 * a + t;
      if (j < c.n_proj) {
        int e[3] = {t == 1 ? 1 : 0, t == 2 ? 1 : 0, t == 3 ? 1 : 0};
        if (s > 0) e[s - 1] += 1;
        const float2 M = sm.mres[al_ * 10 + fs_mono(e[0], e[1], e[2])];
        const double sc = c.dv * (double)c.pnormf[j];
        const float2 v = make_float2((float)(sc * M.x), (float)(sc * M.y));
        Pab[4 * j + s] = v;
        if (same_next && s == 0) Pu[j] = v;
      }
    }
    __syncthreads();
  }
}

// ----------------------------------------------------------------------------
// Taylor stage m on a 16^3 grid, one CTA per (unit, band), one thread per
// (x, y) column; same arithmetic contract as k_stage_bulk: t_m, the psi
// accumulation, the projections of t_m (m < 4) or, at m = 4, those of
// psi(t_{n+1}) for the next step (P) and for the current (Pa).  The z
// contractions run on mma.sync.
// ----------------------------------------------------------------------------
template <int NZU>
__global__ void __launch_bounds__(FS_NP, 2) k_stage_fused(LaunchSet L, const float2* __restrict__ tin,
                                                          float2* __restrict__ tout, float2* __restrict__ psi,
                                                          float2* __restrict__ P, float2* __restrict__ Pa, int m,
                                                          int same_next) {
  constexpr int N = FS_N, NP = FS_NP;
  extern __shared__ __align__(128) unsigned char fs_raw[];
  FsSmem& sm = *reinterpret_cast<FsSmem*>(fs_raw);
  const CellDev& c = L.cell;
  const int b = blockIdx.x % c.n_bands;
  const int u = L.unit_ids[blockIdx.x / c.n_bands];
  if (!unit_active(L, u)) return;
  const UnitDev U = L.units[u];
  const SubDev S = L.subs[U.sub];
  const int tid = threadIdx.x, col = tid;
  const bool proj = c.use_proj != 0;
  const float2* ph = (const float2*)L.ph_half + (long long)u * L.ph_stride;
  float2* Pu = P + U.p_off + (long long)b * c.n_proj;
  const long long base = U.psi_off + (long long)b * FS_NPTS;
  const float2 zero = make_float2(0.f, 0.f);
  const uint32_t bar = bk_smem(&sm.mbar);
  if (tid == 0) bk_mbar_init(bar, 1);
  fz_load<NZU>(sm, c);
  __syncthreads();
  if (tid == 0) {
    // the band of t_{m-1} and the sub-simulation's v_eff, on one barrier
    bk_mbar_expect_tx(bar, FS_NPTS * (uint32_t)(sizeof(float2) + sizeof(float)));
    fs_copy_band(sm.xb, tin + base, bar);
    bk_copy_g2s(bk_smem(sm.vbuf), S.veff, FS_NPTS * sizeof(float), bar);
  }
  // psi of the column in registers (m >= 2), in flight while the ket runs
  float2 pq[N];
#pragma unroll
  for (int z = 0; z < N; ++z) pq[z] = m >= 2 ? psi[base + z * NP + col] : zero;
  if (proj) fs_unit_tables(sm, c, ph, Pu);
  __syncthreads();
  if (proj) {
    fs_ket<NZU>(sm, c, sm.yb, true);
  } else {
#pragma unroll
    for (int z = 0; z < N; ++z) sm.yb[z * FS_PU + col] = zero;
  }
  const float* qt = reinterpret_cast<const float*>(L.qt_half) + 4 * u;
  const float dg0 = c.hlapf[0][0] + c.hlapf[1][0] + c.hlapf[2][0] + qt[3];
  const bool ok = bk_mbar_wait(bar, 0, BK_WAIT_POLLS);
  if (!__syncthreads_and(ok)) {
    if (tid == 0) {
      atomicOr(S.status, BK_STATUS_TIMEOUT);
      bk_mbar_wait(bar, 0, BK_WAIT_POLLS);
    }
    return;
  }
  fs_march<false>(sm, c, sm.xb, sm.yb, m, (float)(S.dt * L.dt_scale) / (float)m, qt[0], qt[1], qt[2], dg0, pq, tout, psi, base);
  if (!proj) return;
  __syncthreads();
  uint32_t ah[2][4][4], al[2][4][4];
  fs_load_u(sm.yb, ah, al);
  __syncthreads();   // both buffers free for the projection scratch
  uint2* bz = reinterpret_cast<uint2*>(sm.xb);
  if (m < 4) {
    fs_project_pass<1, 2 * NZU, SEP_NA, NZU>(sm, c, 0, 0, ah, al, bz, sm.yb);
    if (tid < c.n_proj) Pu[tid] = fs_proj_value(sm, c, tid);
    return;
  }
  fs_stage4_projections<NZU>(sm, L, c, u, U, b, Pu, Pa, same_next, ah, al, bz, sm.yb);
}

// ----------------------------------------------------------------------------
// The whole time step in one launch (cells whose atoms form z groups of at
// most two: NZU = 4) with the star stencil and mma.sync contractions (variant 3;
// variant 0 is k_step_fft), one CTA per (unit, band): the band of psi is brought in
// once, the four Taylor terms live in the two plane buffers (t_{m-1} in one,
// V_NL and then t_m in the other, roles swapping each stage), psi accumulates
// in registers, and each stage's projections go straight to the next stage's
// ket.  Memory traffic per step: psi read and written once, P and Pa.  Same
// arithmetic per stage as k_stage_fused; psi is summed as
// (((t_0 + t_1) + t_2) + t_3) + t_4.
// ----------------------------------------------------------------------------
template <int NZU>
__global__ void __launch_bounds__(FS_NP, 2) k_step_fused(LaunchSet L, float2* __restrict__ psi,
                                                         float2* __restrict__ P, float2* __restrict__ Pa,
                                                         int same_next) {
  static_assert(NZU == 4, "the projection scratch of a stage fits one plane buffer only with z groups");
  constexpr int N = FS_N;
  extern __shared__ __align__(128) unsigned char fs_raw[];
  FsSmem& sm = *reinterpret_cast<FsSmem*>(fs_raw);
  const CellDev& c = L.cell;
  const int b = blockIdx.x % c.n_bands;
  const int u = L.unit_ids[blockIdx.x / c.n_bands];
  if (!unit_active(L, u)) return;
  const UnitDev U = L.units[u];
  const SubDev S = L.subs[U.sub];
  const int tid = threadIdx.x;
  const float2* ph = (const float2*)L.ph_half + (long long)u * L.ph_stride;
  float2* Pu = P + U.p_off + (long long)b * c.n_proj;
  const long long base = U.psi_off + (long long)b * FS_NPTS;
  const uint32_t bar = bk_smem(&sm.mbar);
  if (tid == 0) bk_mbar_init(bar, 1);
  fz_load<NZU>(sm, c);
  __syncthreads();
  if (tid == 0) {
    bk_mbar_expect_tx(bar, FS_NPTS * (uint32_t)(sizeof(float2) + sizeof(float)));
    fs_copy_band(sm.xb, psi + base, bar);
    bk_copy_g2s(bk_smem(sm.vbuf), S.veff, FS_NPTS * sizeof(float), bar);
  }
  fs_unit_tables(sm, c, ph, Pu);
  __syncthreads();
  const float* qt = reinterpret_cast<const float*>(L.qt_half) + 4 * u;
  const float q0 = qt[0], q1 = qt[1], q2 = qt[2];
  const float dg0 = c.hlapf[0][0] + c.hlapf[1][0] + c.hlapf[2][0] + qt[3];
  float2 acc[N];
  uint32_t ah[2][4][4], al[2][4][4];
  float2* tin = sm.xb;
  float2* vio = sm.yb;
  bool waited = false;
#pragma unroll 1
  for (int m = 1; m <= 4; ++m) {
    fs_ket<NZU>(sm, c, vio, m == 1);
    if (!waited) {
      const bool ok = bk_mbar_wait(bar, 0, BK_WAIT_POLLS);
      if (!__syncthreads_and(ok)) {
        if (tid == 0) {
          atomicOr(S.status, BK_STATUS_TIMEOUT);
          bk_mbar_wait(bar, 0, BK_WAIT_POLLS);
        }
        return;
      }
      waited = true;
    } else {
      __syncthreads();
    }
    fs_march<true>(sm, c, tin, vio, m, (float)(S.dt * L.dt_scale) / (float)m, q0, q1, q2, dg0, acc, nullptr, psi, base);
    __syncthreads();
    fs_load_u(vio, ah, al);
    if (m < 4) {
      // projections of t_m for the next stage; scratch in the buffer of t_{m-1}
      fs_project_pass<1, 2 * NZU, SEP_NA, NZU>(sm, c, 0, 0, ah, al, reinterpret_cast<uint2*>(tin + 2 * NZU * FS_NP),
                                               tin);
      if (tid < SEP_NP) {
        float2 w = make_float2(0.f, 0.f);
        if (tid < c.n_proj) {
          const float2 p = fs_proj_value(sm, c, tid);
          const float e = c.wkbf[tid];
          w = make_float2(e * p.x, e * p.y);
        }
        sm.wt[tid] = w;
      }
      __syncthreads();
      float2* t = tin;
      tin = vio;
      vio = t;
    } else {
      __syncthreads();   // both buffers free for the projection scratch
      fs_stage4_projections<NZU>(sm, L, c, u, U, b, Pu, Pa, same_next, ah, al, reinterpret_cast<uint2*>(tin), vio);
    }
  }
}

// ----------------------------------------------------------------------------
// Projections P[u][b][j] of float orbitals on a 16^3 grid (q_half tables),
// one CTA per (unit, band): the same tensor-core pass as the fused stage, so
// the projections of a restored state equal those the stage leaves, bit for bit.
// ----------------------------------------------------------------------------
template <int NZU>
__global__ void __launch_bounds__(FS_NP, 2) k_bra_fused(LaunchSet L, const float2* __restrict__ src,
                                                        float2* __restrict__ P) {
  extern __shared__ __align__(128) unsigned char fs_raw[];
  FsSmem& sm = *reinterpret_cast<FsSmem*>(fs_raw);
  const CellDev& c = L.cell;
  const int b = blockIdx.x % c.n_bands;
  const int u = L.unit_ids[blockIdx.x / c.n_bands];
  if (!unit_active(L, u)) return;
  const UnitDev U = L.units[u];
  const int tid = threadIdx.x;
  const float2* ph = (const float2*)L.ph_half + (long long)u * L.ph_stride;
  const float2* sb = src + U.psi_off + (long long)b * FS_NPTS + tid;
  fz_load<NZU>(sm, c);
#pragma unroll
  for (int z = 0; z < FS_N; ++z) sm.yb[z * FS_PU + tid] = sb[z * FS_NP];
  fs_load_z(sm.zt, c, ph);
  fs_load_cols(sm, c, ph);
  __syncthreads();
  uint32_t ah[2][4][4], al[2][4][4];
  fs_load_u(sm.yb, ah, al);
  __syncthreads();
  fs_project_pass<1, 2 * NZU, SEP_NA, NZU>(sm, c, 0, 0, ah, al, reinterpret_cast<uint2*>(sm.xb), sm.yb);
  if (tid < c.n_proj) P[U.p_off + (long long)b * c.n_proj + tid] = fs_proj_value(sm, c, tid);
}

// ----------------------------------------------------------------------------
// Projections of the current, Pa[u][b][j][alpha] = <beta~_j|u>, <d_alpha beta~_j|u>
// on the q_obs tables, one CTA per (unit, band): the second-order pass of the
// whole-step kernel's stage 4 (monomials of degree <= 2), for the evaluations
// of J outside a step (J(0-), J(0+), a restored state).
// ----------------------------------------------------------------------------
template <int NZU>
__global__ void __launch_bounds__(FS_NP, 2) k_pa_fused(LaunchSet L, const float2* __restrict__ src,
                                                       float2* __restrict__ Pa) {
  extern __shared__ __align__(128) unsigned char fs_raw[];
  FsSmem& sm = *reinterpret_cast<FsSmem*>(fs_raw);
  const CellDev& c = L.cell;
  const int b = blockIdx.x % c.n_bands;
  const int u = L.unit_ids[blockIdx.x / c.n_bands];
  if (!unit_active(L, u)) return;
  const UnitDev U = L.units[u];
  const int tid = threadIdx.x;
  const float2* ph = (const float2*)L.ph_obs + (long long)u * L.ph_stride;
  const float2* sb = src + U.psi_off + (long long)b * FS_NPTS + tid;
  fz_load<NZU>(sm, c);
#pragma unroll
  for (int z = 0; z < FS_N; ++z) sm.yb[z * FS_PU + tid] = sb[z * FS_NP];
  fs_load_z(sm.zt, c, ph);
  fs_load_cols(sm, c, ph);
  __syncthreads();
  uint32_t ah[2][4][4], al[2][4][4];
  fs_load_u(sm.yb, ah, al);
  __syncthreads();   // yb becomes the z-sum scratch
  float2* Pab = Pa + U.pa_off + 4LL * b * c.n_proj;
  constexpr int NPASS = NZU == SEP_NA ? 2 : 1, NAP = SEP_NA / NPASS;
#pragma unroll 1
  for (int half = 0; half < NPASS; ++half) {
    fs_project_pass<2, 3 * NZU / NPASS, NAP, NZU>(sm, c, half * (3 * NZU / NPASS), half * NAP, ah, al,
                                                  reinterpret_cast<uint2*>(sm.xb), sm.yb);
    // rows (a, c_x, c_y, c_z) of projector type t: monomials w_t and w_t + e_alpha
    const int o = tid;
    if (o < 4 * 4 * NAP) {
      const int al_ = o >> 4, t = (o >> 2) & 3, sa = o & 3;
      const int a = half * NAP + al_;
      const int j = 4 * a + t;
      if (j < c.n_proj) {
        int e[3] = {t == 1 ? 1 : 0, t == 2 ? 1 : 0, t == 3 ? 1 : 0};
        if (sa > 0) e[sa - 1] += 1;
        const float2 M = sm.mres[al_ * 10 + fs_mono(e[0], e[1], e[2])];
        const double sc = c.dv * (double)c.pnormf[j];
        Pab[4 * j + sa] = make_float2((float)(sc * M.x), (float)(sc * M.y));
      }
    }
    __syncthreads();
  }
}

// ----------------------------------------------------------------------------
// Observation pass on 16^3 grids: one CTA per (unit, band group), the group's bands in turn through a
// ring of FO_SLOTS band buffers filled by bulk copies.  A slot's "full"
// mbarrier completes when its band has landed, its "empty" mbarrier when all
// warps are done with it; thread 0 refills a slot once it is empty, so warps
// never meet at a CTA barrier between bands.
// Bound by shared memory's bandwidth when every point read its eight forward
// neighbours (9.25 reads a point, 78% of the wavefronts).  The current's sums run
// over whole lines, so a thread takes a line along each axis in turn into registers:
// three reads a point.  65 536 orbitals 590 -> 467 us, 16 384 174 -> 135 us.
// Per column and plane it accumulates occ sum_b |u|^2 (rho; over bands as an
// unevaluated float pair s + e updated by the error-free two-sum, which keeps
// the sum to about 2^-44 relative, i.e. FP64-grade, without FP64 arithmetic),
// per thread sum Re(u* (-i grad u)) (FP32 within a band; over bands again as a
// two-sum float pair, so that GB300's narrow FP64 pipe is left alone) and
// per band sum |u|^2 (per-warp partials, added over warps in order at the
// end).  Point tile 0 of the partial buffers is the only one.  The band groups
// (CellDev::obs_bg) fill the GPU when there are few units: 8 units of 16 bands,
// 37 -> 17 us with two bands a group.
// ----------------------------------------------------------------------------
#define FO_SLOTS 3
#define FO_MAXB 128   // bands of the per-warp norm table

struct FoSmem {
  float2 buf[FO_SLOTS][FS_NPTS];
  float nrm[8][FO_MAXB];
  double redj[8][3];
  unsigned long long full[FO_SLOTS];
  unsigned long long empty[FO_SLOTS];
  int fail;
};

// One arrival of the calling thread on a shared-memory mbarrier.
__device__ __forceinline__ void fo_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}

__global__ void __launch_bounds__(FS_NP, 2) k_observe_fused(LaunchSet L, const float2* __restrict__ psi,
                                                            double* __restrict__ rho_part,
                                                            double* __restrict__ jk_part,
                                                            double* __restrict__ nrm_part) {
  step_enter();
  constexpr int ND = ZM_ND, N = FS_N, NP = FS_NP;
  extern __shared__ __align__(128) unsigned char fo_raw[];
  FoSmem& sm = *reinterpret_cast<FoSmem*>(fo_raw);
  const CellDev& c = L.cell;
  const int u = L.unit_ids[blockIdx.x];
  if (!unit_active(L, u)) return;
  const UnitDev U = L.units[u];
  const SubDev S = L.subs[U.sub];
  const int tid = threadIdx.x, col = tid, lane = tid & 31, warp = tid >> 5;
  const int n_warps = (int)(blockDim.x >> 5);
  const int ix = col & (N - 1), iy = col / N;
  const int grp = blockIdx.y, b0 = grp * c.obs_bg;
  const int nb = min(c.obs_bg, c.n_bands - b0);   // bands of the group
  const float2* src = psi + U.psi_off + (long long)b0 * FS_NPTS;
  volatile int* fail = &sm.fail;
  if (tid == 0) {
    for (int k = 0; k < FO_SLOTS; ++k) {
      bk_mbar_init(bk_smem(&sm.full[k]), 1);
      bk_mbar_init(bk_smem(&sm.empty[k]), (uint32_t)n_warps);
    }
    *fail = 0;
  }
  __syncthreads();
  if (tid == 0)
    for (int k = 0; k < FO_SLOTS && k < nb; ++k) {
      bk_mbar_expect_tx(bk_smem(&sm.full[k]), FS_NPTS * (uint32_t)sizeof(float2));
      bk_copy_g2s(bk_smem(sm.buf[k]), src + (long long)k * FS_NPTS, FS_NPTS * sizeof(float2), bk_smem(&sm.full[k]));
    }
  float2 rho[N / 2], rho_e[N / 2];   // planes (2 i, 2 i + 1)
#pragma unroll
  for (int z = 0; z < N / 2; ++z) rho[z] = rho_e[z] = make_float2(0.f, 0.f);
  float js[3] = {0.f, 0.f, 0.f}, je[3] = {0.f, 0.f, 0.f};   // current over bands: js + je per axis
  int issued = nb < FO_SLOTS ? nb : FO_SLOTS;   // bands whose copy thread 0 has issued
  for (int b = 0; b < nb; ++b) {
    if (*fail) break;
    const int slot = b % FO_SLOTS;
    const uint32_t parity = (uint32_t)((b / FO_SLOTS) & 1);
    if (!bk_mbar_wait(bk_smem(&sm.full[slot]), parity, BK_WAIT_POLLS)) {
      *fail = 1;
      break;
    }
    const float2* tb = sm.buf[slot];
    float2 ln[N];
    // along x: row (y, z) = thread, from a point that differs between lanes (no bank conflicts;
    // the periodic sums do not depend on where a line begins)
#pragma unroll
    for (int x = 0; x < N; ++x) ln[x] = tb[tid * N + ((x + tid) & (N - 1))];
    const float bx = line_current(ln, c.gradwf[0]);
#pragma unroll
    for (int y = 0; y < N; ++y) ln[y] = tb[iy * NP + y * N + ix];   // line (x, z = iy)
    const float by = line_current(ln, c.gradwf[1]);
#pragma unroll
    for (int z = 0; z < N; ++z) ln[z] = tb[z * NP + col];
    const float bz = line_current(ln, c.gradwf[2]);
    float nbs = 0.f;
#pragma unroll
    for (int z = 0; z < N; z += 2) {
      const float2 n2v = make_float2(ln[z].x * ln[z].x + ln[z].y * ln[z].y,
                                     ln[z + 1].x * ln[z + 1].x + ln[z + 1].y * ln[z + 1].y);
      // two-sum: rho + n2v = t + err exactly
      const float2 t = fft_add(rho[z / 2], n2v), bb = fft_sub(t, rho[z / 2]);
      rho_e[z / 2] = fft_add(rho_e[z / 2], fft_add(fft_sub(rho[z / 2], fft_sub(t, bb)), fft_sub(n2v, bb)));
      rho[z / 2] = t;
      nbs += n2v.x;
      nbs += n2v.y;
    }
    {
      const float bv[3] = {bx, by, bz};
#pragma unroll
      for (int ax = 0; ax < 3; ++ax) {
        const float t = js[ax] + bv[ax], bb = t - js[ax];
        je[ax] += (js[ax] - (t - bb)) + (bv[ax] - bb);
        js[ax] = t;
      }
    }
    for (int off = 16; off > 0; off >>= 1) nbs += __shfl_xor_sync(0xffffffffu, nbs, off);
    if (lane == 0) {
      sm.nrm[warp][b] = nbs;
      fo_arrive(bk_smem(&sm.empty[slot]));   // the warp is done with this slot (reads ordered by the shuffles)
    }
    if (tid == 0 && b + FO_SLOTS < nb) {
      // refill the slot with band b + FO_SLOTS once every warp is done with it
      if (!bk_mbar_wait(bk_smem(&sm.empty[slot]), parity, BK_WAIT_POLLS)) {
        *fail = 1;
        break;
      }
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      bk_mbar_expect_tx(bk_smem(&sm.full[slot]), FS_NPTS * (uint32_t)sizeof(float2));
      bk_copy_g2s(bk_smem(sm.buf[slot]), src + (long long)(b + FO_SLOTS) * FS_NPTS, FS_NPTS * sizeof(float2),
                  bk_smem(&sm.full[slot]));
      issued = b + FO_SLOTS + 1;
    }
  }
  if (__syncthreads_or(*fail)) {
    if (tid == 0) {
      atomicOr(S.status, BK_STATUS_TIMEOUT);
      // let every issued copy land before the CTA's shared memory is released
      for (int k = (issued > FO_SLOTS ? issued - FO_SLOTS : 0); k < issued; ++k)
        bk_mbar_wait(bk_smem(&sm.full[k % FO_SLOTS]), (uint32_t)((k / FO_SLOTS) & 1), BK_WAIT_POLLS);
    }
    return;
  }
#pragma unroll
  for (int z = 0; z < N; ++z) {
    const float r = z & 1 ? rho[z / 2].y : rho[z / 2].x, e = z & 1 ? rho_e[z / 2].y : rho_e[z / 2].x;
    rho_part[U.rho_off + (long long)grp * FS_NPTS + z * NP + col] = c.occ * ((double)r + (double)e);
  }
  double jx = (double)js[0] + (double)je[0], jy = (double)js[1] + (double)je[1], jz = (double)js[2] + (double)je[2];
  for (int off = 16; off > 0; off >>= 1) {
    jx += __shfl_xor_sync(0xffffffffu, jx, off);
    jy += __shfl_xor_sync(0xffffffffu, jy, off);
    jz += __shfl_xor_sync(0xffffffffu, jz, off);
  }
  if (lane == 0) {
    sm.redj[warp][0] = jx;
    sm.redj[warp][1] = jy;
    sm.redj[warp][2] = jz;
  }
  __syncthreads();
  if (tid < 3) {
    double sum = 0.0;
    for (int w = 0; w < n_warps; ++w) sum += sm.redj[w][tid];
    jk_part[U.jk_off + 3 * grp + tid] = sum;
  }
  for (int b = tid; b < nb; b += blockDim.x) {
    double sum = 0.0;
    for (int w = 0; w < n_warps; ++w) sum += (double)sm.nrm[w][b];
    nrm_part[U.nrm_off + b0 + b] = sum;
  }
}
