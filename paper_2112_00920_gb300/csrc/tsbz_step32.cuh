// The whole time step of a band in one launch, FP32 on 16^3 grids whose atoms form
// at most 4 z groups of at most two (variant 0): the kinetic operator by its Fourier
// symbol, the projector contractions along z on tcgen05.
//
// What bounds it: instruction issue at 16 warps per SM (128 registers, two CTAs);
// HBM sees psi once.  The star stencil needs 16 in-plane loads a point and
// stage; the periodic grid's discrete Fourier basis diagonalises it (real symbol,
// one number per axis, CellDev::ksym), so six 16-point line transforms in
// registers replace it with 8 shared accesses and about 50 instructions a point.
// One thread per (x, y) column.  The column of t stays in registers from one stage
// to the next; the Taylor sum, v_eff and the tensor-core operands live in tensor
// memory; the one line buffer is turned in place (rows of 17: no bank conflicts,
// and every address a constant offset).  The x and y transforms of a plane belong
// to one half-warp, so only the two exchanges with the columns need the CTA's
// barrier.  The projector work rides along: the z sums of t_m run on the tensor
// cores under the next stage's transforms, one warp per atom forms their x and y
// sums and, from them, the atom's ket tables.
// The ket's MMAs run under the column's inverse transform.
// Taylor terms are kept as s_m = dt h^m psi; the rest of (-i dt)^m / m! enters the sum only,
// psi's increment (see tsbz_any.cu).
// Measured, 65 536 orbitals: 10.50 (four star stencils, k_step_fused with its contractions
// on tcgen05) -> 6.10 ms, 6.18 with the symbol's table and the increment summed apart (their
// reason stands at tsbz_symbol.cuh and tsbz_any.cu); 121 instructions a point and stage, projections
// of the current included, 52% of the issue slots.  Without any transform it takes 4.8 ms, with the
// butterflies in scalar instead of packed arithmetic 6.5 ms.
//
// Contractions (see tsbz_fused.cuh for the factorisation).  Atoms are addressed by
// slot 2 g + j, the j-th atom of z group g (empty slots have zero tables).
//   bra: z sums S[col][q] = sum_z u Z_q as a GEMM (256 x 32)(32 x 2 NQ), q = (D + 1) g + k,
//        Z = d_z^k F_z; then per slot the x sums over a row and the y sums over lanes.
//   ket: conj(V_NL t)(col, z) = sum_q A[col][q] Z_q(z) as a GEMM (256 x 16)(16 x 32),
//        A = F_y (G00 + d_y G10), F_y G01 with G = F_x conj(W), W = pn E P.
// Each thread's row of A goes to tensor memory split into TF32 hi and lo (three
// products, FP32 accumulate); B (hi, lo) sits in shared memory in the canonical
// K-major layout; one thread issues the MMAs (M = 128 per half of the columns).
// Tensor-memory columns of a CTA, 32 per half of the columns: [0, 64) the first-order
// bra accumulator (16) and v_eff (16); [64, 128) the Taylor sum, and after it the
// second-order accumulator; and [128, 256), 64 per half, the bra's A (hi, lo 32 each)
// or the ket's A (hi, lo 16 each) and accumulator, whichever is live.
#pragma once
#include "tsbz_fft.cuh"
#include "tsbz_fused.cuh"
#include "tsbz_symbol.cuh"
#include "tsbz_umma.cuh"

#define FX_N 16
#define FX_NP 256                  // columns (threads)
#define FX_PTS 4096
#define FX_ROW 17                  // row pitch (float2) of the line buffer and of the z sums
#define FX_PL (FX_N * FX_ROW)      // plane pitch
#define FX_G 4                     // z groups
#define FX_S 8                     // atom slots
#define FX_COLS 256u               // tensor-memory columns
#define FX_BRA_D 0
#define FX_VEFF 16
#define FX_ACC 64
#define FX_BRA2_D 64
#define FX_BRA_A 128
#define FX_KET_A 128
#define FX_KET_D 160

struct FxSmem {
  float2 buf[FX_N * FX_PL];          // line transforms; second-order z sums
  float2 sums[2 * FX_G * FX_PL];     // first-order z sums
  unsigned char bket[4096];          // B of the ket (hi, lo)
  unsigned char bbra[4096];          // B of the first-order bra (hi, lo)
  unsigned char bbra2[8192];         // B of the second-order bra (hi, lo)
  float4 zt[FX_G * FX_N];            // z factors per group (Re F, Im F, d, 0)
  float4 xt[FX_S * FX_N];            // x and y factors per slot
  float4 yt[FX_S * FX_N];
  float4 xpk[FX_S * FX_N * 3];       // d_x^w F_x as (Re, Re, Im, Im) pairs, w = 0..2
  float2 gt[FX_S * 3 * FX_N];        // ket column tables
  float psc[4 * FX_S];               // dV pn: projection from a monomial sum
  float wsc[4 * FX_S];               // pn E times that: W from a monomial sum
  float2 mres[FX_S * 10];            // monomial sums
  Symbol<float> lam[3 * FX_N];       // kinetic symbol per axis and frequency
  float4 lam3[4 * FX_NP];            // and of the thread's line (k_x, k_z) at k_y = 4 i .. 4 i + 3
  int atom[FX_S];                    // atom of a slot (-1: empty)
  unsigned long long mbar;           // completion of the MMAs (one phase per commit)
  uint32_t tslot;
};

struct FxState {
  uint32_t tbase;   // tensor-memory base of the CTA
  uint32_t bar;     // shared address of FxSmem::mbar
  uint32_t phase;   // parity of the next completion
};

// byte offset of element (row n, k) of a K-major operand with 128-byte core
// matrices: K-direction stride 128, 8-row groups sbo apart
__device__ __forceinline__ int fx_boff(int n, int k, int sbo) {
  return (n >> 3) * sbo + (k >> 2) * 128 + (n & 7) * 16 + (k & 3) * 4;
}

// Allocation at the start of a kernel and release at its end (barriers inside).
__device__ __forceinline__ FxState fx_open(FxSmem& sm) {
  if ((threadIdx.x >> 5) == 0) um_alloc(bk_smem(&sm.tslot), FX_COLS);
  if (threadIdx.x == 0) bk_mbar_init(bk_smem(&sm.mbar), 1);
  um_fence_before();
  __syncthreads();
  um_fence_after();
  FxState x;
  x.tbase = sm.tslot;
  x.bar = bk_smem(&sm.mbar);
  x.phase = 0;
  return x;
}

__device__ __forceinline__ void fx_close(const FxState& x) {
  um_fence_before();
  __syncthreads();
  if ((threadIdx.x >> 5) == 0) {
    um_fence_after();
    um_dealloc(x.tbase, FX_COLS);
  }
}

// Failure path (every thread) after a poll that ran out: record it, give the MMAs in
// flight one more bounded wait, release the tensor memory.
__device__ __forceinline__ void fx_bail(const FxState& x, int* status) {
  if (threadIdx.x == 0) {
    atomicOr(status, BK_STATUS_TIMEOUT);
    bk_mbar_wait(x.bar, x.phase ^ 1u, BK_WAIT_POLLS);
  }
  fx_close(x);
}

// Completion of the last commit without a CTA barrier: the caller collects the
// result and checks it at its next barrier.
__device__ __forceinline__ bool fx_poll(FxState& x) {
  const bool ok = bk_mbar_wait(x.bar, x.phase, BK_WAIT_POLLS);
  x.phase ^= 1u;
  um_fence_after();
  return ok;
}

// Atom of a slot (-1: empty).
__device__ __forceinline__ int fx_atom(const CellDev& c, int s) {
  const int g = s >> 1, j = s & 1;
  return g < c.n_zg && j < c.zg_off[g + 1] - c.zg_off[g] ? c.zg_mem[c.zg_off[g] + j] : -1;
}
// Slots and scales of the cell (read after a barrier).
__device__ __forceinline__ void fx_scales(FxSmem& sm, const CellDev& c) {
  const int s = threadIdx.x;
  if (s < 4 * FX_S) {
    const int a = fx_atom(c, s >> 2), j = 4 * a + (s & 3);
    const float p = a < 0 ? 0.f : c.dvf * c.pnormf[j];
    if ((s & 3) == 0) sm.atom[s >> 2] = a;
    sm.psc[s] = p;
    sm.wsc[s] = a < 0 ? 0.f : p * c.wkbf[j];
  }
}

// Factor tables of one phase table; read after a barrier.
__device__ __forceinline__ void fx_tables(FxSmem& sm, const CellDev& c, const float2* ph) {
  const int tid = threadIdx.x, i = tid & (FX_N - 1), ax = (tid / FX_N) & 1, s = tid / (2 * FX_N);
  const int a = fx_atom(c, s);
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (a >= 0) {
    const int idx = (a * 3 + ax) * FX_N + i;
    const float g = c.g1f[idx];
    const float2 p = ph[idx];
    v = make_float4(g * p.x, g * p.y, c.d1f[idx], 0.f);
  }
  if (ax) {
    sm.yt[s * FX_N + i] = v;
  } else {
    sm.xt[s * FX_N + i] = v;
    float fr = v.x, fi = v.y;
#pragma unroll
    for (int w = 0; w < 3; ++w) {
      sm.xpk[(s * FX_N + i) * 3 + w] = make_float4(fr, fr, fi, fi);
      fr = __fmul_rn(v.z, fr);
      fi = __fmul_rn(v.z, fi);
    }
  }
  if (tid < FX_G * FX_N) {
    const int z = tid & (FX_N - 1), a0 = fx_atom(c, 2 * (tid / FX_N));
    float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
    if (a0 >= 0) {
      const int idx = (a0 * 3 + 2) * FX_N + z;
      const float g = c.g1f[idx];
      const float2 p = ph[idx];
      f = make_float4(g * p.x, g * p.y, c.d1f[idx], 0.f);
    }
    sm.zt[tid] = f;
  }
}

// B of the ket, K = 16 (Re rows of q, then Im rows), N = 32 (n = 2 z + c): hi at 0, lo at 2 KiB.
__device__ __forceinline__ void fx_build_ket(FxSmem& sm) {
  constexpr int Q = 2 * FX_G;
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int i = threadIdx.x + r * FX_NP, k = i >> 5, n = i & 31;
    const int q = k & (Q - 1), z = n >> 1, cc = n & 1;
    const float4 f = sm.zt[(q >> 1) * FX_N + z];
    const float sc = (q & 1) ? f.z : 1.f;
    const float zr = sc * f.x, zi = sc * f.y;
    uint32_t hi, lo;
    fs_split(k < Q ? (cc ? zi : zr) : (cc ? zr : -zi), hi, lo);
    *reinterpret_cast<uint32_t*>(sm.bket + fx_boff(n, k, 512)) = hi;
    *reinterpret_cast<uint32_t*>(sm.bket + 2048 + fx_boff(n, k, 512)) = lo;
  }
}

// B of an order-D bra, n = 2 q + c' (component of S; N = 16 D), k = 2 z + c (component of u): hi, then lo.
template <int D> __device__ __forceinline__ void fx_build_bra(FxSmem& sm, unsigned char* bz) {
  constexpr int NPAD = 16 * D, NQ = (D + 1) * FX_G, LO = NPAD / 8 * 1024;
#pragma unroll
  for (int r = 0; r < 32 * NPAD / FX_NP; ++r) {
    const int i = threadIdx.x + r * FX_NP, n = i >> 5, k = i & 31;
    const int q = n >> 1, cs = n & 1, z = k >> 1, cu = k & 1;
    float v = 0.f;
    if (q < NQ) {
      const int g = q / (D + 1), kz = q - g * (D + 1);
      const float4 f = sm.zt[g * FX_N + z];
      const float sc = kz == 0 ? 1.f : (kz == 1 ? f.z : f.z * f.z);
      const float zr = sc * f.x, zi = sc * f.y;
      v = cs == 0 ? (cu == 0 ? zr : -zi) : (cu == 0 ? zi : zr);
    }
    uint32_t hi, lo;
    fs_split(v, hi, lo);
    *reinterpret_cast<uint32_t*>(bz + fx_boff(n, k, 1024)) = hi;
    *reinterpret_cast<uint32_t*>(bz + LO + fx_boff(n, k, 1024)) = lo;
  }
}

// This thread's column u(z), split, as a row of the bra's A.
__device__ __forceinline__ void fx_stage(const float2 (&u)[FX_N], const FxState& x) {
  const int warp = threadIdx.x >> 5, h = warp >> 2, qd = warp & 3;
#pragma unroll
  for (int kk = 0; kk < 2; ++kk) {
    uint32_t hi[16], lo[16];
#pragma unroll
    for (int zz = 0; zz < 8; ++zz) {
      fs_split(u[8 * kk + zz].x, hi[2 * zz], lo[2 * zz]);
      fs_split(u[8 * kk + zz].y, hi[2 * zz + 1], lo[2 * zz + 1]);
    }
    um_st16(um_addr(x.tbase, qd, FX_BRA_A + 64 * h + 16 * kk), hi);
    um_st16(um_addr(x.tbase, qd, FX_BRA_A + 64 * h + 32 + 16 * kk), lo);
  }
}

// The MMAs of an order-D bra (one thread, after a barrier behind fx_stage and B's writes).
template <int D> __device__ __forceinline__ void fx_issue_bra(const FxState& x, const unsigned char* bz) {
  constexpr int NPAD = 16 * D, LO = NPAD / 8 * 1024;
  constexpr uint32_t idesc = um_idesc_tf32(128, NPAD);
  um_fence_after();
  const uint32_t b0 = bk_smem(bz), b1 = b0 + LO;
#pragma unroll
  for (int hh = 0; hh < 2; ++hh) {
    const uint32_t d = x.tbase + (D == 1 ? FX_BRA_D : FX_BRA2_D) + 32 * hh;
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
      const uint32_t a_hi = x.tbase + FX_BRA_A + 64 * hh + 8 * ks, a_lo = a_hi + 32;
      const uint64_t bh = um_sdesc(b0 + 256 * ks, 128, 1024), bl = um_sdesc(b1 + 256 * ks, 128, 1024);
      um_mma_tf32_ts(d, a_lo, bh, idesc, ks > 0);
      um_mma_tf32_ts(d, a_hi, bl, idesc, true);
    }
#pragma unroll
    for (int ks = 0; ks < 4; ++ks)   // the large products last (see um_mma_tf32_ts)
      um_mma_tf32_ts(d, x.tbase + FX_BRA_A + 64 * hh + 8 * ks, um_sdesc(b0 + 256 * ks, 128, 1024), idesc, true);
  }
  um_commit(x.bar);
}

// The thread's row of the bra's accumulator into zs[q][row][x] (after fx_poll).
template <int D> __device__ __forceinline__ void fx_collect(const FxState& x, float2* zs) {
  const int tid = threadIdx.x, warp = tid >> 5, h = warp >> 2, qd = warp & 3;
  float2* o = zs + (tid / FX_N) * FX_ROW + (tid & (FX_N - 1));
  const uint32_t at = um_addr(x.tbase, qd, (D == 1 ? FX_BRA_D : FX_BRA2_D) + 32 * h);
  if constexpr (D == 1) {
    float d[16];
    um_ld16(at, d);
#pragma unroll
    for (int q = 0; q < 2 * FX_G; ++q) o[q * FX_PL] = make_float2(d[2 * q], d[2 * q + 1]);
  } else {
    float d[32];
    um_ld32(at, d);
#pragma unroll
    for (int q = 0; q < 3 * FX_G; ++q) o[q * FX_PL] = make_float2(d[2 * q], d[2 * q + 1]);
  }
}

__device__ __forceinline__ float2 fx_lane_sum(float2 v) {   // over the 16 lanes of a half-warp
#pragma unroll
  for (int off = 1; off < 16; off <<= 1) {
    v.x = __fadd_rn(v.x, __shfl_xor_sync(0xffffffffu, v.x, off));
    v.y = __fadd_rn(v.y, __shfl_xor_sync(0xffffffffu, v.y, off));
  }
  return v;
}

// Monomial sums M(i, j, k) = sum_r F_x F_y F_z d_x^i d_y^j d_z^k u(r) of slot `warp`
// from the z sums.  Lanes 0 .. 15 (rows of k = 0) end with v = M_000, M_100, M_010 (D = 2:
// M_200, M_110, M_020 too), lanes 16 .. 31 (k = 1) with M_001 (M_101, M_011); m2 = M_002 (D = 2).
// The orders share the operations of their common sums, rounding for rounding.
template <int D>
__device__ __forceinline__ void fx_moments(const FxSmem& sm, const float2* zs, float2 (&v)[3 * D], float2& m2) {
  const int lane = threadIdx.x & 31, s = threadIdx.x >> 5, k = lane >> 4, i = lane & 15;
  const float4* xw = sm.xpk + s * FX_N * 3;
  const float2* row = zs + ((D + 1) * (s >> 1) + k) * FX_PL + i * FX_ROW;
  const float2 zero = make_float2(0.f, 0.f);
  // packed products: A_w += d^w Re F_x (s_re, s_im), B_w += d^w Im F_x (s_re, s_im);
  // R_w = (A_w.x - B_w.y, A_w.y + B_w.x)
  float2 A[D + 1], B[D + 1];
#pragma unroll
  for (int w = 0; w <= D; ++w) A[w] = B[w] = zero;
#pragma unroll
  for (int x = 0; x < FX_N; ++x) {
    const float2 sv = row[x];
#pragma unroll
    for (int w = 0; w <= D; ++w) {
      const float4 p = xw[x * 3 + w];
      A[w] = __ffma2_rn(make_float2(p.x, p.y), sv, A[w]);
      B[w] = __ffma2_rn(make_float2(p.z, p.w), sv, B[w]);
    }
  }
  float2 R[D + 1];
#pragma unroll
  for (int w = 0; w <= D; ++w) R[w] = make_float2(__fsub_rn(A[w].x, B[w].y), __fadd_rn(A[w].y, B[w].x));
  const float4 fy = sm.yt[s * FX_N + i];
  const float2 Fy = make_float2(fy.x, fy.y), Fd = make_float2(__fmul_rn(fy.z, fy.x), __fmul_rn(fy.z, fy.y));
  v[0] = fx_lane_sum(fs_cmul_rn(Fy, R[0]));
  v[1] = fx_lane_sum(fs_cmul_rn(Fy, R[1]));
  v[2] = fx_lane_sum(fs_cmul_rn(Fd, R[0]));
  if constexpr (D == 2) {
    v[3] = fx_lane_sum(fs_cmul_rn(Fy, R[2]));
    v[4] = fx_lane_sum(fs_cmul_rn(Fd, R[1]));
    v[5] = fx_lane_sum(fs_cmul_rn(make_float2(fy.z * Fd.x, fy.z * Fd.y), R[0]));
    // k = 2: row i, half of the x range per half-warp
    const float2* r2 = zs + (3 * (s >> 1) + 2) * FX_PL + i * FX_ROW + 8 * k;
    float2 a = zero, b = zero;
#pragma unroll
    for (int x = 0; x < 8; ++x) {
      const float4 p = xw[(8 * k + x) * 3];
      a = __ffma2_rn(make_float2(p.x, p.y), r2[x], a);
      b = __ffma2_rn(make_float2(p.z, p.w), r2[x], b);
    }
    float2 r = make_float2(a.x - b.y, a.y + b.x);
    r.x += __shfl_xor_sync(0xffffffffu, r.x, 16);
    r.y += __shfl_xor_sync(0xffffffffu, r.y, 16);
    m2 = fx_lane_sum(fs_cmul_rn(Fy, r));
  }
}

// P[j] = dV pn M of the slot's atom from a first-order pass.
__device__ __forceinline__ void fx_store_p(const FxSmem& sm, const float2* zs, float2* __restrict__ Pu) {
  const int lane = threadIdx.x & 31, s = threadIdx.x >> 5, a = sm.atom[s];
  float2 v[3], m2;
  fx_moments<1>(sm, zs, v, m2);
  if (a < 0 || (lane & 15)) return;
  const float* sc = sm.psc + 4 * s;
  if (lane == 0) {
#pragma unroll
    for (int t = 0; t < 3; ++t) Pu[4 * a + t] = make_float2(sc[t] * v[t].x, sc[t] * v[t].y);
  } else {
    Pu[4 * a + 3] = make_float2(sc[3] * v[0].x, sc[3] * v[0].y);
  }
}

// Rows (a_j, c_jx, c_jy, c_jz) of the slot's atom from a second-order pass into Pa, and
// a_j into Pnext if given.
__device__ __forceinline__ void fx_store_pa(FxSmem& sm, const float2* zs, float2* __restrict__ Pab,
                                            float2* __restrict__ Pnext) {
  const int lane = threadIdx.x & 31, s = threadIdx.x >> 5, a = sm.atom[s];
  float2 v[6], m2;
  fx_moments<2>(sm, zs, v, m2);
  float2* M = sm.mres + s * 10;
  if (lane == 0) {
    M[0] = v[0];
    M[1] = v[1];
    M[2] = v[2];
    M[4] = v[3];
    M[5] = v[4];
    M[7] = v[5];
    M[9] = m2;
  } else if (lane == 16) {
    M[3] = v[0];
    M[6] = v[1];
    M[8] = v[2];
  }
  __syncwarp();
  if (a < 0 || lane >= 16) return;
  // monomials w_t and w_t + e_alpha of projector type t
  const int t = lane >> 2, al = lane & 3;
  int e[3] = {t == 1 ? 1 : 0, t == 2 ? 1 : 0, t == 3 ? 1 : 0};
  if (al > 0) e[al - 1] += 1;
  const float2 m = M[fs_mono(e[0], e[1], e[2])];
  const float sc = sm.psc[4 * s + t];
  const float2 p = make_float2(sc * m.x, sc * m.y);
  Pab[4 * (4 * a + t) + al] = p;
  if (Pnext && al == 0) Pnext[4 * a + t] = p;
}

// A whole order-D pass over the staged column: z sums in zs (read after the
// function); false when the MMAs did not complete.  build: B is formed in bz here (else
// it is there already, fenced).
template <int D>
__device__ __forceinline__ bool fx_pass(FxSmem& sm, FxState& x, unsigned char* bz, float2* zs, bool build) {
  if (build) {
    fx_build_bra<D>(sm, bz);
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  }
  um_fence_before();
  __syncthreads();
  if (threadIdx.x == 0) fx_issue_bra<D>(x, bz);
  const bool ok = fx_poll(x);
  fx_collect<D>(x, zs);
  return __syncthreads_and(ok) != 0;
}

// Ket tables of slot `warp` from its weights W (lane-wise: see the callers):
// lanes 0 .. 15 write G00, G10 of x = lane, lanes 16 .. 31 G01.
__device__ __forceinline__ void fx_ket_tables(FxSmem& sm, float2 ws, float2 wx, float2 wy, float2 wz) {
  const int lane = threadIdx.x & 31, s = threadIdx.x >> 5, i = lane & 15;
  const float4 fx = sm.xt[s * FX_N + i];
  const float2 F = make_float2(fx.x, fx.y);
  float2* gt = sm.gt + s * 3 * FX_N + i;
  if (lane < 16) {
    gt[0] = sep_cmul(F, make_float2(fmaf(fx.z, wx.x, ws.x), -fmaf(fx.z, wx.y, ws.y)));
    gt[FX_N] = sep_cmul(F, make_float2(wy.x, -wy.y));
  } else {
    gt[2 * FX_N] = sep_cmul(F, make_float2(wz.x, -wz.y));
  }
}

// W of slot `warp` from the band's projections (lane t < 4 gets projector t), and the
// ket tables from it (every lane of the warp).
__device__ __forceinline__ float2 fx_load_w(const CellDev& c, const float2* __restrict__ Pu) {
  const int lane = threadIdx.x & 31, a = fx_atom(c, threadIdx.x >> 5);
  float2 w = make_float2(0.f, 0.f);
  if (a >= 0 && lane < 4) {
    const float2 p = Pu[4 * a + lane];
    const float e = c.wkbf[4 * a + lane];
    w = make_float2(e * p.x, e * p.y);
  }
  return w;
}
__device__ __forceinline__ void fx_ket_from_w(FxSmem& sm, float2 w) {
  float2 v[4];
#pragma unroll
  for (int t = 0; t < 4; ++t)
    v[t] = make_float2(__shfl_sync(0xffffffffu, w.x, t), __shfl_sync(0xffffffffu, w.y, t));
  fx_ket_tables(sm, v[0], v[1], v[2], v[3]);
}

// One CTA takes `per` bands of a unit in turn: under a constant field the unit's
// tables and operand matrices, v_eff and the symbol serve them all, and the next
// band is on its way to L2.  The set-up is a chain of dependent loads, about 1.0 ms
// of the 6.9 ms launch with one band per CTA (65 536 orbitals).
// FRESH: the projections of psi are formed from the band (else taken from P).
template <bool FRESH>
__global__ void __launch_bounds__(FX_NP, 2) k_step_fft(LaunchSet L, float2* __restrict__ psi, float2* __restrict__ P,
                                                       float2* __restrict__ Pa, int same_next, int want_pa, int per) {
  step_enter();
  constexpr int N = FX_N, NP = FX_NP, Q = 2 * FX_G;
  extern __shared__ __align__(128) unsigned char fs_raw[];
  FxSmem& sm = *reinterpret_cast<FxSmem*>(fs_raw);
  const CellDev& c = L.cell;
  const int groups = (c.n_bands + per - 1) / per;
  const int u = L.unit_ids[blockIdx.x / groups];
  const UnitDev U = L.units[u];
  const int tid = threadIdx.x, lo = tid & (N - 1), hi = tid / N;   // as a column: ix, iy
  const int warp = tid >> 5, h = warp >> 2, qd = warp & 3;
  const int b0 = (blockIdx.x % groups) * per, b1 = min(b0 + per, c.n_bands);
  const long long off = (long long)u * L.ph_stride;
  float2* band = psi + U.psi_off + (long long)b0 * FX_PTS + tid;
  // every load of the set-up is issued before the first barrier
  float2 t[N];
#pragma unroll
  for (int z = 0; z < N; ++z) t[z] = band[z * NP];
  const SubDev S = L.subs[U.sub];
  if (*S.active == 0) return;
  float2 w = fx_load_w(c, P + U.p_off + (long long)b0 * c.n_proj);
  fx_tables(sm, c, (const float2*)L.ph_half + off);
  fx_scales(sm, c);
  if (tid < 3 * N) sm.lam[tid] = symbol_unit<float>(L, u)[tid];
  FxState x = fx_open(sm);   // (and the barrier behind the tables)
  {
    float v[N];
    const float* veff = reinterpret_cast<const float*>(S.veff) + tid;
#pragma unroll
    for (int z = 0; z < N; ++z) v[z] = veff[z * NP];
    um_st16(um_addr(x.tbase, qd, FX_VEFF + 32 * h), reinterpret_cast<uint32_t(&)[16]>(v));
  }
  {
    const Symbol<float> xz = symbol_add(sm.lam[lo], sm.lam[2 * N + hi]);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = symbol_value(symbol_add(xz, sm.lam[N + 4 * i + k]));
      sm.lam3[i * NP + tid] = make_float4(v[0], v[1], v[2], v[3]);
    }
  }
  fx_build_ket(sm);
  fx_build_bra<1>(sm, sm.bbra);
  const bool keep = same_next && per > 1;   // one second-order B for all bands
  if (keep) fx_build_bra<2>(sm, sm.bbra2);
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");   // the B's, issued behind later barriers
  float2* colp = sm.buf + hi * FX_ROW + lo;            // the column: planes FX_PL apart
  float2* rowp = sm.buf + hi * FX_PL + lo * FX_ROW;    // row y = lo of plane z = hi
  float2* linp = sm.buf + hi * FX_PL + lo;             // line x = lo of plane z = hi
  const float dt = (float)(S.dt * L.dt_scale);
#pragma unroll 1
  for (int b = b0; b < b1; ++b, band += FX_PTS) {
    float2* Pu = P + U.p_off + (long long)b * c.n_proj;
    if (b > b0) {
#pragma unroll
      for (int z = 0; z < N; ++z) t[z] = band[z * NP];
      w = fx_load_w(c, Pu);
      __syncthreads();   // the last band's sums are consumed
      if (!same_next) {
        fx_tables(sm, c, (const float2*)L.ph_half + off);
        __syncthreads();
        fx_build_bra<1>(sm, sm.bbra);
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      }
    }
    if (b + 1 < b1) {
      const char* next = reinterpret_cast<const char*>(band - tid + FX_PTS) + 128 * tid;
      asm volatile("prefetch.global.L2 [%0];\n" ::"l"(next));
    }
    if (FRESH) {
      fx_stage(t, x);
      um_fence_before();
      __syncthreads();
      if (tid == 0) fx_issue_bra<1>(x, sm.bbra);
    } else {
      fx_ket_from_w(sm, w);
    }
    float coef = 1.f;
    bool ok = true;
#pragma unroll 1
    for (int m = 1; m <= 4; ++m) {
      const bool chain = m > 1 || FRESH;
      float2 f[N];
#pragma unroll
      for (int z = 0; z < N; ++z) f[z] = t[z];
      fft_line<N, -1>(f);
#pragma unroll
      for (int z = 0; z < N; ++z) colp[z * FX_PL] = f[z];
      if (chain) {
        ok = ok && fx_poll(x);   // z sums of s_{m-1}
        fx_collect<1>(x, sm.sums);
      }
      if (!__syncthreads_and(ok)) {
        if (chain) {
          fx_bail(x, S.status);
        } else {
          fx_close(x);
        }
        return;
      }
      if (chain) {
        float2 v[3], m2;
        fx_moments<1>(sm, sm.sums, v, m2);
        const float* sc = sm.wsc + 4 * warp;
        fx_ket_tables(sm, make_float2(sc[0] * v[0].x, sc[0] * v[0].y), make_float2(sc[1] * v[1].x, sc[1] * v[1].y),
                      make_float2(sc[2] * v[2].x, sc[2] * v[2].y), make_float2(sc[3] * v[0].x, sc[3] * v[0].y));
      }
      // forward along x and y, the symbol, back: within the half-warp's plane
#pragma unroll
      for (int k = 0; k < N; ++k) f[k] = rowp[k];
      fft_line<N, -1>(f);
#pragma unroll
      for (int k = 0; k < N; ++k) rowp[k] = f[k];
      __syncwarp();
#pragma unroll
      for (int y = 0; y < N; ++y) f[y] = linp[y * FX_ROW];
      fft_line<N, -1>(f);
      {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float4 l = sm.lam3[i * NP + tid];
          f[4 * i] = __fmul2_rn(make_float2(l.x, l.x), f[4 * i]);
          f[4 * i + 1] = __fmul2_rn(make_float2(l.y, l.y), f[4 * i + 1]);
          f[4 * i + 2] = __fmul2_rn(make_float2(l.z, l.z), f[4 * i + 2]);
          f[4 * i + 3] = __fmul2_rn(make_float2(l.w, l.w), f[4 * i + 3]);
        }
      }
      fft_line<N, 1>(f);
#pragma unroll
      for (int y = 0; y < N; ++y) linp[y * FX_ROW] = f[y];
      __syncwarp();
#pragma unroll
      for (int k = 0; k < N; ++k) f[k] = rowp[k];
      fft_line<N, 1>(f);
#pragma unroll
      for (int k = 0; k < N; ++k) rowp[k] = f[k];
      __syncthreads();
      {
        // the ket's A row of the column
        float2 av[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) av[q] = make_float2(0.f, 0.f);
#pragma unroll
        for (int s = 0; s < FX_S; ++s) {
          const float4 fy = sm.yt[s * N + hi];
          const float2 g0 = sm.gt[(s * 3 + 0) * N + lo], g1 = sm.gt[(s * 3 + 1) * N + lo];
          const float2 g2 = sm.gt[(s * 3 + 2) * N + lo];
          const float2 e = __ffma2_rn(make_float2(fy.z, fy.z), g1, g0);
          float2& a0 = av[2 * (s >> 1)];
          float2& a1 = av[2 * (s >> 1) + 1];
          a0.x = fmaf(fy.x, e.x, fmaf(-fy.y, e.y, a0.x));
          a0.y = fmaf(fy.x, e.y, fmaf(fy.y, e.x, a0.y));
          a1.x = fmaf(fy.x, g2.x, fmaf(-fy.y, g2.y, a1.x));
          a1.y = fmaf(fy.x, g2.y, fmaf(fy.y, g2.x, a1.y));
        }
        uint32_t ah[16], al[16];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
          fs_split(av[q].x, ah[q], al[q]);
          fs_split(av[q].y, ah[Q + q], al[Q + q]);
        }
        um_st16(um_addr(x.tbase, qd, FX_KET_A + 64 * h), ah);
        um_st16(um_addr(x.tbase, qd, FX_KET_A + 64 * h + 16), al);
      }
      um_fence_before();
      __syncthreads();
      if (tid == 0) {
        um_fence_after();
        constexpr uint32_t idesc = um_idesc_tf32(128, 32);
        const uint32_t b0 = bk_smem(sm.bket), b1 = b0 + 2048;
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
          const uint32_t d = x.tbase + FX_KET_D + 64 * hh;
#pragma unroll
          for (int ks = 0; ks < 2; ++ks) {
            const uint32_t a_hi = x.tbase + FX_KET_A + 64 * hh + 8 * ks, a_lo = a_hi + 16;
            const uint64_t bh = um_sdesc(b0 + 256 * ks, 128, 512), bl = um_sdesc(b1 + 256 * ks, 128, 512);
            um_mma_tf32_ts(d, a_lo, bh, idesc, ks > 0);
            um_mma_tf32_ts(d, a_hi, bl, idesc, true);
          }
#pragma unroll
          for (int ks = 0; ks < 2; ++ks)
            um_mma_tf32_ts(d, x.tbase + FX_KET_A + 64 * hh + 8 * ks, um_sdesc(b0 + 256 * ks, 128, 512), idesc, true);
        }
        um_commit(x.bar);
      }
      // the kinetic term of the column, under the ket's MMAs
#pragma unroll
      for (int z = 0; z < N; ++z) f[z] = colp[z * FX_PL];
      fft_line<N, 1>(f);
      // s_m = kinetic + v s_{m-1} + V_NL s_{m-1}
      {
        float v[16];
        um_ld16(um_addr(x.tbase, qd, FX_VEFF + 32 * h), v);
#pragma unroll
        for (int z = 0; z < N; ++z) t[z] = __ffma2_rn(make_float2(v[z], v[z]), t[z], f[z]);
      }
      ok = fx_poll(x);
      {
        float d[32];
        um_ld32(um_addr(x.tbase, qd, FX_KET_D + 64 * h), d);   // conj(V_NL s_{m-1})
#pragma unroll
        for (int z = 0; z < N; ++z) {
          t[z].x += d[2 * z];
          t[z].y -= d[2 * z + 1];
        }
      }
      if (m == 1) {
#pragma unroll
        for (int z = 0; z < N; ++z) t[z] = __fmul2_rn(make_float2(dt, dt), t[z]);
      } else {
        coef *= dt / (float)m;
      }
      if (m < 4) fx_stage(t, x);   // the bra's A
      // the increment of psi: (-i)^m coef s_m summed over m
      {
        float2 a[N];
        if (m == 1) {
#pragma unroll
          for (int z = 0; z < N; ++z) a[z] = make_float2(t[z].y, -t[z].x);
        } else {
          um_ld32(um_addr(x.tbase, qd, FX_ACC + 32 * h), reinterpret_cast<float(&)[32]>(a));
          const float sg = m == 4 ? coef : -coef;
          if (m == 3) {
#pragma unroll
            for (int z = 0; z < N; ++z) {
              a[z].x = fmaf(sg, t[z].y, a[z].x);
              a[z].y = fmaf(-sg, t[z].x, a[z].y);
            }
          } else {
#pragma unroll
            for (int z = 0; z < N; ++z) a[z] = __ffma2_rn(make_float2(sg, sg), t[z], a[z]);
          }
        }
        if (m < 4) {
          um_st32(um_addr(x.tbase, qd, FX_ACC + 32 * h), reinterpret_cast<float(&)[32]>(a));
        } else {
#pragma unroll
          for (int z = 0; z < N; ++z) t[z] = fft_add(band[z * NP], a[z]);
        }
      }
      um_fence_before();
      if (!__syncthreads_and(ok)) {   // at m = 4: every buffer is free
        fx_bail(x, S.status);
        return;
      }
      if (m < 4 && tid == 0) fx_issue_bra<1>(x, sm.bbra);
    }
#pragma unroll
    for (int z = 0; z < N; ++z) band[z * NP] = t[z];
    if (want_pa) {
      // projections of the new psi: those of the next step (P, q of the next step) and of
      // the current (Pa, q at t_{n+1}); a constant field makes both q's the step's own, so
      // the tables stay and the next step's are the current's first-order sums
      fx_stage(t, x);
      bool done = true;
      if (!same_next) {
        fx_tables(sm, c, (const float2*)L.ph_next + off);
        __syncthreads();
        done = fx_pass<1>(sm, x, sm.bbra, sm.sums, true);
        if (done) {
          fx_store_p(sm, sm.sums, Pu);
          __syncthreads();
          fx_tables(sm, c, (const float2*)L.ph_obs + off);
          __syncthreads();
        }
      }
      done = done && fx_pass<2>(sm, x, sm.bbra2, sm.buf, !keep);
      if (!done) {
        fx_bail(x, S.status);
        return;
      }
      fx_store_pa(sm, sm.buf, Pa + U.pa_off + 4LL * b * c.n_proj, same_next ? Pu : nullptr);
    }
  }
  fx_close(x);
}

// Projections outside a step, one CTA per (unit, band), by the same passes: P on the
// q_half tables (PA = false; so a restored state's equal those the step leaves, bit
// for bit) or the current's Pa on the q_obs tables (J(0-), J(0+), restored states).
template <bool PA>
__global__ void __launch_bounds__(FX_NP, 2) k_project_fft(LaunchSet L, const float2* __restrict__ src,
                                                          float2* __restrict__ out) {
  extern __shared__ __align__(128) unsigned char fs_raw[];
  FxSmem& sm = *reinterpret_cast<FxSmem*>(fs_raw);
  const CellDev& c = L.cell;
  const int b = blockIdx.x % c.n_bands;
  const int u = L.unit_ids[blockIdx.x / c.n_bands];
  if (!unit_active(L, u)) return;
  const UnitDev U = L.units[u];
  fx_scales(sm, c);
  FxState x = fx_open(sm);
  const float2* band = src + U.psi_off + (long long)b * FX_PTS + threadIdx.x;
  float2 t[FX_N];
#pragma unroll
  for (int z = 0; z < FX_N; ++z) t[z] = band[z * FX_NP];
  fx_tables(sm, c, (const float2*)(PA ? L.ph_obs : L.ph_half) + (long long)u * L.ph_stride);
  fx_stage(t, x);
  __syncthreads();
  if (!fx_pass<PA ? 2 : 1>(sm, x, sm.bbra2, sm.buf, true)) {
    fx_bail(x, L.subs[U.sub].status);
    return;
  }
  if (PA)
    fx_store_pa(sm, sm.buf, out + U.pa_off + 4LL * b * c.n_proj, nullptr);
  else
    fx_store_p(sm, sm.buf, out + U.p_off + (long long)b * c.n_proj);
  fx_close(x);
}
