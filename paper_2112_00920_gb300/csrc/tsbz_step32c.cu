// The whole time step of a band in one launch, FP32 on 32^3 grids (cell B): a
// cluster of 8 CTAs holds the band, each CTA four y rows (128 columns, two threads a
// column with the even and the odd planes).
//
// What bounds it: instruction issue at 16 warps per SM; psi crosses HBM once per
// step, where the per-stage slab kernels moved it eight times and waited on a
// barrier per plane.  The kinetic operator is diagonal in the Fourier basis along
// z and x, which are local to a CTA (32-point lines, two threads each: one
// decimation step, then 16 points in registers); along y the star stencil runs on
// the transformed rows, the neighbour CTAs' four rows on either side read through
// distributed shared memory (the same volume as a transform's two exchanges,
// with one exchange instead of two; the same barrier publishes the partial projections).
// Projectors: z sums of the columns on tcgen05 (three bfloat16 parts, A in tensor
// memory), x sums per (atom, row) over the atom's box, y sums over the CTA's rows,
// and the eight CTAs' partial sums added in rank order through distributed
// shared memory.  The ket goes back the same way, its contraction along z on
// tcgen05 under the line transforms.  Atoms whose x (y, z) tables are identical share
// them: at most 8 classes per axis (a 2 x 2 x 2 diamond supercell has 8).
// Taylor terms are s_m = dt h^m psi; the rest of (-i dt)^m / m! enters the sum only (see
// tsbz_any.cu; psi stays in the sum here: adding it last spilled, 2.00 -> 2.08 ms, and
// gained nothing on so many points).
// Measured: 8 k-points x 128 bands of the 64-atom cell, stages and projections 3.31 ->
// 1.98 ms per step (36% of issue slots, the rest barriers and the latency of the
// remote rows).
// Every wait on an MMA is bounded; a CTA that gave up keeps taking part in the
// cluster's barriers and reports at the end.
// Tensor-memory columns: Taylor sum [0, 64), v_eff [64, 96), bra accumulator of the large
// products [96, 128), and [128, 256): the bra's A (three parts) and its accumulator of
// the small products, or the ket's A (hi, lo) and accumulators.  The second-order bra
// accumulates in [0, 96).
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "tsbz_bulk.cuh"
#include "tsbz_fft.cuh"
#include "tsbz_internal.h"
#include "tsbz_launch.cuh"
#include "tsbz_symbol.cuh"
#include "tsbz_umma.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int QN = 32;            // points per axis
constexpr int QT = 256;           // threads
constexpr int QR = 4;             // rows per CTA
constexpr int QC = 8;             // CTAs per cluster
constexpr int QP = 33;            // row pitch (float2): no bank conflicts along any axis
constexpr int QBUF = QR * QN * QP;
constexpr int QA = 64;            // atom slots
constexpr int QG = 8;             // z groups, x and y classes
constexpr int Q_ACC = 0, Q_VEFF = 64, Q_OP = 128;
constexpr int Q_BRA_D = 96, Q_BRA_S = 208, Q_BRA2_D = 0, Q_BRA2_S = 48;   // accumulators of large and small products
constexpr uint32_t Q_COLS = 256;
constexpr int Q_KET_B = 16384, Q_BRA_B = 12288, Q_BRA2_B = 18432;
constexpr size_t Q_IMG = Q_KET_B + Q_BRA_B + Q_BRA2_B;   // B images of a unit: ket, first- and second-order bra

struct QSmem {
  float2 b1[QBUF];                 // line buffers [row][z or k_z][x or k_x]
  float2 b2[QBUF];
  unsigned char bket[Q_KET_B];     // B of the ket (hi, lo)
  unsigned char bbra[Q_BRA_B];     // B of the first-order bra (three parts)
  float4 xt[QG * QN];              // x factors per class (Re F, Im F, d, 0)
  float4 yt[QG * QR];              // y factors per class on the CTA's rows
  float2 tab[QA * QR * 3];         // ket tables per (slot, row); second-order partial sums
  float2 part[QA * 4];             // this CTA's partial monomial sums
  Symbol<float> lx[QN], lz[QN];    // kinetic symbol along x and z
  float wl[4], wg[4], wd;          // stencil along y and its diagonal, transforms' 1/N^2 folded in
  unsigned long long ymask[QR];    // slots whose y factor is non-zero on the row
  int atom[QA];                    // atom of a slot (-1: none)
  unsigned char xc[QA], yc[QA], zg[QA];
  int xs[QG], xl[QG];              // x box of a class: start, length
  unsigned long long mbar;         // completion of the MMAs
  unsigned long long mimg;         // arrival of the B images
  uint32_t tslot;
};

__device__ __forceinline__ uint32_t q_tf32(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;\n" : "=r"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ void q_split(float x, uint32_t& hi, uint32_t& lo) {
  hi = q_tf32(x);
  lo = q_tf32(x - __uint_as_float(hi));
}
__device__ __forceinline__ float2 q_mul(float2 a, float2 b) {
  return make_float2(__fmaf_rn(a.x, b.x, -__fmul_rn(a.y, b.y)), __fmaf_rn(a.x, b.y, __fmul_rn(a.y, b.x)));
}
__device__ __forceinline__ float2 q_mac(float2 a, float2 b, float2 c) {   // c + a b
  return make_float2(__fmaf_rn(a.x, b.x, __fmaf_rn(-a.y, b.y, c.x)), __fmaf_rn(a.x, b.y, __fmaf_rn(a.y, b.x, c.y)));
}
__device__ __forceinline__ float2 q_axpy(float s, float2 b, float2 a) {
  return make_float2(__fmaf_rn(s, b.x, a.x), __fmaf_rn(s, b.y, a.y));
}
__device__ __forceinline__ float2 q_add(float2 a, float2 b) {
  return make_float2(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y));
}

// One decimation step of a 32-point line and a 16-point transform: thread half s gets
// the outputs k = 2 m + s in f[m].  src: the line, `stride` apart.
template <int SIGN>
__device__ __forceinline__ void q_line(const float2* src, int stride, int s, float2 (&f)[16]) {
  if (s == 0) {
#pragma unroll
    for (int j = 0; j < 16; ++j) f[j] = fft_add(src[j * stride], src[(j + 16) * stride]);
  } else {
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const float2 d = fft_sub(src[j * stride], src[(j + 16) * stride]);
      const float c = (float)fft_cos32(j), n = (float)(SIGN * fft_sin32(j));   // times exp(SIGN 2 pi i j / 32)
      f[j] = j == 0 ? d : make_float2(fmaf(d.x, c, -d.y * n), fmaf(d.x, n, d.y * c));
    }
  }
  fft_line<16, SIGN>(f);
}

struct QState {
  uint32_t tbase, bar, phase;
};

__device__ __forceinline__ bool q_poll(QState& x) {
  const bool ok = bk_mbar_wait(x.bar, x.phase, BK_WAIT_POLLS);
  x.phase ^= 1u;
  um_fence_after();
  return ok;
}

__device__ __forceinline__ void q_st8(uint32_t taddr, const uint32_t (&r)[8]) {
  __syncwarp();
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};\n"
      "tcgen05.wait::st.sync.aligned;\n" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
      : "memory");
}

// The cluster's barrier in two halves (every thread of every CTA, alternating).
__device__ __forceinline__ void q_arrive() { asm volatile("barrier.cluster.arrive.release;\n" ::: "memory"); }
__device__ __forceinline__ void q_wait() { asm volatile("barrier.cluster.wait.acquire;\n" ::: "memory"); }

// Slots, classes and boxes of the cell; ends with a barrier.
__device__ void q_cell(QSmem& sm, const CellDev& c) {
  const int tid = threadIdx.x;
  if (tid < QA) {
    const bool in = tid < c.zs_off[c.zs_n];
    const int a = in ? c.zs_mem[tid] : -1;
    int g = 0;
    while (in && tid >= c.zs_off[g + 1]) ++g;
    sm.atom[tid] = a;
    sm.zg[tid] = (unsigned char)g;
    sm.xc[tid] = in ? c.xc_of[a] : 0;
    sm.yc[tid] = in ? c.yc_of[a] : 0;
  }
  if (tid < QG) {
    const bool in = tid < c.xc_n;
    sm.xs[tid] = in ? c.pbox[c.xc_rep[tid] * 6] : 0;
    sm.xl[tid] = in ? c.pbox[c.xc_rep[tid] * 6 + 1] : 0;
  }
  __syncthreads();
}

// z factor of group g at plane z times d^k.
__device__ __forceinline__ float2 q_zfactor(const CellDev& c, const float2* ph, int g, int z, int k) {
  const int i = (c.zs_mem[c.zs_off[g]] * 3 + 2) * QN + z;
  float s = c.g1f[i];
  const float d = c.d1f[i];
  for (int e = 0; e < k; ++e) s *= d;
  return make_float2(s * ph[i].x, s * ph[i].y);
}

// B of an order-D bra (N = 32 or 48): n = 2 q + c', q = (D + 1) g + k; K = 64:
// kk = 32 h + 2 j + c for z = 2 j + h.  Three parts (um_split3), N/8 KiB each.  A warp writes one
// 8 x 16-byte core matrix (no bank conflicts), a lane both components of a plane.
template <int D> __device__ void q_build_bra(unsigned char* bz, const CellDev& c, const float2* ph) {
  constexpr int NN = D == 1 ? 32 : 48, PART = NN / 8 * 1024;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll 2
  for (int m = warp; m < NN / 8 * 8; m += QT / 32) {
    const int n = 8 * (m >> 3) + (lane >> 2), kk = 8 * (m & 7) + 2 * (lane & 3);
    const int q = n >> 1, g = q / (D + 1), k = q - g * (D + 1), z = (kk & 30) + (kk >> 5);
    float2 f = make_float2(0.f, 0.f);
    if (g < c.zs_n) f = q_zfactor(c, ph, g, z, k);
    uint32_t r[3];
    um_split3((n & 1) == 0 ? make_float2(f.x, -f.y) : make_float2(f.y, f.x), r);
#pragma unroll
    for (int i = 0; i < 3; ++i) *reinterpret_cast<uint32_t*>(bz + PART * i + 128 * m + 4 * lane) = r[i];
  }
}

// B of the ket: n = 2 (16 h' + j) + c for z = 2 j + h' (N = 64); K = 32: kk = 16 h + 8 part + i for
// q = 8 h + i, part 0 the real, 1 the imaginary coefficient.
__device__ void q_build_ket(unsigned char* bz, const CellDev& c, const float2* ph) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll 2
  for (int m = warp; m < 64; m += QT / 32) {
    const int n = 8 * (m >> 3) + (lane >> 2), kk = 4 * (m & 7) + (lane & 3);
    const int zi = n >> 1, cc = n & 1, z = 2 * (zi & 15) + (zi >> 4);
    const int q = 8 * (kk >> 4) + (kk & 7), part = (kk >> 3) & 1, g = q >> 1;
    float2 f = make_float2(0.f, 0.f);
    if (g < c.zs_n) f = q_zfactor(c, ph, g, z, q & 1);
    uint32_t hi, lo;
    q_split(part == 0 ? (cc ? f.y : f.x) : (cc ? f.x : -f.y), hi, lo);
    *reinterpret_cast<uint32_t*>(bz + 128 * m + 4 * lane) = hi;
    *reinterpret_cast<uint32_t*>(bz + 8192 + 128 * m + 4 * lane) = lo;
  }
}

// The B matrices depend on the unit's tables only: one CTA per unit writes their images
// after the field kernel rebuilt the tables (q_half for the stages, q_obs for the
// current), and the step's CTAs fetch them by bulk copies.  Built in each of a
// unit's 1024 CTAs they took 0.26 of 2.29 ms (128 bands).
__global__ void __launch_bounds__(QT) k_images32(LaunchSet L, unsigned char* __restrict__ img) {
  step_enter();
  const CellDev& c = L.cell;
  const int u = L.unit_ids[blockIdx.x];
  if (!unit_active(L, u)) return;
  unsigned char* o = img + (size_t)blockIdx.x * Q_IMG;
  const float2* phh = (const float2*)L.ph_half + (long long)u * L.ph_stride;
  const float2* pho = (const float2*)L.ph_obs + (long long)u * L.ph_stride;
  if (blockIdx.y == 0) q_build_ket(o, c, phh);
  if (blockIdx.y == 1) q_build_bra<1>(o + Q_KET_B, c, phh);
  if (blockIdx.y == 2) q_build_bra<2>(o + Q_KET_B + Q_BRA_B, c, pho);
}

// x factors of the classes, y factors on the CTA's rows, rows' slot masks; ends with a barrier.
__device__ void q_tables(QSmem& sm, const CellDev& c, const float2* ph, int r0) {
  const int tid = threadIdx.x;
  {
    const int cl = tid >> 5, i = tid & 31;   // 8 classes x 32 points
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (cl < c.xc_n) {
      const int k = c.xc_rep[cl] * 3 * QN + i;
      const float g = c.g1f[k];
      v = make_float4(g * ph[k].x, g * ph[k].y, c.d1f[k], 0.f);
    }
    sm.xt[tid] = v;
  }
  if (tid < QG * QR) {
    const int cl = tid >> 2, r = tid & 3;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (cl < c.yc_n) {
      const int k = (c.yc_rep[cl] * 3 + 1) * QN + r0 + r;
      const float g = c.g1f[k];
      v = make_float4(g * ph[k].x, g * ph[k].y, c.d1f[k], g);
    }
    sm.yt[tid] = v;
  }
  __syncthreads();
  if (tid < QR * 2) {   // 32 slots each
    const int r = tid >> 1, s0 = 32 * (tid & 1);
    unsigned m = 0;
    for (int s = 0; s < 32; ++s)
      if (sm.atom[s0 + s] >= 0 && sm.yt[sm.yc[s0 + s] * QR + r].w != 0.f) m |= 1u << s;
    reinterpret_cast<unsigned*>(&sm.ymask[r])[tid & 1] = m;
  }
  __syncthreads();
}

// Tensor-memory columns of a thread half's operands, one or the other live: the bra's A, 16 words
// per part, and the ket's A and accumulator.  The next stage's bra is written while the other
// half may still read its ket accumulator, so neither half's columns meet the other's.
__host__ __device__ constexpr int q_bra_a(int h, int part) { return part < 2 ? Q_OP + 32 * h + 16 * part : Q_OP + 64 + 48 * h; }
__host__ __device__ constexpr int q_ket_a(int h) { return Q_OP + 32 * h; }
__host__ __device__ constexpr int q_ket_d(int h) { return Q_OP + 64 + 32 * h; }

// The column's planes as a row of the bra's A.
__device__ __forceinline__ void q_stage(const float2 (&u)[16], const QState& x) {
  const int warp = threadIdx.x >> 5, h = warp >> 2, qd = warp & 3;
  uint32_t p[3][16];
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    uint32_t r[3];
    um_split3(u[j], r);
#pragma unroll
    for (int i = 0; i < 3; ++i) p[i][j] = r[i];
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) um_st16(um_addr(x.tbase, qd, q_bra_a(h, i)), p[i]);
}

// The MMAs of an order-D bra (one thread, behind a barrier after q_stage and B's fenced writes):
// the products of the first parts by themselves, the five next ones (down to 2^-18) in an
// accumulator of their own; what is left out is below 2^-26.
template <int D> __device__ __forceinline__ void q_issue_bra(const QState& x, const unsigned char* bz) {
  constexpr int NN = D == 1 ? 32 : 48, PART = NN / 8 * 1024;
  constexpr uint32_t idesc = um_idesc_bf16(128, NN);
  um_fence_after();
  const uint32_t b = bk_smem(bz);
  const uint32_t d0 = x.tbase + (D == 1 ? Q_BRA_D : Q_BRA2_D), d1 = x.tbase + (D == 1 ? Q_BRA_S : Q_BRA2_S);
  // (part of A, part of B), the smallest products first
  constexpr int pa[6] = {2, 0, 1, 1, 0, 0}, pb[6] = {0, 2, 1, 0, 1, 0};
#pragma unroll
  for (int i = 0; i < 6; ++i)
#pragma unroll
    for (int ks = 0; ks < 4; ++ks)
      um_mma_bf16_ts(i < 5 ? d1 : d0, x.tbase + q_bra_a(ks >> 1, pa[i]) + 8 * (ks & 1),
                     um_sdesc(b + PART * pb[i] + 256 * ks, 128, 1024), idesc, ks > 0 || (i > 0 && i < 5));
  um_commit(x.bar);
}

// The thread's share of its column's z sums into zs[q][row][x] (after q_poll).
template <int D> __device__ __forceinline__ void q_collect(const QState& x, float2* zs) {
  constexpr int DC = D == 1 ? Q_BRA_D : Q_BRA2_D, DS = D == 1 ? Q_BRA_S : Q_BRA2_S;
  const int tid = threadIdx.x, warp = tid >> 5, h = warp >> 2, qd = warp & 3;
  const int col = tid & 127, o = (col >> 5) * QP + (col & 31);
  float d[16], e[16];
  um_ld16(um_addr(x.tbase, qd, DC + (D == 1 ? 16 : 32) * h), d);   // q = 8 h .. (D = 2: 16 h ..)
  um_ld16(um_addr(x.tbase, qd, DS + (D == 1 ? 16 : 32) * h), e);
#pragma unroll
  for (int i = 0; i < 8; ++i)
    zs[((D == 1 ? 8 : 16) * h + i) * QR * QP + o] =
        make_float2(__fadd_rn(d[2 * i], e[2 * i]), __fadd_rn(d[2 * i + 1], e[2 * i + 1]));
  if constexpr (D == 2) {
    um_ld16(um_addr(x.tbase, qd, DC + 16), d);   // q = 8 .. 15, four for each half
    um_ld16(um_addr(x.tbase, qd, DS + 16), e);
#pragma unroll
    for (int i = 0; i < 16; ++i) d[i] = __fadd_rn(d[i], e[i]);
#pragma unroll
    for (int i = 0; i < 4; ++i)
      zs[(8 + 4 * h + i) * QR * QP + o] =
          h ? make_float2(d[8 + 2 * i], d[9 + 2 * i]) : make_float2(d[2 * i], d[2 * i + 1]);
  }
}

// The CTA's partial monomial sums of order <= D of slot tid / 4 over its rows: thread
// (slot, row); lane row 0 stores them.  D = 1: out[4 slot + (000, 100, 010, 001)];
// D = 2: out[10 slot + mono].  The orders share the operations of their common sums.
template <int D> __device__ __forceinline__ void q_moments(const QSmem& sm, const float2* zs, float2* out) {
  const int s = threadIdx.x >> 2, r = threadIdx.x & 3;
  const float2 zero = make_float2(0.f, 0.f);
  float2 R0[D + 1], R1[D], R2 = zero;   // k = 0: w <= D; k = 1: w < D; k = 2: w = 0
#pragma unroll
  for (int w = 0; w <= D; ++w) R0[w] = zero;
#pragma unroll
  for (int w = 0; w < D; ++w) R1[w] = zero;
  const float4 fy = sm.yt[sm.yc[s] * QR + r];
  if ((sm.ymask[r] >> s) & 1) {
    const int xc = sm.xc[s], start = sm.xs[xc], len = sm.xl[xc];
    const float4* xt = sm.xt + xc * QN;
    const float2* z0 = zs + ((D + 1) * sm.zg[s] * QR + r) * QP;
#pragma unroll 3
    for (int j = 0; j < len; ++j) {
      const int x = (start + j) & (QN - 1);
      const float4 f = xt[x];
      const float2 F = make_float2(f.x, f.y);
      const float2 p0 = q_mul(F, z0[x]), p1 = q_mul(F, z0[QR * QP + x]);
      R0[0] = q_add(R0[0], p0);
      R0[1] = q_axpy(f.z, p0, R0[1]);
      R1[0] = q_add(R1[0], p1);
      if constexpr (D == 2) {
        R0[D] = q_axpy(__fmul_rn(f.z, f.z), p0, R0[D]);
        R1[D - 1] = q_axpy(f.z, p1, R1[D - 1]);
        R2 = q_add(R2, q_mul(F, z0[2 * QR * QP + x]));
      }
    }
  }
  const float2 F = make_float2(fy.x, fy.y);
  constexpr int NM = D == 1 ? 4 : 10;
  float2 m[NM];
  const float2 a0 = q_mul(F, R0[0]);
  m[0] = a0;
  m[1] = q_mul(F, R0[1]);
  m[2] = make_float2(__fmul_rn(fy.z, a0.x), __fmul_rn(fy.z, a0.y));
  m[3] = q_mul(F, R1[0]);
  if constexpr (D == 2) {   // 200 110 101 020 011 002
    m[4] = q_mul(F, R0[D]);
    m[5] = make_float2(fy.z * m[1].x, fy.z * m[1].y);
    m[6] = q_mul(F, R1[D - 1]);
    m[7] = make_float2(fy.z * m[2].x, fy.z * m[2].y);
    m[8] = make_float2(fy.z * m[3].x, fy.z * m[3].y);
    m[9] = q_mul(F, R2);
  }
#pragma unroll
  for (int e = 0; e < NM; ++e)
#pragma unroll
    for (int off = 1; off < 4; off <<= 1) {
      m[e].x = __fadd_rn(m[e].x, __shfl_xor_sync(0xffffffffu, m[e].x, off));
      m[e].y = __fadd_rn(m[e].y, __shfl_xor_sync(0xffffffffu, m[e].y, off));
    }
  if (r == 0)
#pragma unroll
    for (int e = 0; e < NM; ++e) out[NM * s + e] = m[e];
}

// Sum over the cluster's CTAs, in rank order, of entry i of the partial sums `p`.
__device__ __forceinline__ float2 q_total(cg::cluster_group& cl, float2* p, int i) {
  float2 v = make_float2(0.f, 0.f);
#pragma unroll
  for (int r = 0; r < QC; ++r) v = q_add(v, cl.map_shared_rank(p, r)[i]);
  return v;
}

// Rows (a_j, c_jx, c_jy, c_jz) from the second-order pass of the staged columns into Pab
// (and a_j into Pnext if given).  The CTA of rank r writes the slots 8 r .. 8 r + 7.
// img: the unit's images; parity: of the copy's arrival.
__device__ bool q_current(QSmem& sm, cg::cluster_group& cl, QState& x, const CellDev& c, const unsigned char* img,
                          uint32_t parity, float2* __restrict__ Pab, float2* __restrict__ Pnext) {
  unsigned char* bz = reinterpret_cast<unsigned char*>(sm.b1);
  const uint32_t bar = bk_smem(&sm.mimg);
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  um_fence_before();
  __syncthreads();
  bool ok = true;
  if (threadIdx.x == 0) {
    bk_mbar_expect_tx(bar, Q_BRA2_B);
    bk_copy_g2s(bk_smem(bz), img + Q_KET_B + Q_BRA_B, Q_BRA2_B, bar);
    ok = bk_mbar_wait(bar, parity, BK_WAIT_POLLS);
    q_issue_bra<2>(x, bz);
  }
  ok = q_poll(x) && ok;
  q_collect<2>(x, sm.b2);
  __syncthreads();
  q_moments<2>(sm, sm.b2, sm.tab);
  cl.sync();
  const int tid = threadIdx.x, s = (int)cl.block_rank() * 8 + (tid >> 4), o = tid & 15;
  if (tid < 128 && sm.atom[s] >= 0) {
    const int t = o >> 2, al = o & 3, a = sm.atom[s];
    int e[3] = {t == 1, t == 2, t == 3};
    if (al > 0) e[al - 1] += 1;
    const int deg = e[0] + e[1] + e[2];
    const int mo = deg == 0 ? 0 : deg == 1 ? (e[0] ? 1 : (e[1] ? 2 : 3))
                 : e[0] == 2 ? 4 : e[0] == 1 ? (e[1] ? 5 : 6) : e[1] == 2 ? 7 : e[1] ? 8 : 9;
    const float2 M = q_total(cl, sm.tab, 10 * s + mo);
    const float sc = __fmul_rn(c.dvf, c.pnormf[4 * a + t]);
    const float2 p = make_float2(__fmul_rn(sc, M.x), __fmul_rn(sc, M.y));
    Pab[4 * (4 * a + t) + al] = p;
    if (Pnext && al == 0) Pnext[4 * a + t] = p;
  }
  return ok;
}

__device__ __forceinline__ QState q_open(QSmem& sm) {
  if ((threadIdx.x >> 5) == 0) um_alloc(bk_smem(&sm.tslot), Q_COLS);
  if (threadIdx.x == 0) {
    bk_mbar_init(bk_smem(&sm.mbar), 1);
    bk_mbar_init(bk_smem(&sm.mimg), 1);
  }
  um_fence_before();
  __syncthreads();
  um_fence_after();
  return QState{sm.tslot, bk_smem(&sm.mbar), 0u};
}

// Every CTA of the cluster: report, release the tensor memory, leave together.
__device__ __forceinline__ void q_close(cg::cluster_group& cl, const QState& x, bool ok, int* status) {
  if (!ok && (threadIdx.x & 31) == 0) atomicOr(status, BK_STATUS_TIMEOUT);
  um_fence_before();
  cl.sync();
  if ((threadIdx.x >> 5) == 0) {
    um_fence_after();
    um_dealloc(x.tbase, Q_COLS);
  }
}

// One time step of every band (arguments as launch_step64).
__global__ void __cluster_dims__(QC, 1, 1) __launch_bounds__(QT, 2)
    k_step_fft32(LaunchSet L, const unsigned char* __restrict__ images, float2* __restrict__ psi,
                 float2* __restrict__ P, float2* __restrict__ Pa, int fresh_p, int want_pa, int same_next) {
  step_enter();
  extern __shared__ __align__(128) unsigned char q_raw[];
  QSmem& sm = *reinterpret_cast<QSmem*>(q_raw);
  cg::cluster_group cl = cg::this_cluster();
  const CellDev& c = L.cell;
  const int rank = (int)cl.block_rank(), orb = blockIdx.x / QC;
  const int b = orb % c.n_bands;
  const int u = L.unit_ids[orb / c.n_bands];
  if (!unit_active(L, u)) return;   // the whole cluster
  const UnitDev U = L.units[u];
  const SubDev S = L.subs[U.sub];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, h = warp >> 2, qd = warp & 3;
  const int col = tid & 127, ry = col >> 5, ix = col & 31, r0 = rank * QR;
  float2* Pu = P + U.p_off + (long long)b * c.n_proj;
  const long long at = (long long)h * QN * QN + (r0 + ry) * QN + ix;   // plane z = 2 j + h: + 2 j QN^2
  float2* band = psi + U.psi_off + (long long)b * c.npts + at;
  const float2* ph = (const float2*)L.ph_half + (long long)u * L.ph_stride;
  const float* qt = reinterpret_cast<const float*>(L.qt_half) + 4 * u;
  const unsigned char* img = images + (size_t)(orb / c.n_bands) * Q_IMG;
  QState x = q_open(sm);
  if (tid == 0) {
    const uint32_t bar = bk_smem(&sm.mimg);
    bk_mbar_expect_tx(bar, Q_KET_B + Q_BRA_B);
    bk_copy_g2s(bk_smem(sm.bket), img, Q_KET_B, bar);
    bk_copy_g2s(bk_smem(sm.bbra), img + Q_KET_B, Q_BRA_B, bar);
  }
  float2 t[16];
  {
    float v[16];
    const float* veff = reinterpret_cast<const float*>(S.veff) + at;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      t[j] = band[2 * j * QN * QN];
      v[j] = veff[2 * j * QN * QN];
    }
    um_st16(um_addr(x.tbase, qd, Q_VEFF + 16 * h), reinterpret_cast<uint32_t(&)[16]>(v));
    um_st32(um_addr(x.tbase, qd, Q_ACC + 32 * h), reinterpret_cast<float(&)[32]>(t));
  }
  constexpr float inv = 1.f / (QN * QN);
  if (tid < 64) {
    const int ax = tid < 32 ? 0 : 2, k = tid & 31;
    (ax == 0 ? sm.lx : sm.lz)[k] = symbol_unit<float>(L, u)[ax * QN + k];
  } else if (tid < 68) {
    sm.wl[tid - 64] = c.hlapf[1][tid - 63] * inv;
    sm.wg[tid - 64] = qt[1] * c.gradwf[1][tid - 63] * inv;
  } else if (tid == 68) {
    sm.wd = fmaf(0.5f * qt[1], qt[1], c.hlapf[1][0]) * inv;
  }
  q_cell(sm, c);
  q_tables(sm, c, ph, r0);
  const int line = (ry * QN + ix) * QP;                  // as a line: row ry, plane (frequency) ix
  float2* c1 = sm.b1 + ry * QN * QP + ix;                // the column, planes QP apart
  float2* c2 = sm.b2 + ry * QN * QP + ix;
  const float2* up = cl.map_shared_rank(sm.b1, (rank + 1) & (QC - 1));
  const float2* dn = cl.map_shared_rank(sm.b1, (rank + QC - 1) & (QC - 1));
  const float dt = (float)(S.dt * L.dt_scale);
  float coef = 1.f;
  bool ok = bk_mbar_wait(bk_smem(&sm.mimg), 0, BK_WAIT_POLLS);
  q_arrive();   // (this CTA's b1 is free)
#pragma unroll 1
  for (int m = 1; m <= 4; ++m) {
    const bool chain = m > 1 || fresh_p;   // projections of s_{m-1} from the column, else from P
    float2 f[16];
    if (chain) q_stage(t, x);
    q_wait();   // the neighbours are done with this CTA's b1 and partial sums
#pragma unroll
    for (int j = 0; j < 16; ++j) c1[(2 * j + h) * QP] = t[j];
    um_fence_before();
    __syncthreads();
    if (chain && tid == 0) q_issue_bra<1>(x, sm.bbra);
    // forward along z under the z sums' MMAs
    q_line<-1>(c1, QP, h, f);
#pragma unroll
    for (int i = 0; i < 16; ++i) c2[(2 * i + h) * QP] = f[i];
    __syncthreads();
    if (chain) {
      ok = q_poll(x) && ok;
      q_collect<1>(x, sm.b1);
      um_fence_before();
      __syncthreads();
      q_moments<1>(sm, sm.b1, sm.part);
      __syncthreads();
    }
    // forward along x
    q_line<-1>(sm.b2 + line, 1, h, f);
#pragma unroll
    for (int i = 0; i < 16; ++i) sm.b1[line + 2 * i + h] = f[i];
    cl.sync();   // rows and partial sums of every CTA
    {
      const int s = tid >> 2, a = sm.atom[s], j = 4 * a + (tid & 3);
      float2 w = make_float2(0.f, 0.f);
      if (a >= 0) {
        float2 p;
        if (chain) {
          const float2 M = q_total(cl, sm.part, tid);
          const float sc = __fmul_rn(c.dvf, c.pnormf[j]);
          p = make_float2(__fmul_rn(sc, M.x), __fmul_rn(sc, M.y));
        } else {
          p = Pu[j];
        }
        const float e = c.wkbf[j];
        w = make_float2(e * p.x, e * p.y);
      }
      sm.b2[tid] = w;   // (the rows before the x transform are consumed)
    }
    __syncwarp();
    {
      // ket tables of (slot, row): F_y conj(W_s + d_y W_py), F_y conj(W_px), F_y conj(W_pz)
      const int s = tid >> 2, r = tid & 3;
      const float4 fy = sm.yt[sm.yc[s] * QR + r];
      const float2 F = make_float2(fy.x, fy.y);
      const float2 ws = sm.b2[4 * s], wx = sm.b2[4 * s + 1], wy = sm.b2[4 * s + 2], wz = sm.b2[4 * s + 3];
      float2* o = sm.tab + 3 * tid;
      o[0] = q_mul(F, make_float2(fmaf(fy.z, wy.x, ws.x), -fmaf(fy.z, wy.y, ws.y)));
      o[1] = q_mul(F, make_float2(wx.x, -wx.y));
      o[2] = q_mul(F, make_float2(wz.x, -wz.y));
    }
    __syncthreads();
    {
      // the ket's A row of the column: groups 4 h .. 4 h + 3
      float2 av[8];
      const unsigned long long rows = sm.ymask[ry];
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        float2 a0 = make_float2(0.f, 0.f), a1 = a0;
        const int e0 = c.zs_off[4 * h + g], n = c.zs_off[4 * h + g + 1] - e0;
        unsigned long long bits = n > 0 ? (rows >> e0) & (n >= 64 ? ~0ull : (1ull << n) - 1) : 0ull;
        while (bits) {
          const int s = e0 + __ffsll((long long)bits) - 1;
          bits &= bits - 1;
          const float4 fx = sm.xt[sm.xc[s] * QN + ix];
          const float2* o = sm.tab + 3 * (4 * s + ry);
          const float2 F = make_float2(fx.x, fx.y);
          a0 = q_mac(F, q_axpy(fx.z, o[1], o[0]), a0);
          a1 = q_mac(F, o[2], a1);
        }
        av[2 * g] = a0;
        av[2 * g + 1] = a1;
      }
      uint32_t rh[8], rl[8], ih[8], il[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        q_split(av[i].x, rh[i], rl[i]);
        q_split(av[i].y, ih[i], il[i]);
      }
      const uint32_t o = um_addr(x.tbase, qd, q_ket_a(h));
      q_st8(o, rh);
      q_st8(o + 8, ih);
      q_st8(o + 16, rl);
      q_st8(o + 24, il);
    }
    um_fence_before();
    __syncthreads();
    if (tid == 0) {
      // the ket's MMAs, under the transforms that follow
      um_fence_after();
      constexpr uint32_t idesc = um_idesc_tf32(128, 32);
      const uint32_t b0 = bk_smem(sm.bket), b1 = b0 + 8192;
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {   // planes of half hh
        const uint32_t d = x.tbase + q_ket_d(hh);
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {
          const uint32_t a_hi = x.tbase + q_ket_a(ks >> 1) + 8 * (ks & 1), a_lo = a_hi + 16;
          const uint64_t bh = um_sdesc(b0 + 4096 * hh + 256 * ks, 128, 1024);
          const uint64_t bl = um_sdesc(b1 + 4096 * hh + 256 * ks, 128, 1024);
          um_mma_tf32_ts(d, a_lo, bh, idesc, ks > 0);
          um_mma_tf32_ts(d, a_hi, bl, idesc, true);
        }
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {   // the large products last
          const uint32_t a_hi = x.tbase + q_ket_a(ks >> 1) + 8 * (ks & 1);
          um_mma_tf32_ts(d, a_hi, um_sdesc(b0 + 4096 * hh + 256 * ks, 128, 1024), idesc, true);
        }
      }
      um_commit(x.bar);
    }
    // symbol along x and z, stencil along y: thread (k_x = lane, k_z = warp + 8 i), four rows
    float2 wl[4], wg[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      wl[e] = make_float2(sm.wl[e], sm.wl[e]);
      wg[e] = make_float2(sm.wg[e], sm.wg[e]);
    }
    // (the diagonal stays apart: added to the symbol it would round that of long waves at its own size)
    const Symbol<float> lx = sm.lx[lane];
    const float2 wd = make_float2(sm.wd, sm.wd);
#pragma unroll 2
    for (int i = 0; i < 4; ++i) {
      const int kz = warp + 8 * i, o = kz * QP + lane;
      float2 w[12];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        w[r] = dn[r * QN * QP + o];
        w[4 + r] = sm.b1[r * QN * QP + o];
        w[8 + r] = up[r * QN * QP + o];
      }
      const float l = symbol_value(symbol_add(lx, sm.lz[kz]));
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        float2 k = __ffma2_rn(wd, w[4 + r], __fmul2_rn(make_float2(l, l), w[4 + r]));
        float2 g = make_float2(0.f, 0.f);
#pragma unroll
        for (int e = 1; e <= 4; ++e) {
          const float2 a = w[4 + r + e], d = w[4 + r - e];
          k = __ffma2_rn(wl[e - 1], fft_add(a, d), k);
          g = __ffma2_rn(wg[e - 1], fft_sub(a, d), g);
        }
        sm.b2[r * QN * QP + o] = make_float2(k.x + g.y, k.y - g.x);   // -i q grad
      }
    }
    q_arrive();
    __syncthreads();
    // back along x (in place: the line's two threads sit in warps w and w + 4) and z
    q_line<1>(sm.b2 + line, 1, h, f);
    asm volatile("bar.sync %0, 64;\n" ::"r"(1 + qd) : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) sm.b2[line + 2 * i + h] = f[i];
    __syncthreads();
    q_line<1>(c2, QP, h, f);
    {
      float v[16];
      um_ld16(um_addr(x.tbase, qd, Q_VEFF + 16 * h), v);
#pragma unroll
      for (int j = 0; j < 16; ++j) t[j] = __ffma2_rn(make_float2(v[j], v[j]), t[j], f[j]);
    }
    ok = q_poll(x) && ok;
    {
      float d[32];
      um_ld32(um_addr(x.tbase, qd, q_ket_d(h)), d);   // conj(V_NL s_{m-1})
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        t[j].x += d[2 * j];
        t[j].y -= d[2 * j + 1];
      }
    }
    if (m == 1) {
#pragma unroll
      for (int j = 0; j < 16; ++j) t[j] = __fmul2_rn(make_float2(dt, dt), t[j]);
    } else {
      coef *= dt / (float)m;
    }
    {
      // psi += (-i)^m coef s_m
      float2 a[16];
      um_ld32(um_addr(x.tbase, qd, Q_ACC + 32 * h), reinterpret_cast<float(&)[32]>(a));
      const float sg = m == 1 || m == 4 ? coef : -coef;
      if (m & 1) {
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          a[j].x = fmaf(sg, t[j].y, a[j].x);
          a[j].y = fmaf(-sg, t[j].x, a[j].y);
        }
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) a[j] = __ffma2_rn(make_float2(sg, sg), t[j], a[j]);
      }
      if (m < 4) {
        um_st32(um_addr(x.tbase, qd, Q_ACC + 32 * h), reinterpret_cast<float(&)[32]>(a));
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) t[j] = a[j];
      }
    }
  }
#pragma unroll
  for (int j = 0; j < 16; ++j) band[2 * j * QN * QN] = t[j];
  q_wait();   // the neighbours are done with b1
  if (want_pa) {
    // a constant field leaves the step's tables in place (q_obs = q_half)
    __syncthreads();   // this CTA is done with its tables
    if (!same_next) q_tables(sm, c, (const float2*)L.ph_obs + (long long)u * L.ph_stride, r0);
    q_stage(t, x);
    ok = q_current(sm, cl, x, c, img, 1, Pa + U.pa_off + 4LL * b * c.n_proj, same_next ? Pu : nullptr) && ok;
  }
  q_close(cl, x, ok, S.status);
}

// Projections of the current outside a step.
__global__ void __cluster_dims__(QC, 1, 1) __launch_bounds__(QT, 2)
    k_pa_fft32(LaunchSet L, const unsigned char* __restrict__ images, const float2* __restrict__ src,
               float2* __restrict__ Pa) {
  extern __shared__ __align__(128) unsigned char q_raw[];
  QSmem& sm = *reinterpret_cast<QSmem*>(q_raw);
  cg::cluster_group cl = cg::this_cluster();
  const CellDev& c = L.cell;
  const int rank = (int)cl.block_rank(), orb = blockIdx.x / QC;
  const int b = orb % c.n_bands;
  const int u = L.unit_ids[orb / c.n_bands];
  if (!unit_active(L, u)) return;
  const UnitDev U = L.units[u];
  const int tid = threadIdx.x, h = tid >> 7, col = tid & 127;
  const float2* band = src + U.psi_off + (long long)b * c.npts + (long long)h * QN * QN +
                       (rank * QR + (col >> 5)) * QN + (col & 31);
  const float2* ph = (const float2*)L.ph_obs + (long long)u * L.ph_stride;
  QState x = q_open(sm);
  float2 t[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) t[j] = band[2 * j * QN * QN];
  q_stage(t, x);
  q_cell(sm, c);
  q_tables(sm, c, ph, rank * QR);
  const bool ok = q_current(sm, cl, x, c, images + (size_t)(orb / c.n_bands) * Q_IMG, 0,
                            Pa + U.pa_off + 4LL * b * c.n_proj, nullptr);
  q_close(cl, x, ok, L.subs[U.sub].status);
}

bool q_cell_ok(const CellDev& c) {
  return c.n1 == QN && c.n2 == QN && c.n3 == QN && c.nd == 4 && c.use_proj && c.n_atoms <= QA && c.zs_n > 0 &&
         c.zs_n <= QG && c.xc_n > 0 && c.yc_n > 0;
}
bool q_taken(const LaunchSet& L) { return L.variant == 0 && L.images != nullptr && q_cell_ok(L.cell); }

template <typename K> void q_attr(K* k) {
  cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(QSmem));
}

static_assert(sizeof(QSmem) <= 115712, "two CTAs per SM");

}  // namespace

size_t step_fft32_images(const CellDev& c, int n_units) { return q_cell_ok(c) ? Q_IMG * (size_t)n_units : 0; }

void launch_images_fft32(const LaunchSet& L, void* stream) {
  if (L.n_units == 0 || !q_taken(L)) return;
  step_launch(k_images32, dim3(L.n_units, 3), QT, 0, stream, L, (unsigned char*)L.images);
}

bool launch_step_fft32(const LaunchSet& L, void* psi, void* P, void* Pa, int fresh_p, int want_pa, int same_next,
                       void* stream) {
  if (L.n_units == 0 || !q_taken(L)) return false;
  q_attr(k_step_fft32);
  step_launch(k_step_fft32, (unsigned)L.n_units * L.cell.n_bands * QC, QT, sizeof(QSmem), stream, L,
              (const unsigned char*)L.images, (float2*)psi, (float2*)P, (float2*)Pa, fresh_p, want_pa, same_next);
  return true;
}

bool launch_pa_fft32(const LaunchSet& L, const void* src, void* Pa, void* stream) {
  if (L.n_units == 0 || !q_taken(L)) return false;
  q_attr(k_pa_fft32);
  k_pa_fft32<<<(unsigned)L.n_units * L.cell.n_bands * QC, QT, sizeof(QSmem), (cudaStream_t)stream>>>(
      L, (const unsigned char*)L.images, (const float2*)src, (float2*)Pa);
  return true;
}
