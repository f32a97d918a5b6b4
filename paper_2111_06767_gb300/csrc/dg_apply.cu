// Matrix-free DG operator A u on affine hexahedral LGL elements (Sec. II).
//
// Poisson fluxes (Eq. poisson_fluxform), strong form in two steps (Eqs. dg_op_auxvars and
// dg_op_primal), generalized internal-penalty flux (Eq. numflux) with the penalty of
// Eq. penalty and homogeneous Dirichlet boundary fluxes (Eq. bc), massive form (b = M f).
// Integrals use LGL collocation quadrature: M is diagonal, MD_i = M D_i and the lifting acts
// on face points only.
//
// Per element, with g_d = (2/h_d) Dhat_d u the local gradient:
//   v_d   = g_d + s (u_ext - u_int) / (w_0 h_d)                      on face points of normal s e_d
//   A u   = -M sum_d (2/h_d) Dhat_d v_d
//           - sum_faces Bf [ s/2 (g_ext - g_int) + (sigma_d - 1/(w_0 h_d)) (u_ext - u_int) ]
// where Bf = J_f w_a w_b is the face quadrature weight. At an external face Eq. bc with
// (n F_v)^b = n u_b, u_b = 0, and (n F_u)^b = (n F_u)^int is the ghost state u_ext = -u_int,
// g_ext = g_int, which this kernel uses on Dirichlet faces. On a homogeneous Neumann face of the
// box (Eq. bc with (n F_v)^b = (n F_v)^int and a zero prescribed normal flux (n F_u)^b = 0) the
// ghost state is u_ext = u_int, g_ext = -g_int: no jump, no lifting and a zero numerical flux.
//
// Kernels: apply_dir_kernel and apply_par_kernel (dir_apply.cuh) for every order, precision and
// output; apply_elem4_kernel for the plain FP32 apply at N = 4; coarse_smooth_kernel, which runs
// the apply inside a fused smoother.
#include <algorithm>
#include <mutex>
#include <set>
#include <type_traits>

#include "bounds.cuh"
#include "dir_apply.cuh"
#include "internal.h"
#include "lines.cuh"
#include "pdl.cuh"
#include "schwarz_dev.cuh"
#include "tcgen05.cuh"

namespace dg {

namespace {

// Operator tables in constant memory, so that with unrolled (compile-time) indices they are operands
// of the FMA instructions themselves: the LGL weights of every supported N and Dhat of N = 4.
constexpr int wtab_off(int N) { return N * (N - 1) / 2 - 1; }  // sum_{m=2}^{N-1} m
constexpr int kWTab = wtab_off(DG_MAX_N + 1);
__constant__ float2 cDD4[16], cB4[8];
__constant__ double cW64[kWTab];
__constant__ float cW32[kWTab], cWlo32[kWTab];  // value and rounding error

// Tables of the direction-by-direction kernel (dir_apply.cuh)
__constant__ double2 cPQ64[kDirPairs], cQP64[kDirPairs];
__constant__ float2 cPQ32[kDirPairs], cQP32[kDirPairs];
__constant__ double cV64[kDirVec];
__constant__ float cV32[kDirVec];
template <int N, typename T>
struct DirTab;
template <int N>
struct DirTab<N, double> {
  static __device__ __forceinline__ double2 PQ(int i) { return cPQ64[i]; }
  static __device__ __forceinline__ double2 QP(int i) { return cQP64[i]; }
  static __device__ __forceinline__ double vec(int i) { return cV64[i]; }
  static __device__ __forceinline__ double w(int l) { return cW64[wtab_off(N) + l]; }
  static __device__ __forceinline__ double w_lo(int) { return 0.0; }
};
template <int N>
struct DirTab<N, float> {
  static __device__ __forceinline__ float2 PQ(int i) { return cPQ32[i]; }
  static __device__ __forceinline__ float2 QP(int i) { return cQP32[i]; }
  static __device__ __forceinline__ float vec(int i) { return cV32[i]; }
  static __device__ __forceinline__ float w(int l) { return cW32[wtab_off(N) + l]; }
  static __device__ __forceinline__ float w_lo(int l) { return cWlo32[wtab_off(N) + l]; }
};

__device__ __forceinline__ void row4_g(const float* __restrict__ p, float (&r)[4]) {
  const float4 v = __ldg(reinterpret_cast<const float4*>(p));
  r[0] = v.x;
  r[1] = v.y;
  r[2] = v.z;
  r[3] = v.w;
}

// ------------------------------------------------------------------ element-per-thread apply (N = 4, FP32)
//
// At N = 4 an element is 64 values, few enough for one thread to hold the element, one gradient
// component and the result in registers, so the three contractions need no exchange between
// threads at all. A CTA owns a brick of BX x BY x BZ elements. One TMA load stages the brick with a
// one-element halo ((BX+2) x (BY+2) x (BZ+2) elements; elements outside the domain arrive as zeros
// and are replaced by the ghost state) in shared memory, each element padded from 64 to 68 words:
// the 16-byte reads of consecutive elements at one offset then fall into distinct banks. A thread
// reads its element and its six face neighbours from there (a neighbour's normal derivative at the
// shared face needs its whole element), works direction by direction (gradient component, face
// lifting and fluxes, divergence), and the result leaves through the same padded layout with one
// TMA store, which clips elements outside the domain. The flux of a face point enters the per-point
// sum before the mass-matrix scaling, divided by that point's M: Bf / M = Jf_d / (J w_0) at every
// face point of a face normal to d. Values are held as pairs of x-neighbouring points, so that the
// contractions and most face terms run as packed two-wide FP32 FMAs (one instruction per pair):
// the thread's 64-value working set leaves too few warps per SM to hide latency otherwise.
// What bounds it: the instructions of 8 warps per SM (255 registers a thread), with the wait for the staged box
// between them; so the gradient stays in reference units (one scaling per direction, squared, at the divergence), a
// face point is five operations, and Dhat is read from constant memory as pairs. Measured at 96^3 elements (56.6M
// points): 162 us with scalar constants and scaled gradients (3190 instructions an element), 147 us with the
// reference units, 129 us with the pairs (2190; 0.52 of the HBM copy rate). Bricks staged without their edges (seven
// boxes): 136 us, 4 x 4 x 4 and 8 x 4 x 2 bricks of that form 127 us, not worth four more tensor maps a launch.
constexpr int kE4Slot = 68;  // words per staged element

struct E4Tab {
  static __device__ __forceinline__ float2 DD(int o) { return cDD4[o]; }  // (D, D)
  static __device__ __forceinline__ float2 B(int o) { return cB4[o]; }    // pairs of the x-contraction
  static __device__ __forceinline__ float w(int o) { return cW32[wtab_off(4) + o]; }
};

template <int BX, int BY, int BZ>
struct E4Shape {
  static constexpr int PX = BX + 2, PY = BY + 2, PZ = BZ + 2;
  static constexpr int THREADS = BX * BY * BZ;
  static constexpr int IN_WORDS = PX * PY * PZ * kE4Slot;
  static constexpr int SMEM = IN_WORDS * 4 + 16 + 128;  // staged box, mbarrier, alignment slack
  static constexpr int PER_SM = (228 * 1024) / (SMEM + 1024) > 8 ? 8 : (228 * 1024) / (SMEM + 1024);
  static_assert(PER_SM >= 1 && SMEM <= 227 * 1024, "staged brick must fit in shared memory");
  static_assert(BX <= 254 && BY <= 254 && BZ <= 254, "TMA boxes are at most 256 elements per dimension");
};

__device__ __forceinline__ void ld4p(const float* p, float2 (&r)[2]) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  r[0] = make_float2(v.x, v.y);
  r[1] = make_float2(v.z, v.w);
}

__device__ __forceinline__ void ld4s(const float* p, float (&r)[4]) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  r[0] = v.x;
  r[1] = v.y;
  r[2] = v.z;
  r[3] = v.w;
}

// One face in reference units: gi and ge are the derivatives along the reference coordinate (physical / dxi), and
// ue, ge are zero where there is no neighbour (the staged box is filled with zeros there). The jump uE - ui is then
// ue + bj ui and the derivative's ge + bg gi, with (bj, bg) = (-1, -1) where the neighbour exists, (-2, 0) on a
// Dirichlet and (0, -2) on a Neumann face, and a face point is five operations: two of these, the flux
// cf (s / 2 dxi dg + sml jump) into the pre-mass sum (cf = Bf / M of the point), and the lifting.
struct E4Face {
  float bj, bg, ch, cs, sl;
  __device__ __forceinline__ E4Face(float s, bool has, bool neu, float dxi, float lift, float sml, float cf) {
    bj = has ? -1.f : (neu ? 0.f : -2.f);
    bg = has ? -1.f : (neu ? -2.f : 0.f);
    ch = 0.5f * s * dxi * cf;
    cs = cf * sml;
    sl = s * lift / dxi;
  }
  // returns the lifted derivative, adds the flux to acc
  __device__ __forceinline__ float apply(float ui, float gi, float ue, float ge, float& acc) const {
    const float jump = fmaf(bj, ui, ue), dg = fmaf(bg, gi, ge);
    acc = fmaf(cs, jump, fmaf(ch, dg, acc));
    return fmaf(sl, jump, gi);
  }
  // two face points at once
  __device__ __forceinline__ float2 apply(float2 ui, float2 gi, float2 ue, float2 ge, float2& acc) const {
    const float2 jump = __ffma2_rn(make_float2(bj, bj), ui, ue), dg = __ffma2_rn(make_float2(bg, bg), gi, ge);
    acc = __ffma2_rn(make_float2(cs, cs), jump, __ffma2_rn(make_float2(ch, ch), dg, acc));
    return __ffma2_rn(make_float2(sl, sl), jump, gi);
  }
};

template <int BX, int BY, int BZ>
__global__ void __launch_bounds__(BX* BY* BZ, E4Shape<BX, BY, BZ>::PER_SM)
    apply_elem4_kernel(const ApplyArgs<float> A, const __grid_constant__ CUtensorMap mu,
                       const __grid_constant__ CUtensorMap mo, int* __restrict__ err) {
  using S = E4Shape<BX, BY, BZ>;
  using C = E4Tab;
  constexpr int SL = kE4Slot, PX = S::PX, PY = S::PY;
  constexpr int wO = 0;
  extern __shared__ __align__(128) unsigned char e4_raw[];
  // 128-byte aligned for TMA; offset from the shared array itself, so that the compiler keeps
  // every access in the shared window (LDS/STS rather than generic loads)
  float* sm = reinterpret_cast<float*>(e4_raw + ((128u - (smem_u32(e4_raw) & 127u)) & 127u));
  const uint32_t bar = smem_u32(sm + S::IN_WORDS);
  const OpGeom<float>& g = A.g;
  const int tid = threadIdx.x;
  const int tx = tid % BX, ty = (tid / BX) % BY, tz = tid / (BX * BY);
  const int nbx = (g.nx + BX - 1) / BX, nby = (g.ny + BY - 1) / BY;
  const int blk = blockIdx.x;
  const int x0 = (blk % nbx) * BX, y0 = ((blk / nbx) % nby) * BY, z0 = (blk / (nbx * nby)) * BZ;
  const int cx = x0 + tx, cy = y0 + ty, cz = z0 + tz;
  const bool hxm = cx > 0, hxp = cx + 1 < g.nx, hym = cy > 0, hyp = cy + 1 < g.ny, hzm = cz > 0, hzp = cz + 1 < g.nz;
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  pdl_launch_dependents();
  pdl_wait();
  if (tid == 0) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(S::IN_WORDS * 4)
                 : "memory");
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
        "%5}], [%6];" ::"r"(smem_u32(sm)),
        "l"(&mu), "r"(0), "r"(x0 - 1), "r"(y0 - 1), "r"(z0 - 1), "r"(bar)
        : "memory");
  }
  if (!__syncthreads_and(mbar_wait(bar, 0, err))) {
    if (tid == 0) mbar_wait(bar, 0, err);  // let the copy land (bounded) before the CTA leaves
    __syncthreads();
    return;
  }
  const float* me = sm + (((tz + 1) * PY + ty + 1) * PX + tx + 1) * SL;
  constexpr int DX = SL, DY = PX * SL, DZ = PY * PX * SL;  // neighbour offsets in words
  // element, gradient component and pre-mass sum as pairs of x-neighbouring points ([k][j][i / 2]):
  // the y- and z-contractions combine whole pairs with one packed FMA (Dhat entry in both halves)
  float2 U[4][4][2], ACC[4][4][2], G[4][4][2];
#define E4(a, k, j, i) ((i) & 1 ? a[k][j][(i) >> 1].y : a[k][j][(i) >> 1].x)
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float4 v = *reinterpret_cast<const float4*>(me + k * 16 + j * 4);
      U[k][j][0] = make_float2(v.x, v.y);
      U[k][j][1] = make_float2(v.z, v.w);
      ACC[k][j][0] = ACC[k][j][1] = make_float2(0.f, 0.f);
    }
  const float w0 = C::w(wO);
  const float cfx = g.Jf[0] / (g.J * w0), cfy = g.Jf[1] / (g.J * w0), cfz = g.Jf[2] / (g.J * w0);
  const float smx = g.sigma[0] - g.lift[0], smy = g.sigma[1] - g.lift[1], smz = g.sigma[2] - g.lift[2];
  const float sx = g.dxi[0] * g.dxi[0], sy = g.dxi[1] * g.dxi[1], sz = g.dxi[2] * g.dxi[2];
  const float2 dx2 = make_float2(sx, sx), dy2 = make_float2(sy, sy), dz2 = make_float2(sz, sz);
  // x: gradient component along the thread's lines, faces from the x-neighbours' lines, divergence.
  // Along a line the pairs multiply 2 x 2 blocks of Dhat: (y0, y1) = (D00, D11) (x0, x1) +
  // (D01, D10) (x1, x0) + (D02, D13) (x2, x3) + (D03, D12) (x3, x2), and likewise for (y2, y3).
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float2 sw[2] = {make_float2(U[k][j][0].y, U[k][j][0].x), make_float2(U[k][j][1].y, U[k][j][1].x)};
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        float2 a = __fmul2_rn(C::B(4 * q), U[k][j][0]);
        a = __ffma2_rn(C::B(4 * q + 1), sw[0], a);
        a = __ffma2_rn(C::B(4 * q + 2), U[k][j][1], a);
        a = __ffma2_rn(C::B(4 * q + 3), sw[1], a);
        G[k][j][q] = a;
      }
    }
  const E4Face fmx(-1.f, hxm, g.neumann & 1, g.dxi[0], g.lift[0], smx, cfx),
      fpx(1.f, hxp, (g.neumann >> 1) & 1, g.dxi[0], g.lift[0], smx, cfx);
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float r[4];
      ld4s(me - DX + k * 16 + j * 4, r);
      float ge = 0.f;
#pragma unroll
      for (int l = 0; l < 4; ++l) ge += C::DD(12 + l).x * r[l];
      G[k][j][0].x = fmx.apply(U[k][j][0].x, G[k][j][0].x, r[3], ge, ACC[k][j][0].x);
      ld4s(me + DX + k * 16 + j * 4, r);
      ge = 0.f;
#pragma unroll
      for (int l = 0; l < 4; ++l) ge += C::DD(l).x * r[l];
      G[k][j][1].y = fpx.apply(U[k][j][1].y, G[k][j][1].y, r[0], ge, ACC[k][j][1].y);
    }
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float2 sw[2] = {make_float2(G[k][j][0].y, G[k][j][0].x), make_float2(G[k][j][1].y, G[k][j][1].x)};
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        float2 a = __fmul2_rn(C::B(4 * q), G[k][j][0]);
        a = __ffma2_rn(C::B(4 * q + 1), sw[0], a);
        a = __ffma2_rn(C::B(4 * q + 2), G[k][j][1], a);
        a = __ffma2_rn(C::B(4 * q + 3), sw[1], a);
        ACC[k][j][q] = __ffma2_rn(dx2, a, ACC[k][j][q]);
      }
    }
  // y
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        float2 a = make_float2(0.f, 0.f);
#pragma unroll
        for (int l = 0; l < 4; ++l) {
          a = __ffma2_rn(C::DD(j * 4 + l), U[k][l][p], a);
        }
        G[k][j][p] = a;
      }
  {
    const E4Face fm(-1.f, hym, (g.neumann >> 2) & 1, g.dxi[1], g.lift[1], smy, cfy),
        fp(1.f, hyp, (g.neumann >> 3) & 1, g.dxi[1], g.lift[1], smy, cfy);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      float2 r[4][2];
#pragma unroll
      for (int l = 0; l < 4; ++l) ld4p(me - DY + k * 16 + l * 4, r[l]);
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        float2 ge = make_float2(0.f, 0.f);
#pragma unroll
        for (int l = 0; l < 4; ++l) {
          ge = __ffma2_rn(C::DD(12 + l), r[l][p], ge);
        }
        G[k][0][p] = fm.apply(U[k][0][p], G[k][0][p], r[3][p], ge, ACC[k][0][p]);
      }
#pragma unroll
      for (int l = 0; l < 4; ++l) ld4p(me + DY + k * 16 + l * 4, r[l]);
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        float2 ge = make_float2(0.f, 0.f);
#pragma unroll
        for (int l = 0; l < 4; ++l) {
          ge = __ffma2_rn(C::DD(l), r[l][p], ge);
        }
        G[k][3][p] = fp.apply(U[k][3][p], G[k][3][p], r[0][p], ge, ACC[k][3][p]);
      }
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        float2 a = make_float2(0.f, 0.f);
#pragma unroll
        for (int l = 0; l < 4; ++l) {
          a = __ffma2_rn(C::DD(j * 4 + l), G[k][l][p], a);
        }
        ACC[k][j][p] = __ffma2_rn(dy2, a, ACC[k][j][p]);
      }
  // z
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        float2 a = make_float2(0.f, 0.f);
#pragma unroll
        for (int l = 0; l < 4; ++l) {
          a = __ffma2_rn(C::DD(k * 4 + l), U[l][j][p], a);
        }
        G[k][j][p] = a;
      }
  {
    const E4Face fm(-1.f, hzm, (g.neumann >> 4) & 1, g.dxi[2], g.lift[2], smz, cfz),
        fp(1.f, hzp, (g.neumann >> 5) & 1, g.dxi[2], g.lift[2], smz, cfz);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float2 r[4][2];
#pragma unroll
      for (int l = 0; l < 4; ++l) ld4p(me - DZ + l * 16 + j * 4, r[l]);
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        float2 ge = make_float2(0.f, 0.f);
#pragma unroll
        for (int l = 0; l < 4; ++l) {
          ge = __ffma2_rn(C::DD(12 + l), r[l][p], ge);
        }
        G[0][j][p] = fm.apply(U[0][j][p], G[0][j][p], r[3][p], ge, ACC[0][j][p]);
      }
#pragma unroll
      for (int l = 0; l < 4; ++l) ld4p(me + DZ + l * 16 + j * 4, r[l]);
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        float2 ge = make_float2(0.f, 0.f);
#pragma unroll
        for (int l = 0; l < 4; ++l) {
          ge = __ffma2_rn(C::DD(l), r[l][p], ge);
        }
        G[3][j][p] = fp.apply(U[3][j][p], G[3][j][p], r[0][p], ge, ACC[3][j][p]);
      }
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        float2 a = make_float2(0.f, 0.f);
#pragma unroll
        for (int l = 0; l < 4; ++l) {
          a = __ffma2_rn(C::DD(k * 4 + l), G[l][j][p], a);
        }
        ACC[k][j][p] = __ffma2_rn(dz2, a, ACC[k][j][p]);
      }
  // A u = -M acc (+ diag u); b - A u with b
  const bool valid = cx < g.nx && cy < g.ny && cz < g.nz;
  const int64_t e = valid ? ((int64_t)cz * g.ny + cy) * g.nx + cx : 0;
  const float2 w01 = make_float2(C::w(wO), C::w(wO + 1)), w10 = make_float2(w01.y, w01.x);  // weights are symmetric
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float m = -g.J * (j == 0 || j == 3 ? w01.x : w01.y) * (k == 0 || k == 3 ? w01.x : w01.y);
      ACC[k][j][0] = __fmul2_rn(__fmul2_rn(make_float2(m, m), w01), ACC[k][j][0]);
      ACC[k][j][1] = __fmul2_rn(__fmul2_rn(make_float2(m, m), w10), ACC[k][j][1]);
    }
  if (A.diag && valid) {
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      float dl[4];
      row4_g(A.diag + e * 64 + q * 4, dl);
#pragma unroll
      for (int i = 0; i < 4; ++i) E4(ACC, q >> 2, q & 3, i) += dl[i] * E4(U, q >> 2, q & 3, i);
    }
  }
  if (A.b && valid) {
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      float bl[4];
      row4_g(A.b + e * 64 + q * 4, bl);
#pragma unroll
      for (int i = 0; i < 4; ++i) E4(ACC, q >> 2, q & 3, i) = bl[i] - E4(ACC, q >> 2, q & 3, i);
    }
  }
#undef E4
  __syncthreads();  // every read of the staged box is done: its first slots take the result
  float* o = sm + tid * SL;
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int j = 0; j < 4; ++j)
      *reinterpret_cast<float4*>(o + k * 16 + j * 4) =
          make_float4(ACC[k][j][0].x, ACC[k][j][0].y, ACC[k][j][1].x, ACC[k][j][1].y);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();
  if (tid == 0) {
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3, %4}], [%5];" ::"l"(&mo),
                 "r"(0), "r"(x0), "r"(y0), "r"(z0), "r"(smem_u32(sm))
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
  }
}

// Tensor maps of the element-per-thread apply: u (or the result) as a 4-D tensor [nz][ny][nx][64]
// read or written in boxes of (BX, BY, BZ) elements of 68 words (the 4 words past an element are
// outside the tensor: zeros on loads, not written on stores). No swizzle.
bool e4_map(CUtensorMap* m, const float* base, int nx, int ny, int nz, int bx, int by, int bz) {
  auto fn = tensor_map_encoder();
  if (!fn) return false;
  const cuuint64_t dims[4] = {64, (cuuint64_t)nx, (cuuint64_t)ny, (cuuint64_t)nz};
  const cuuint64_t strides[3] = {256, 256ull * nx, 256ull * nx * ny};
  const cuuint32_t box[4] = {(cuuint32_t)kE4Slot, (cuuint32_t)bx, (cuuint32_t)by, (cuuint32_t)bz};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, (void*)base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
         CUDA_SUCCESS;
}

// False (nothing launched) where the element-per-thread kernel cannot run this apply: subdomain
// output, buffers not 16-byte aligned, no error flag, or a tensor map the driver does not encode.
template <int BX, int BY, int BZ>
bool launch_elem4(const ApplyArgs<float>& A, int* err, cudaStream_t s) {
  using S = E4Shape<BX, BY, BZ>;
  auto kern = apply_elem4_kernel<BX, BY, BZ>;
  const OpGeom<float>& g = A.g;
  if (A.rS || !err || (((uintptr_t)A.u | (uintptr_t)A.out) & 15)) return false;
  CUtensorMap mu, mo;
  if (!e4_map(&mu, A.u, g.nx, g.ny, g.nz, BX + 2, BY + 2, BZ + 2) || !e4_map(&mo, A.out, g.nx, g.ny, g.nz, BX, BY, BZ))
    return false;
  {
    static std::mutex mu_attr;
    static std::set<int> done;
    int dev = 0;
    DG_CUDA(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lk(mu_attr);
    if (!done.count(dev)) {
      DG_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, S::SMEM));
      done.insert(dev);
    }
  }
  const int nb = ((g.nx + BX - 1) / BX) * ((g.ny + BY - 1) / BY) * ((g.nz + BZ - 1) / BZ);
  launch_pdl(kern, dim3(nb), dim3(S::THREADS), (size_t)S::SMEM, s, A, mu, mo, err);
  return true;
}

// What bounds it: in FP64 the FP64 pipe (about 12.5 N + 40 operations per point and direction line of
// N, two thirds of them the even-odd contractions, at 75-85 % of the probed 0.6 T/s); in FP32 the L1
// data pipe (81 % busy at N = 8, issue slots 71 %, DRAM 26 %). Measured, 48^3 elements at N = 8: FP32
// 370 -> 201 us; 37 x 41 x 29 at N = 7: FP32 162 -> 80 us; 43^3 at N = 9: FP64
// 9.71 -> 5.67 ms; 16^3 at N = 6: FP64 128 -> 92 us (against one x-line per thread with the y- and
// z-contractions read from shared memory, and in FP32 against blocks of such lines).
template <int N, typename T, int EPB>
__global__ void __launch_bounds__(EPB* N* N) apply_dir_kernel(const ApplyArgs<T> A) {
  extern __shared__ __align__(16) unsigned char dir_smem[];
  apply_dir_block<N, T, EPB, DirTab<N, T>, true>(A, blockIdx.x, reinterpret_cast<T*>(dir_smem));
}

// 2^3 elements at N = 6, FP64: 18.7 us a launch one direction after the other -> 8.3 us; 8^3 at N = 6:
// 24.8 -> 18.6 us; FP32 2^3 at N = 8: 6.4 -> 5.0 us.
template <int N, typename T, int EPB>
__global__ void __launch_bounds__(3 * EPB * N * N) apply_par_kernel(const ApplyArgs<T> A) {
  extern __shared__ __align__(16) unsigned char dir_smem[];
  apply_par_block<N, T, EPB, DirTab<N, T>, true>(A, blockIdx.x, reinterpret_cast<T*>(dir_smem));
}

// Brick of at most cap elements for a grid: fewest (bricks x cost of one), where a brick costs its
// elements plus a part for every face whose neighbour is read from global memory.
template <typename T>
int choose_brick(ApplyArgs<T>& A, int cap) {
  const OpGeom<T>& g = A.g;
  double best = 1e300;
  int nb = 0;
  for (int sx = 0; (1 << sx) <= cap; ++sx)
    for (int sy = 0; (1 << (sx + sy)) <= cap; ++sy) {
      const int bx = 1 << sx, by = 1 << sy;
      if ((sx && bx / 2 >= g.nx) || (sy && by / 2 >= g.ny)) continue;
      for (int bz = 1; bx * by * bz <= cap && bz <= g.nz; ++bz) {
        const int qx = (g.nx + bx - 1) / bx, qy = (g.ny + by - 1) / by, qz = (g.nz + bz - 1) / bz;
        const double n = (double)qx * qy * qz;
        const double cost = n * (bx * by * bz + 0.15 * 2 * (bx * by + by * bz + bx * bz) + 0.1 * cap);
        if (cost < best) {
          best = cost;
          nb = qx * qy * qz;
          A.bsx = sx;
          A.bsy = sy;
          A.bz = bz;
          A.nbx = qx;
          A.nby = qy;
        }
      }
    }
  return nb;
}

// One of the two kernels (PAR: directions side by side) with bricks of at most EPB elements.
template <int N, typename T, int EPB, bool PAR>
void launch_dir(ApplyArgs<T> A, cudaStream_t s) {
  using S = typename std::conditional<PAR, ParShape<N, T, EPB>, DirShape<N, T, EPB>>::type;
  static_assert(S::SMEM <= 200 * 1024, "brick must fit in shared memory");
  void (*kern)(const ApplyArgs<T>);
  if constexpr (PAR) kern = apply_par_kernel<N, T, EPB>;
  else kern = apply_dir_kernel<N, T, EPB>;
  if constexpr (S::SMEM > 40 * 1024) {  // with the static tables, above the default 48 KiB
    static std::mutex mu;
    static std::set<int> done;
    int dev = 0;
    DG_CUDA(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lk(mu);
    if (!done.count(dev)) {
      DG_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, S::SMEM));
      done.insert(dev);
    }
  }
  const int nb = choose_brick(A, EPB);
  launch_pdl(kern, dim3(nb), dim3(S::THREADS), (size_t)S::SMEM, s, A);
}

// Elements per CTA: few (a warp or two), middle, many; p with the directions side by side.
template <int N>
struct DirEpb;
template <> struct DirEpb<2> { static constexpr int s = 8, m = 32, l = 64, p = 8; };
template <> struct DirEpb<3> { static constexpr int s = 4, m = 16, l = 32, p = 4; };
template <> struct DirEpb<4> { static constexpr int s = 2, m = 16, l = 32, p = 2; };
template <> struct DirEpb<5> { static constexpr int s = 2, m = 8, l = 16, p = 1; };
template <> struct DirEpb<6> { static constexpr int s = 2, m = 8, l = 12, p = 1; };
template <> struct DirEpb<7> { static constexpr int s = 1, m = 4, l = 8, p = 1; };
template <> struct DirEpb<8> { static constexpr int s = 1, m = 4, l = 8, p = 1; };
template <> struct DirEpb<9> { static constexpr int s = 1, m = 4, l = 6, p = 1; };
template <> struct DirEpb<10> { static constexpr int s = 1, m = 2, l = 4, p = 1; };

// Launch shapes: 1, 2, 3 few / middle / many elements per CTA, 4 the directions side by side, 7 the
// element-per-thread kernel (FP32, N = 4, plain output); 0 picks one of them by grid size: side by side
// while the lines of one direction leave a scheduler of every SM without a warp (152 SMs x 4 warps;
// FP64 at N = 8, 8^3 elements, just above: 33.7 us in bricks, 36.4 side by side), else the middle shape
// once it gives every SM two bricks. The autotuner times them per level.
template <int N, typename T>
void launch_apply_n(const OpGeom<T>& g, const Pair<T>* wf, const T* u, const T* diag, const T* b, T* out,
                    const SubdomainOut& so, int variant, int* err, cudaStream_t s) {
  const int E = g.nx * g.ny * g.nz;
  if (E == 0) return;
  constexpr unsigned a = LineVec<N, T>::w - 1;  // lines move in vectors of this many bytes
  DG_REQUIRE(!(((uintptr_t)u | (uintptr_t)diag | (uintptr_t)b | (uintptr_t)out | (uintptr_t)so.rS) & a),
             "DG apply vectors must be aligned to " + std::to_string(a + 1) + " bytes");
  using DE = DirEpb<N>;
  const ApplyArgs<T> A{g, wf, u, diag, b, out, E, static_cast<T*>(so.rS), so.ld, so.ov, so.rec};
  if constexpr (N == 4 && std::is_same<T, float>::value) {
    if (variant == 7 && !so.rS && launch_elem4<8, 4, 4>(A, err, s)) return;
  }
  if (variant < 1 || variant > 4)
    variant = (int64_t)E * N * N <= 152 * 128 ? 4 : ((E + DE::m - 1) / DE::m >= 2 * 152 ? 2 : 1);
  if (variant == 1) launch_dir<N, T, DE::s, false>(A, s);
  else if (variant == 2) launch_dir<N, T, DE::m, false>(A, s);
  else if (variant == 3) launch_dir<N, T, DE::l, false>(A, s);
  else launch_dir<N, T, DE::p, true>(A, s);
}

// ------------------------------------------------------------------ fused coarse-level smoother
//
// On coarse levels (tens of elements) each of the three kernels of a Schwarz step is limited by its
// own latency, not by work. This kernel runs all steps of one smoothing call in a single
// cooperative launch: residual into r_S (or the gather of b when u = 0), the subdomain solves as a
// CUDA-core GEMM over (class, 16-row) units, the weighted scatter into u, each phase separated by a
// grid-wide barrier. Data written by other CTAs inside the kernel are read through L2 only.

constexpr uint32_t kBarrierPolls = 1u << 22;  // polls before a barrier wait gives up

// Grid-wide barrier over a cooperative launch (all CTAs co-resident). Returns false, with the error
// flag set, if the wait gave up; the caller then leaves the kernel.
__device__ __forceinline__ bool grid_barrier(unsigned* bar, unsigned n_blocks, int* err) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    volatile unsigned* gen = bar + 1;
    const unsigned g = *gen;
    __threadfence();
    if (atomicAdd(bar, 1u) == n_blocks - 1) {
      atomicExch(bar, 0u);
      __threadfence();
      atomicAdd(bar + 1, 1u);
    } else {
      uint32_t polls = 0;
      while (*gen == g) {
        if (++polls > kBarrierPolls) {
          atomicExch(err, 1);
          ok = 0;
          break;
        }
        __nanosleep(64);
      }
    }
    __threadfence();
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// Rows row0 .. row0 + 15 of du_S for every column of one class: 128 threads = 16 rows x 8 K-groups
// of 16; the class's columns are staged in shared memory 8 at a time in 128-wide K tiles; the 8
// partial sums of each output are added in a fixed order.
__device__ __forceinline__ void coarse_gemm_unit(const float* __restrict__ invm, int ld, const float* X, float* Y,
                                                 int4 unit, float alpha) {
  __shared__ __align__(16) float sx[8][136];  // 128 K values per column, one pad word per 16
  __shared__ float red[8][16][9];
  const int tid = threadIdx.x;
  const int kg = tid & 7, r = tid >> 3;  // r < 16 for the first 128 threads
  const int cls = unit.x, row0 = unit.y, col0 = unit.z, ncols = unit.w;
  const float* arow = invm + ((size_t)cls * ld + row0 + r) * ld;
  for (int c0 = 0; c0 < ncols; c0 += 8) {
    const int nc = min(8, ncols - c0);
    float acc[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[c] = 0.0f;
    for (int kt = 0; kt < ld; kt += 128) {
      __syncthreads();  // sx and red of the previous round are consumed
      for (int q = tid; q < 8 * 128; q += blockDim.x) {
        const int c = q >> 7, kk = q & 127;
        sx[c][kk + (kk >> 4)] = (c < nc && kt + kk < ld) ? __ldcg(X + (size_t)(col0 + c0 + c) * ld + kt + kk) : 0.0f;
      }
      __syncthreads();
      const int kb = kt + kg * 16;
      if (tid < 128 && kb < ld) {
        float a[16];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float4 v = __ldg(reinterpret_cast<const float4*>(arow + kb) + q);
          a[4 * q] = v.x;
          a[4 * q + 1] = v.y;
          a[4 * q + 2] = v.z;
          a[4 * q + 3] = v.w;
        }
#pragma unroll
        for (int i = 0; i < 16; ++i)
#pragma unroll
          for (int c = 0; c < 8; ++c) acc[c] += a[i] * sx[c][kg * 17 + i];
      }
    }
    if (tid < 128) {
#pragma unroll
      for (int c = 0; c < 8; ++c) red[kg][r][c] = acc[c];
    }
    __syncthreads();
    if (tid < 128) {
      const int rr = tid >> 3, cc = tid & 7;
      if (cc < nc) {
        float sum = 0.0f;
#pragma unroll
        for (int g = 0; g < 8; ++g) sum += red[g][rr][cc];
        Y[(size_t)(col0 + c0 + cc) * ld + row0 + rr] = alpha * sum;
      }
    }
  }
}

template <int N, int EPB>
__global__ void __launch_bounds__(EPB* N* N) coarse_smooth_kernel(const CoarseArgs a) {
  // a wait of an earlier launch gave up and the host has not read the flag yet: skip the work
  // (its inputs are incomplete) instead of waiting again
  if (*reinterpret_cast<volatile int*>(a.err) != 0) return;
  constexpr int N3 = N * N * N;
  extern __shared__ __align__(16) float coarse_smem[];
  const unsigned G = gridDim.x + (unsigned)a.stall;
  const int E = a.ap.E;
  const int nblk = a.n_bricks;
  for (int it = 0; it < a.iterations; ++it) {
    if (it == 0 && a.u_zero) {
      for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < E * N3; t += gridDim.x * blockDim.x)
        gather_point<N, float>(a.sg, a.ap.rec, __ldg(a.ap.b + t), a.ap.rS, t / N3, t % N3);
    } else {
      for (int blk = blockIdx.x; blk < nblk; blk += gridDim.x) {
        __syncthreads();  // the previous group is done with the shared blocks
        apply_dir_block<N, float, EPB, DirTab<N, float>, false, true>(a.ap, blk, coarse_smem);
      }
    }
    if (!grid_barrier(a.bar, G, a.err)) return;
    for (int un = blockIdx.x; un < a.n_units; un += gridDim.x)
      coarse_gemm_unit(a.invm, a.sg.ld, a.ap.rS, a.duS, a.units[un], a.alpha);
    if (!grid_barrier(a.bar, G, a.err)) return;
    // du_S and u were written by other CTAs of this kernel: read through L2 only
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < E * N3; t += gridDim.x * blockDim.x) {
      int64_t idx[7];
      int col[7];
      float w[7];
      scatter_look_up<N, 7, float>(a.sg, a.ap.rec, a.shares, t / N3, t % N3, idx, col, w);
      float acc = 0.0f;
#pragma unroll
      for (int sl = 0; sl < 7; ++sl)
        if (idx[sl] >= 0) acc += w[sl] * __ldcg(a.duS + idx[sl]);
      float* up = const_cast<float*>(a.ap.u) + t;
      *up = __ldcg(up) + acc;
    }
    if (it + 1 < a.iterations && !grid_barrier(a.bar, G, a.err)) return;
  }
}

// threads per CTA: whole elements, at least the 128 the GEMM units use
template <int N>
struct CoarseShape {
  static constexpr int epb = (128 + N * N - 1) / (N * N);
  static constexpr int threads = epb * N * N;
};

template <int N>
void launch_coarse_n(CoarseArgs a, cudaStream_t s) {
  using CS = CoarseShape<N>;
  constexpr int SMEM = DirShape<N, float, CS::epb>::SMEM;
  static_assert(SMEM <= 40 * 1024, "brick and GEMM staging within the default shared memory");
  a.n_bricks = choose_brick(a.ap, CS::epb);
  static_assert(CS::threads >= 128, "GEMM units need 128 threads");
  int dev = 0, sms = 0, per_sm = 0;
  DG_CUDA(cudaGetDevice(&dev));
  DG_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  DG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, coarse_smooth_kernel<N, CS::epb>, CS::threads, SMEM));
  DG_REQUIRE(per_sm >= 1, "fused coarse smoother does not fit on an SM");
  const int E = a.ap.E;
  const int work = std::max(E, a.n_units);
  const int G = std::min(work, per_sm * sms);
  DG_CUDA(cudaMemsetAsync(a.bar, 0, 2 * sizeof(unsigned), s));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(G);
  cfg.blockDim = dim3(CS::threads);
  cfg.dynamicSmemBytes = SMEM;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  DG_CUDA(cudaLaunchKernelEx(&cfg, coarse_smooth_kernel<N, CS::epb>, a));
}

}  // namespace

void upload_operator_tables() {
  static std::mutex mu;
  static std::set<int> done;
  int dev = 0;
  DG_CUDA(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lk(mu);
  if (done.count(dev)) return;
  std::vector<double> W(kWTab);
  std::vector<float> Wlo32(kWTab);
  for (int N = 2; N <= DG_MAX_N; ++N) {
    const LglTables t = make_lgl(N);
    for (int l = 0; l < N; ++l) {
      W[wtab_off(N) + l] = t.w[l];
      Wlo32[wtab_off(N) + l] = (float)(t.w[l] - (float)t.w[l]);
    }
  }
  const LglTables t4 = make_lgl(4);
  const std::vector<float> D4(t4.D, t4.D + 16), W32(W.begin(), W.end());
  std::vector<double2> PQ(kDirPairs), QP(kDirPairs);
  std::vector<float2> PQ32(kDirPairs), QP32(kDirPairs);
  std::vector<double> V(kDirVec);
  for (int N = 2; N <= DG_MAX_N; ++N) {
    const LglTables t = make_lgl(N);
    const int h = N / 2, po = dir_pair_off(N), vo = dir_vec_off(N);
    for (int i = 0; i < h; ++i)
      for (int l = 0; l < h; ++l) {
        const int m = i * N + l, n = i * N + N - 1 - l;  // each sum rounded once
        const double p = (double)((long double)t.D[m] - t.D[n] + ((long double)t.D_lo[m] - t.D_lo[n]));
        const double q = (double)((long double)t.D[m] + t.D[n] + ((long double)t.D_lo[m] + t.D_lo[n]));
        const int at = po + i * h + l;
        PQ[at] = make_double2(p, q);
        QP[at] = make_double2(q, p);
        PQ32[at] = make_float2((float)p, (float)q);
        QP32[at] = make_float2((float)q, (float)p);
      }
    for (int l = 0; l < N; ++l) V[vo + l] = 2.0 * t.D[(N - 1) * N + l];
    for (int l = 0; l < h && N % 2; ++l) {
      V[vo + N + l] = 2.0 * t.D[l * N + h];
      V[vo + N + h + l] = t.D[h * N + l];
    }
  }
  const std::vector<float> V32(V.begin(), V.end());
  DG_CUDA(cudaMemcpyToSymbol(cPQ64, PQ.data(), sizeof(double2) * kDirPairs));
  DG_CUDA(cudaMemcpyToSymbol(cQP64, QP.data(), sizeof(double2) * kDirPairs));
  DG_CUDA(cudaMemcpyToSymbol(cPQ32, PQ32.data(), sizeof(float2) * kDirPairs));
  DG_CUDA(cudaMemcpyToSymbol(cQP32, QP32.data(), sizeof(float2) * kDirPairs));
  DG_CUDA(cudaMemcpyToSymbol(cV64, V.data(), sizeof(double) * kDirVec));
  DG_CUDA(cudaMemcpyToSymbol(cV32, V32.data(), sizeof(float) * kDirVec));
  float2 DD4[16], B4[8];
  for (int o = 0; o < 16; ++o) DD4[o] = make_float2(D4[o], D4[o]);
  for (int q = 0; q < 4; ++q) {  // output pair q / 2, input pair q % 2
    const float* d = &D4[q / 2 * 8 + q % 2 * 2];
    B4[2 * q] = make_float2(d[0], d[5]);
    B4[2 * q + 1] = make_float2(d[1], d[4]);
  }
  DG_CUDA(cudaMemcpyToSymbol(cDD4, DD4, sizeof(DD4)));
  DG_CUDA(cudaMemcpyToSymbol(cB4, B4, sizeof(B4)));
  DG_CUDA(cudaMemcpyToSymbol(cW64, W.data(), sizeof(double) * kWTab));
  DG_CUDA(cudaMemcpyToSymbol(cW32, W32.data(), sizeof(float) * kWTab));
  DG_CUDA(cudaMemcpyToSymbol(cWlo32, Wlo32.data(), sizeof(float) * kWTab));
  done.insert(dev);
}

template <typename T>
void launch_apply(int N, const OpGeom<T>& g, const Pair<T>* wf, const T* u, const T* diag, const T* b, T* out,
                  cudaStream_t s, const SubdomainOut* so_ptr, int variant, int* err) {
  const SubdomainOut so = so_ptr ? *so_ptr : SubdomainOut{};
  switch (N) {
    case 2: launch_apply_n<2, T>(g, wf, u, diag, b, out, so, variant, err, s); break;
    case 3: launch_apply_n<3, T>(g, wf, u, diag, b, out, so, variant, err, s); break;
    case 4: launch_apply_n<4, T>(g, wf, u, diag, b, out, so, variant, err, s); break;
    case 5: launch_apply_n<5, T>(g, wf, u, diag, b, out, so, variant, err, s); break;
    case 6: launch_apply_n<6, T>(g, wf, u, diag, b, out, so, variant, err, s); break;
    case 7: launch_apply_n<7, T>(g, wf, u, diag, b, out, so, variant, err, s); break;
    case 8: launch_apply_n<8, T>(g, wf, u, diag, b, out, so, variant, err, s); break;
    case 9: launch_apply_n<9, T>(g, wf, u, diag, b, out, so, variant, err, s); break;
    case 10: launch_apply_n<10, T>(g, wf, u, diag, b, out, so, variant, err, s); break;
    default: fail(DG_ERR_INVALID_ARG, "unsupported N");
  }
  DG_LAUNCHED(1);
}

int apply_bricks(int N, int variant, int E) {
  constexpr int m[] = {DirEpb<2>::m, DirEpb<3>::m, DirEpb<4>::m, DirEpb<5>::m, DirEpb<6>::m, DirEpb<7>::m,
                       DirEpb<8>::m, DirEpb<9>::m, DirEpb<10>::m};
  constexpr int l[] = {DirEpb<2>::l, DirEpb<3>::l, DirEpb<4>::l, DirEpb<5>::l, DirEpb<6>::l, DirEpb<7>::l,
                       DirEpb<8>::l, DirEpb<9>::l, DirEpb<10>::l};
  return E / (variant == 2 ? m : l)[N - 2];
}

template void launch_apply<double>(int, const OpGeom<double>&, const double2*, const double*, const double*,
                                   const double*, double*, cudaStream_t, const SubdomainOut*, int, int*);
template void launch_apply<float>(int, const OpGeom<float>&, const float2*, const float*, const float*, const float*,
                                  float*, cudaStream_t, const SubdomainOut*, int, int*);

// static shared memory of the fused kernel stays within 48 KiB up to N = 8
bool coarse_smooth_available(int N) { return N >= 2 && N <= 8; }

void launch_coarse_smooth(int N, const CoarseArgs& a, cudaStream_t s) {
  DG_REQUIRE(a.sg.ld % 16 == 0, "fused coarse smoother needs a 16-aligned subdomain stride");
  switch (N) {
    case 2: launch_coarse_n<2>(a, s); break;
    case 3: launch_coarse_n<3>(a, s); break;
    case 4: launch_coarse_n<4>(a, s); break;
    case 5: launch_coarse_n<5>(a, s); break;
    case 6: launch_coarse_n<6>(a, s); break;
    case 7: launch_coarse_n<7>(a, s); break;
    case 8: launch_coarse_n<8>(a, s); break;
    default: fail(DG_ERR_INVALID_ARG, "fused coarse smoother supports N <= 8");
  }
  DG_LAUNCHED(1);
}


// Diagonal of the LGL mass matrix, M = J w_i w_j w_k (Eq. massmat with collocation quadrature).
template <typename T>
__global__ void mass_kernel(int N, T J, const T* __restrict__ w, int64_t ndof, T* __restrict__ mass) {
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= ndof) return;
  int p = (int)(t % (N * N * N));
  int i = p % N, j = (p / N) % N, k = p / (N * N);
  mass[t] = J * w[i] * w[j] * w[k];
}

template <typename T>
void launch_mass_diag(int N, const OpGeom<T>& g, const T* w, int64_t ndof, T* mass, cudaStream_t s) {
  if (ndof == 0) return;
  mass_kernel<T><<<(unsigned)((ndof + 255) / 256), 256, 0, s>>>(N, g.J, w, ndof, mass);
  DG_LAUNCHED(1);
}
template void launch_mass_diag<double>(int, const OpGeom<double>&, const double*, int64_t, double*, cudaStream_t);
template void launch_mass_diag<float>(int, const OpGeom<float>&, const float*, int64_t, float*, cudaStream_t);

__global__ void coords_kernel(int N, int nx, int ny, double lx, double ly, double lz, double hx, double hy, double hz,
                              const double* __restrict__ x1, int64_t ndof, double* X, double* Y, double* Z) {
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= ndof) return;
  const int N3 = N * N * N;
  int64_t e = t / N3;
  int p = (int)(t - e * N3);
  int i = p % N, j = (p / N) % N, k = p / (N * N);
  int ex = (int)(e % nx), ey = (int)((e / nx) % ny), ez = (int)(e / ((int64_t)nx * ny));
  X[t] = lx + hx * (ex + 0.5 * (x1[i] + 1.0));
  Y[t] = ly + hy * (ey + 0.5 * (x1[j] + 1.0));
  Z[t] = lz + hz * (ez + 0.5 * (x1[k] + 1.0));
}

void launch_node_coords(int N, const int n[3], const double lower[3], const double h[3], const double* x1, double* X,
                        double* Y, double* Z, cudaStream_t s) {
  int64_t ndof = (int64_t)n[0] * n[1] * n[2] * N * N * N;
  coords_kernel<<<(unsigned)((ndof + 255) / 256), 256, 0, s>>>(N, n[0], n[1], lower[0], lower[1], lower[2], h[0], h[1],
                                                               h[2], x1, ndof, X, Y, Z);
  DG_LAUNCHED(1);
}

}  // namespace dg
