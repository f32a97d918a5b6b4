// Direction-by-direction DG apply: the device function behind apply_dir_kernel and the fused
// coarse-level smoother (dg_apply.cu, which also holds the constant tables).
//
// A u = -w_i w_j w_k sum_d J (2/h_d)^2 [ Dhat v_d + face terms ], every term of direction d involving only the
// N points of one line along d and, at its two ends, the neighbours' value and normal derivative.
// A thread owns one line per direction and does everything of that direction in registers: gradient
// along the line, lifting and fluxes at the two ends, divergence. Only three things pass through
// shared memory: the element (written once as x-lines, read once as y-lines and once as z-lines),
// the sum over directions (the same way back), and the two end values per line that neighbours
// exchange (4 words written, 4 read). That is about 7 + 24/N shared words per point, where a kernel
// that keeps x-lines and reads the y- and z-contractions from shared memory needs 4 N.
//
// Dhat is centro-antisymmetric (the LGL points are symmetric), so both contractions run on the even
// and odd parts of the line: with o_l = u_l - u_{N-1-l}, e_l = u_l + u_{N-1-l} (l < h = N/2)
//   S_i = (Du)_i + (Du)_{N-1-i} = sum_l P_il o_l,         P_il = D_il - D_{i,N-1-l},
//   T_i = (Du)_i - (Du)_{N-1-i} = sum_l Q_il e_l (+ 2 D_im u_m for odd N, m = h), Q_il = D_il + D_{i,N-1-l},
// half the multiply-adds of the plain product, and (S, T) of v are the odd-even input of the second
// contraction as they stand (e^v = S, o^v = T). In FP32 the two sums are one packed two-wide FMA.
//
// Line units: ghat = Dhat u, lambda = 1 / (2 w_0), p = (C N^2 - 1 / w_0) / w_0; at the ends (0: lower,
// 1: upper) with the exterior value uE and derivative gE,
//   vhat_0 = ghat_0 - lambda (uE_0 - u_0),  vhat_{N-1} = ghat_{N-1} + lambda (uE_1 - u_{N-1}),
//   face terms  -lambda (gE_0 - ghat_0) + p/2 (uE_0 - u_0)  and  lambda (gE_1 - ghat_{N-1}) + p/2 (uE_1 - u_{N-1}).
//
// A CTA owns a brick of at most EPB elements (bx, by powers of two); faces inside the brick
// exchange through shared memory, the others read the neighbour's lines from global memory (L2) and
// contract them with one row of Dhat.
#pragma once

#include "bounds.cuh"
#include "internal.h"
#include "lines.cuh"
#include "pdl.cuh"
#include "schwarz_dev.cuh"

namespace dg {

// Constant tables of every order (filled in dg_apply.cu): per N the pairs (P_il, Q_il) [h][h], the
// pairs (Q_il, P_il) [h][h], the last row 2 D_{N-1,l} [N]; for odd N also 2 D_im and D_ml [h].
constexpr int dir_h(int N) { return N / 2; }
constexpr int dir_pairs(int N) { return N / 2 * (N / 2); }
constexpr int dir_pair_off(int N) { return N <= 2 ? 0 : dir_pair_off(N - 1) + dir_pairs(N - 1); }
constexpr int dir_vec_off(int N) { return N <= 2 ? 0 : dir_vec_off(N - 1) + (N - 1) + 2 * ((N - 1) / 2); }
constexpr int kDirPairs = dir_pair_off(DG_MAX_N + 1), kDirVec = dir_vec_off(DG_MAX_N + 1);

__device__ __forceinline__ float2 pair_fma(float2 c, float2 x, float2 y) { return __ffma2_rn(c, x, y); }
__device__ __forceinline__ float2 pair_mul(float2 c, float2 x) { return __fmul2_rn(c, x); }
__device__ __forceinline__ double2 pair_fma(double2 c, double2 x, double2 y) {
  return make_double2(fma(c.x, x.x, y.x), fma(c.y, x.y, y.y));
}
__device__ __forceinline__ double2 pair_mul(double2 c, double2 x) { return make_double2(c.x * x.x, c.y * x.y); }

template <typename T>
struct PairOf;
template <>
struct PairOf<float> {
  using V = float2;
  static __device__ __forceinline__ V make(float a, float b) { return make_float2(a, b); }
};
template <>
struct PairOf<double> {
  using V = double2;
  static __device__ __forceinline__ V make(double a, double b) { return make_double2(a, b); }
};

// Shared-memory shape. The element block is [k][j][i] with planes padded so that every lane order
// used (x-lines, (k, i) and (j, i) columns, elements back to back) walks consecutive banks:
// P = N (mod the words of a bank sweep), and so element stride = N^2 (mod it).
template <int N, typename T, int EPB>
struct DirShape {
  static constexpr int N2 = N * N, sweep = 128 / (int)sizeof(T);
  static constexpr int P = N2 + ((N - N2) % sweep + sweep) % sweep;
  static constexpr int R = N * P;
  static constexpr int THREADS = EPB * N2;
  static constexpr int XW = EPB * N2;  // words of one exchange array
  static constexpr int SMEM = (2 * EPB * R + 12 * XW) * (int)sizeof(T);
};

// CT: the constant tables (PQ(i), QP(i) pairs, vec(i)) of one precision.
template <int N, typename T, typename CT>
struct DirLine {
  using V2 = typename PairOf<T>::V;
  static constexpr int h = N / 2, H = h > 0 ? h : 1;
  static constexpr bool odd = N % 2 == 1;
  static constexpr int po = dir_pair_off(N), vo = dir_vec_off(N);
  V2 st[H];   // (S_i, T_i)
  T m;        // middle value (odd N)

  __device__ __forceinline__ static T last_row2(int l) { return CT::vec(vo + l); }  // 2 D_{N-1,l}

  // (S, T) of Dhat u
  __device__ __forceinline__ void gradient(const T (&u)[N]) {
    V2 x[H];
#pragma unroll
    for (int l = 0; l < h; ++l) x[l] = PairOf<T>::make(u[l] - u[N - 1 - l], u[l] + u[N - 1 - l]);
#pragma unroll
    for (int i = 0; i < h; ++i) {
      V2 a = pair_mul(CT::PQ(po + i * h), x[0]);
#pragma unroll
      for (int l = 1; l < h; ++l) a = pair_fma(CT::PQ(po + i * h + l), x[l], a);
      if constexpr (odd) a.y += CT::vec(vo + N + i) * u[h];
      st[i] = a;
    }
    m = T(0);
    if constexpr (odd) {
      m = CT::vec(vo + N + h) * x[0].x;
#pragma unroll
      for (int l = 1; l < h; ++l) m += CT::vec(vo + N + h + l) * x[l].x;
    }
  }

  // twice the derivative at the lower and upper end, before lifting
  __device__ __forceinline__ T lower2() const { return st[0].x + st[0].y; }
  __device__ __forceinline__ T upper2() const { return st[0].x - st[0].y; }

  // Lifting into (S, T) with the interior and exterior values lo, hi, u0, u1 at the ends and twice the
  // exterior derivatives G0, G1, then acc = 2 (Dhat vhat + face terms) (FIRST), or acc += q times it;
  // q = (h_x / h_d)^2, and J (2/h_x)^2 / 2 comes with the weights. The face terms join after the even and odd parts
  // are recombined, the larger last: they are the largest terms of the operator, and through S and T each
  // end would carry the other's rounding.
  template <bool FIRST>
  __device__ __forceinline__ void divergence(T lo, T hi, T u0, T G0, T u1, T G1, T lam, T pen, T q, T (&acc)[N]) {
    const T j0 = u0 - lo, j1 = u1 - hi, d0 = G0 - lower2(), d1 = G1 - upper2();
    st[0].x += lam * (j1 - j0);
    st[0].y -= lam * (j0 + j1);
    V2 r[H];  // (T, S) of Dhat vhat
#pragma unroll
    for (int i = 0; i < h; ++i) {
      V2 a = pair_mul(CT::QP(po + i * h), st[0]);
#pragma unroll
      for (int l = 1; l < h; ++l) a = pair_fma(CT::QP(po + i * h + l), st[l], a);
      if constexpr (odd) a.x += CT::vec(vo + N + i) * m;
      r[i] = a;
    }
#pragma unroll
    for (int i = 0; i < h; ++i) {
      T a = r[i].y + r[i].x, b = r[i].y - r[i].x;
      if (i == 0) {
        a -= lam * d0;
        b += lam * d1;
        a += pen * j0;
        b += pen * j1;
      }
      acc[i] = FIRST ? a : acc[i] + q * a;
      acc[N - 1 - i] = FIRST ? b : acc[N - 1 - i] + q * b;
    }
    if constexpr (odd) {
      T mid = CT::vec(vo + N + h) * st[0].y;
#pragma unroll
      for (int l = 1; l < h; ++l) mid += CT::vec(vo + N + h + l) * st[l].y;
      acc[h] = FIRST ? T(2) * mid : acc[h] + (T(2) * q) * mid;
    }
  }
};

// -(wa wk) acc. In FP32 the weights come as value and rounding error: one rounding where the plain products have three
// and the weights' own. Against 64 bits, N = 4..10, in units of rounding in norm: 0.45-0.55; plain products and the
// factors J (2/h_d)^2 / 2 inside the sums 0.58-0.96 (an x-line's fluxes weighted and summed one by one: 0.47-0.85).
// 48^3 at N = 8 199.5 -> 200.7 us, error 9.7e-8 -> 6.1e-8. In FP64, whose pipe the two extra operations a point would load
// (43^3 at N = 9 5670 -> 6070 us), the values alone: 0.47-0.87 units (before the factors moved 0.58-1.12 and 5900 us).
__device__ __forceinline__ float weighted(float2 wa, float wk, float wk_lo, float acc) {
  const float p = wa.x * wk;
  const float e = fmaf(wa.y, wk, fmaf(wa.x, wk_lo, fmaf(wa.x, wk, -p)));
  return -fmaf(p, acc, e * acc);
}
__device__ __forceinline__ double weighted(double2 wa, double wk, double, double acc) { return -(wa.x * wk) * acc; }

template <typename T, bool L2ONLY>
__device__ __forceinline__ T gld1(const T* __restrict__ p) {
  return L2ONLY ? __ldcg(p) : __ldg(p);
}

// One brick (index blk) of the apply, with the calling CTA's EPB N^2 threads; sm: DirShape::SMEM
// bytes. PDL: the set-up before the first read of u overlaps the previous kernel on the stream.
template <int N, typename T, int EPB, typename CT, bool PDL, bool L2ONLY = false>
__device__ __forceinline__ void apply_dir_block(const ApplyArgs<T>& A, int blk, T* sm) {
  using S = DirShape<N, T, EPB>;
  using L = DirLine<N, T, CT>;
  constexpr int N2 = S::N2, N3 = N2 * N, P = S::P, R = S::R, XW = S::XW;
  T* su = sm;                    // the element
  T* sa = sm + EPB * R;          // sum over directions
  T* sx = sm + 2 * EPB * R;      // [direction][side][value, 2 x derivative][element][N^2]
  __shared__ int4 s_rec[EPB][7];  // subdomain records of the brick's elements
  if constexpr (PDL) pdl_launch_dependents();
  const OpGeom<T>& g = A.g;
  const T* __restrict__ u = A.u;
  const int tid = threadIdx.x;
  const int el = tid / N2, t = tid - el * N2;
  const int t0 = t % N, t1 = t / N;  // x-lines (j, k); y-lines (i, k); z-lines (i, j)
  const int nx = g.nx, ny = g.ny, nxy = nx * ny;
  const int bz0 = blk / (A.nbx * A.nby), br = blk - bz0 * (A.nbx * A.nby), by0 = br / A.nbx, bx0 = br - by0 * A.nbx;
  const int sx_ = A.bsx, sy_ = A.bsx + A.bsy;  // log2 of bx, bx by
  const int lx = el & ((1 << A.bsx) - 1), ly = (el >> sx_) & ((1 << A.bsy) - 1), lz = el >> sy_;
  const int cx = (bx0 << A.bsx) + lx, cy = (by0 << A.bsy) + ly, cz = bz0 * A.bz + lz;
  const bool valid = lz < A.bz && cx < nx && cy < ny && cz < g.nz;
  const int e = valid ? cx + nx * (cy + ny * cz) : 0;
  // faces with a neighbour, and those whose neighbour is in the brick
  bool has[6], in[6];
  has[0] = cx > 0; has[1] = cx + 1 < nx; has[2] = cy > 0; has[3] = cy + 1 < ny; has[4] = cz > 0; has[5] = cz + 1 < g.nz;
  in[0] = lx > 0; in[1] = lx + 1 < (1 << A.bsx) && has[1];
  in[2] = ly > 0; in[3] = ly + 1 < (1 << A.bsy) && has[3];
  in[4] = lz > 0; in[5] = lz + 1 < A.bz && has[5];
  if (A.rS) {
    for (int q = tid; q < EPB * 7; q += S::THREADS) {
      const int el2 = q / 7;
      const int c0 = (bx0 << A.bsx) + (el2 & ((1 << A.bsx) - 1)), c1 = (by0 << A.bsy) + ((el2 >> sx_) & ((1 << A.bsy) - 1)),
                c2 = bz0 * A.bz + (el2 >> sy_);
      if ((el2 >> sy_) < A.bz && c0 < nx && c1 < ny && c2 < g.nz)
        s_rec[el2][q - el2 * 7] = __ldg(A.rec + (int64_t)(c0 + nx * (c1 + ny * c2)) * 7 + (q - el2 * 7));
    }
  }
  const typename PairOf<T>::V wa = __ldg(A.wf + t);
  if constexpr (PDL) pdl_wait();
  T v[N];
  if (valid) gld_line<N, T, L2ONLY>(u + (int64_t)e * N3 + t * N, v);
  // neighbours outside the brick: value and derivative at the shared face
  if (valid) {
#pragma unroll
    for (int f = 0; f < 6; ++f) {
      if (!has[f] || in[f]) continue;
      constexpr int kStep[3] = {1, 0, 0};
      const int d = f >> 1, side = f & 1;
      const int step = d == 0 ? kStep[0] : (d == 1 ? nx : nxy);
      const T* p = u + (int64_t)(side ? e + step : e - step) * N3;
      T q[N];
      if (d == 0) {
        gld_line<N, T, L2ONLY>(p + t * N, q);
      } else {
        p += d == 1 ? t1 * N2 + t0 : t;
#pragma unroll
        for (int l = 0; l < N; ++l) q[l] = gld1<T, L2ONLY>(p + l * (d == 1 ? N : N2));
      }
      // the neighbour's upper end (side 0), or its lower end: D_{0,l} = -D_{N-1,N-1-l}
      T G = T(0);
#pragma unroll
      for (int l = 0; l < N; ++l) G += side ? -L::last_row2(N - 1 - l) * q[l] : L::last_row2(l) * q[l];
      sx[(4 * d + 2 * side) * XW + tid] = side ? q[0] : q[N - 1];
      sx[(4 * d + 2 * side + 1) * XW + tid] = G;
    }
  }
  // this line's ends for the neighbours in the brick along d (step in elements of the brick)
  auto give = [&](int d, const L& ln, T lo, T hi, int step) {
    if (in[2 * d]) {
      sx[(4 * d + 2) * XW + tid - step * N2] = lo;
      sx[(4 * d + 3) * XW + tid - step * N2] = ln.lower2();
    }
    if (in[2 * d + 1]) {
      sx[(4 * d) * XW + tid + step * N2] = hi;
      sx[(4 * d + 1) * XW + tid + step * N2] = ln.upper2();
    }
  };
  // the exterior state at both ends: exchanged, or the ghost state of Eq. bc
  auto take = [&](int d, const L& ln, T lo, T hi, T& u0, T& G0, T& u1, T& G1) {
    if (has[2 * d]) {
      u0 = sx[(4 * d) * XW + tid];
      G0 = sx[(4 * d + 1) * XW + tid];
    } else {
      const bool neu = (g.neumann >> (2 * d)) & 1;
      u0 = neu ? lo : -lo;
      G0 = neu ? -ln.lower2() : ln.lower2();
    }
    if (has[2 * d + 1]) {
      u1 = sx[(4 * d + 2) * XW + tid];
      G1 = sx[(4 * d + 3) * XW + tid];
    } else {
      const bool neu = (g.neumann >> (2 * d + 1)) & 1;
      u1 = neu ? hi : -hi;
      G1 = neu ? -ln.upper2() : ln.upper2();
    }
  };
  T* ex = su + el * R;
  T* ax = sa + el * R;
  L ln;
  T acc[N];
  T u0, G0, u1, G1;
  // x
  T lo = T(0), hi = T(0);
  if (valid) {
    sst_line<N>(ex + t1 * P + t0 * N, v);
    lo = v[0];
    hi = v[N - 1];
    ln.gradient(v);
    give(0, ln, lo, hi, 1);
  }
  __syncthreads();
  if (valid) {
    take(0, ln, lo, hi, u0, G0, u1, G1);
    ln.template divergence<true>(lo, hi, u0, G0, u1, G1, g.lam, g.pen, T(1), acc);
    if (g.q[0] != T(1)) {
#pragma unroll
      for (int l = 0; l < N; ++l) acc[l] *= g.q[0];
    }
    sst_line<N>(ax + t1 * P + t0 * N, acc);
    // y
#pragma unroll
    for (int l = 0; l < N; ++l) v[l] = ex[t1 * P + l * N + t0];
    lo = v[0];
    hi = v[N - 1];
    ln.gradient(v);
    give(1, ln, lo, hi, 1 << A.bsx);
  }
  __syncthreads();
  if (valid) {
    take(1, ln, lo, hi, u0, G0, u1, G1);
#pragma unroll
    for (int l = 0; l < N; ++l) acc[l] = ax[t1 * P + l * N + t0];
    ln.template divergence<false>(lo, hi, u0, G0, u1, G1, g.lam, g.pen, g.q[1], acc);
#pragma unroll
    for (int l = 0; l < N; ++l) ax[t1 * P + l * N + t0] = acc[l];
    // z
#pragma unroll
    for (int l = 0; l < N; ++l) v[l] = ex[l * P + t];
    lo = v[0];
    hi = v[N - 1];
    ln.gradient(v);
    give(2, ln, lo, hi, 1 << sy_);
  }
  const int64_t base = (int64_t)e * N3 + t;
  T bl[N];
  if (valid && A.b) {
#pragma unroll
    for (int l = 0; l < N; ++l) bl[l] = __ldg(A.b + base + l * N2);
  }
  __syncthreads();
  if (!valid) return;
  take(2, ln, lo, hi, u0, G0, u1, G1);
#pragma unroll
  for (int l = 0; l < N; ++l) acc[l] = ax[l * P + t];
  ln.template divergence<false>(lo, hi, u0, G0, u1, G1, g.lam, g.pen, g.q[2], acc);
  // A u = -w_i w_j w_k acc (+ diag u): J (2/h_x)^2 / 2 is in wa
#pragma unroll
  for (int l = 0; l < N; ++l) {
    const int m = l < N - 1 - l ? l : N - 1 - l;  // the weights are symmetric
    T r = weighted(wa, CT::w(m), CT::w_lo(m), acc[l]);
    if (A.diag) r += __ldg(A.diag + base + l * N2) * v[l];
    acc[l] = A.b ? bl[l] - r : r;
  }
  if (!A.rS) {
#pragma unroll
    for (int l = 0; l < N; ++l) A.out[base + l * N2] = acc[l];
    return;
  }
  // Straight into the subdomain vectors that contain the point; every row holds one point, so the stores
  // never collide.
#pragma unroll
  for (int sl = 0; sl < 7; ++sl) {
    const int f = sl - 1;
    if (sl > 0 && f < 4 && !slot_covers<N>(sl, t0, t1, 0, A.ov)) continue;
    const int4 rc = s_rec[el][sl];
    if (rc.x < 0 || !DG_IN_BOUNDS(rc.x, A.E)) continue;
    const int row0 = record_row(rc, t0, t1, 0), dk = (int)(short)(rc.w & 0xFFFF);
    T* colp = A.rS + (int64_t)rc.x * A.ld;
#pragma unroll
    for (int l = 0; l < N; ++l) {
      if (f >= 4 && ((f & 1) ? N - 1 - l : l) >= A.ov) continue;
      const int row = row0 + dk * l;
      if (DG_IN_BOUNDS(row, A.ld)) colp[row] = acc[l];
    }
  }
}

// The same with the three directions side by side: 3 EPB N^2 threads, a thread owns one line of one
// direction, and the three partial sums meet in shared memory. Three times the threads for the same
// arithmetic: on grids too small to fill the GPU the time of the call is the length of one thread's
// chain (in FP64 the issue rate of one warp scheduler's FP64 unit), which this cuts to a third.
template <int N, typename T, int EPB>
struct ParShape {
  static constexpr int N2 = N * N, N3 = N2 * N;
  static constexpr int LN = N | 1;  // line stride: odd, so that x-lines of consecutive lanes differ in bank
  static constexpr int THREADS = 3 * EPB * N2;
  static constexpr int XW = EPB * N2;
  static constexpr int SMEM = (3 * EPB * N2 * LN + 12 * XW) * (int)sizeof(T);
};

template <int N, typename T, int EPB, typename CT, bool PDL>
__device__ __forceinline__ void apply_par_block(const ApplyArgs<T>& A, int blk, T* sm) {
  using S = ParShape<N, T, EPB>;
  using L = DirLine<N, T, CT>;
  constexpr int N2 = S::N2, N3 = S::N3, LN = S::LN, XW = S::XW, PS = EPB * N2 * LN;
  T* sx = sm + 3 * PS;  // exchange, as above; sm: [direction][element][k][j][LN]
  __shared__ int s_e[EPB];
  __shared__ int4 s_rec[EPB][7];
  if constexpr (PDL) pdl_launch_dependents();
  const OpGeom<T>& g = A.g;
  const T* __restrict__ u = A.u;
  const int tid = threadIdx.x;
  const int d = tid / XW, r = tid - d * XW;
  const int el = r / N2, t = r - el * N2;
  const int nx = g.nx, ny = g.ny, nxy = nx * ny;
  const int bz0 = blk / (A.nbx * A.nby), br = blk - bz0 * (A.nbx * A.nby), by0 = br / A.nbx, bx0 = br - by0 * A.nbx;
  const int sx_ = A.bsx, sy_ = A.bsx + A.bsy;
  const int lx = el & ((1 << A.bsx) - 1), ly = (el >> sx_) & ((1 << A.bsy) - 1), lz = el >> sy_;
  const int cx = (bx0 << A.bsx) + lx, cy = (by0 << A.bsy) + ly, cz = bz0 * A.bz + lz;
  const bool valid = lz < A.bz && cx < nx && cy < ny && cz < g.nz;
  const int e = valid ? cx + nx * (cy + ny * cz) : 0;
  // along d: position, count, position in the brick, brick length, element steps
  const int c = d == 0 ? cx : (d == 1 ? cy : cz), cn = d == 0 ? nx : (d == 1 ? ny : g.nz);
  const int lc = d == 0 ? lx : (d == 1 ? ly : lz), bn = d == 0 ? 1 << A.bsx : (d == 1 ? 1 << A.bsy : A.bz);
  const int step = d == 0 ? 1 : (d == 1 ? nx : nxy), lstep = d == 0 ? 1 : (d == 1 ? 1 << sx_ : 1 << sy_);
  const bool has0 = c > 0, has1 = c + 1 < cn;
  const bool in0 = lc > 0, in1 = lc + 1 < bn && has1;
  for (int q = tid; q < EPB * 7; q += S::THREADS) {
    const int el2 = q / 7, sl = q - el2 * 7;
    const int c0 = (bx0 << A.bsx) + (el2 & ((1 << A.bsx) - 1)), c1 = (by0 << A.bsy) + ((el2 >> sx_) & ((1 << A.bsy) - 1)),
              c2 = bz0 * A.bz + (el2 >> sy_);
    const bool ok = (el2 >> sy_) < A.bz && c0 < nx && c1 < ny && c2 < g.nz;
    const int e2 = c0 + nx * (c1 + ny * c2);
    if (sl == 0) s_e[el2] = ok ? e2 : -1;
    if (A.rS && ok) s_rec[el2][sl] = __ldg(A.rec + (int64_t)e2 * 7 + sl);
  }
  // first point and stride of the line: x-lines (j, k) = (t0, t1), y-lines (i, k), z-lines (i, j)
  const int t0 = t % N, t1 = t / N;
  const int p0 = d == 0 ? t * N : (d == 1 ? t1 * N2 + t0 : t), ps = d == 0 ? 1 : (d == 1 ? N : N2);
  if constexpr (PDL) pdl_wait();
  T v[N], q0[N], q1[N];
  if (valid) {
    const T* pu = u + (int64_t)e * N3 + p0;
    const bool n0 = has0 && !in0, n1 = has1 && !in1;
#pragma unroll
    for (int l = 0; l < N; ++l) v[l] = __ldg(pu + l * ps);
#pragma unroll
    for (int l = 0; l < N; ++l) q0[l] = n0 ? __ldg(pu - (int64_t)step * N3 + l * ps) : T(0);
#pragma unroll
    for (int l = 0; l < N; ++l) q1[l] = n1 ? __ldg(pu + (int64_t)step * N3 + l * ps) : T(0);
    T G0 = T(0), G1 = T(0);
#pragma unroll
    for (int l = 0; l < N; ++l) {
      G0 += L::last_row2(l) * q0[l];
      G1 += -L::last_row2(N - 1 - l) * q1[l];
    }
    if (n0) {
      sx[(4 * d) * XW + r] = q0[N - 1];
      sx[(4 * d + 1) * XW + r] = G0;
    }
    if (n1) {
      sx[(4 * d + 2) * XW + r] = q1[0];
      sx[(4 * d + 3) * XW + r] = G1;
    }
  }
  L ln;
  if (valid) {
    ln.gradient(v);
    if (in0) {
      sx[(4 * d + 2) * XW + r - lstep * N2] = v[0];
      sx[(4 * d + 3) * XW + r - lstep * N2] = ln.lower2();
    }
    if (in1) {
      sx[(4 * d) * XW + r + lstep * N2] = v[N - 1];
      sx[(4 * d + 1) * XW + r + lstep * N2] = ln.upper2();
    }
  }
  __syncthreads();
  if (valid) {
    T u0, G0, u1, G1;
    const T lo = v[0], hi = v[N - 1];
    if (has0) {
      u0 = sx[(4 * d) * XW + r];
      G0 = sx[(4 * d + 1) * XW + r];
    } else {
      const bool neu = (g.neumann >> (2 * d)) & 1;
      u0 = neu ? lo : -lo;
      G0 = neu ? -ln.lower2() : ln.lower2();
    }
    if (has1) {
      u1 = sx[(4 * d + 2) * XW + r];
      G1 = sx[(4 * d + 3) * XW + r];
    } else {
      const bool neu = (g.neumann >> (2 * d + 1)) & 1;
      u1 = neu ? hi : -hi;
      G1 = neu ? -ln.upper2() : ln.upper2();
    }
    T acc[N];
    ln.template divergence<true>(lo, hi, u0, G0, u1, G1, g.lam, g.pen, T(1), acc);
    // point (k N + j) N + i at (k N + j) LN + i
    T* dst = sm + d * PS + el * N2 * LN + (d == 0 ? t * LN : (d == 1 ? t1 * N * LN + t0 : t1 * LN + t0));
    const int ds = d == 0 ? 1 : (d == 1 ? LN : N * LN);
#pragma unroll
    for (int l = 0; l < N; ++l) dst[l * ds] = acc[l];
  }
  __syncthreads();
  constexpr int IT = (N3 + 3 * N2 - 1) / (3 * N2);
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int pp = tid + it * S::THREADS;
    if (pp >= EPB * N3) break;
    const int el2 = pp / N3, p = pp - el2 * N3;
    const int e2 = s_e[el2];
    if (e2 < 0) continue;
    const int kj = p / N, i = p - kj * N, k = kj / N, j = kj - k * N;
    const int64_t at = (int64_t)e2 * N3 + p;
    const int o = (el2 * N2 + kj) * LN + i;
    const T acc = fma(g.q[2], sm[2 * PS + o], fma(g.q[1], sm[PS + o], g.q[0] * sm[o]));
    const typename PairOf<T>::V wk = __ldg(A.wf + N2 + k);
    T val = weighted(__ldg(A.wf + j * N + i), wk.x, wk.y, acc);
    if (A.diag) val += __ldg(A.diag + at) * __ldg(u + at);
    if (A.b) val = __ldg(A.b + at) - val;
    if (!A.rS) {
      A.out[at] = val;
      continue;
    }
#pragma unroll
    for (int sl = 0; sl < 7; ++sl) {
      if (!slot_covers<N>(sl, i, j, k, A.ov)) continue;
      const int4 rc = s_rec[el2][sl];
      const int row = record_row(rc, i, j, k);
      if (rc.x >= 0 && DG_IN_BOUNDS(rc.x, A.E) && DG_IN_BOUNDS(row, A.ld)) A.rS[(int64_t)rc.x * A.ld + row] = val;
    }
  }
}

}  // namespace dg
