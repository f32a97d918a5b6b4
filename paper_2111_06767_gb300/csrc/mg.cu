// Multigrid intermesh operators (Sec. III.C.2).
//
// Prolongation (Eq. prol): Lagrange interpolation from the parent's LGL points to each child's
// points at parent-logical coordinates (xi - 1)/2 (lower half), (xi + 1)/2 (upper half) or xi
// (the child spans the parent in that dimension). Restriction R = P^T (no mass matrices, since
// it acts on DG residuals that already carry them). Both are sum-factorised into three 1-D passes, data
// staged in shared memory, sums in a fixed order: deterministic, no atomics.
#include "internal.h"
#include "pdl.cuh"
#include "schwarz_dev.cuh"

namespace dg {

struct XferGeom {
  int nf[3], nc[3];
};

// per dimension: which half a fine coordinate is in (0 lower, 1 upper, 2 full) and its parent
__device__ __forceinline__ void parent_of(int cf, int nf, int nc, int& pc, int& half) {
  if (nf == nc) { pc = cf; half = 2; }
  else { pc = cf >> 1; half = cf & 1; }
}

template <int N, typename T>
__device__ __forceinline__ T interp(const T* sI, int half, int t, int j) {
  // sI: [2][N*N] lower/upper interpolation matrices; half 2 = identity
  return half == 2 ? (t == j ? T(1) : T(0)) : sI[half * N * N + t * N + j];
}

template <int N>
struct XferShape {
  static constexpr int n3 = N * N * N;
  static constexpr int threads = n3 > 512 ? 512 : n3;
};

template <int N, typename T>
__global__ void __launch_bounds__(XferShape<N>::threads) prolongate_kernel(XferGeom x, const T* __restrict__ Ilo,
                                                                           const T* __restrict__ Ihi,
                                                                           const T* __restrict__ uc,
                                                                           T* __restrict__ uf) {
  constexpr int N2 = N * N, N3 = N2 * N, NT = XferShape<N>::threads;
  __shared__ T sI[2 * N2];
  __shared__ T s0[N3], s1[N3];
  const int ef = blockIdx.x;
  const int tid = threadIdx.x;
  for (int t = tid; t < N2; t += NT) { sI[t] = Ilo[t]; sI[N2 + t] = Ihi[t]; }
  const int cx = ef % x.nf[0], cy = (ef / x.nf[0]) % x.nf[1], cz = ef / (x.nf[0] * x.nf[1]);
  int px, py, pz, hx, hy, hz;
  parent_of(cx, x.nf[0], x.nc[0], px, hx);
  parent_of(cy, x.nf[1], x.nc[1], py, hy);
  parent_of(cz, x.nf[2], x.nc[2], pz, hz);
  const int ec = px + x.nc[0] * (py + x.nc[1] * pz);
  pdl_launch_dependents();
  pdl_wait();
  for (int t = tid; t < N3; t += NT) s0[t] = uc[(int64_t)ec * N3 + t];
  __syncthreads();
  for (int t = tid; t < N3; t += NT) {  // along x: s1[c][b][i] = sum_a Ix[i][a] uc[c][b][a]
    const int i = t % N, j = (t / N) % N, k = t / N2;
    T a = 0;
#pragma unroll
    for (int l = 0; l < N; ++l) a += interp<N, T>(sI, hx, i, l) * s0[(k * N + j) * N + l];
    s1[t] = a;
  }
  __syncthreads();
  for (int t = tid; t < N3; t += NT) {  // along y
    const int i = t % N, j = (t / N) % N, k = t / N2;
    T a = 0;
#pragma unroll
    for (int l = 0; l < N; ++l) a += interp<N, T>(sI, hy, j, l) * s1[(k * N + l) * N + i];
    s0[t] = a;
  }
  __syncthreads();
  for (int t = tid; t < N3; t += NT) {  // along z
    const int i = t % N, j = (t / N) % N, k = t / N2;
    T a = 0;
#pragma unroll
    for (int l = 0; l < N; ++l) a += interp<N, T>(sI, hz, k, l) * s0[(l * N + j) * N + i];
    uf[(int64_t)ef * N3 + t] += a;
  }
}

// One output plane (z index c) of one coarse element per CTA: the children are first contracted along z
// for that plane, then the halves are joined direction by direction, so that the y pass works on one or two
// children and the x pass on one sum: 14 N multiply-adds per coarse point in place of 24 N with every
// child passed through all three directions, and N times as many CTAs to spread them over (a coarse grid of 8
// elements fills 8 N SMs). At 8 coarse elements of N = 8: FP64 29.6 -> 4.3 us, FP32 5.3 -> 1.6.
template <int N>
struct RestrictShape {
  static constexpr int n2 = N * N;
  static constexpr int threads = (4 * n2 + 31) / 32 * 32;  // one value of each child column per thread
};

template <int N, typename T>
__global__ void __launch_bounds__(RestrictShape<N>::threads) restrict_kernel(XferGeom x, const T* __restrict__ Ilo,
                                                                             const T* __restrict__ Ihi,
                                                                             const T* __restrict__ rf,
                                                                             T* __restrict__ bc, SubdomainGeom sg,
                                                                             const int4* __restrict__ rec,
                                                                             T* __restrict__ rS) {
  constexpr int N2 = N * N, N3 = N2 * N, NT = RestrictShape<N>::threads;
  __shared__ T sI[2 * N2];
  __shared__ T sz[4 * N2], sy[2 * N2];
  const int ec = blockIdx.x / N, c = blockIdx.x - ec * N;
  const int tid = threadIdx.x;
  for (int t = tid; t < N2; t += NT) { sI[t] = Ilo[t]; sI[N2 + t] = Ihi[t]; }
  const int px = ec % x.nc[0], py = (ec / x.nc[0]) % x.nc[1], pz = ec / (x.nc[0] * x.nc[1]);
  const int rx = x.nf[0] == x.nc[0] ? 1 : 2, ry = x.nf[1] == x.nc[1] ? 1 : 2, rz = x.nf[2] == x.nc[2] ? 1 : 2;
  pdl_launch_dependents();
  __syncthreads();
  pdl_wait();
  // sz[dy][dx][j][i] = sum over the children along z of sum_k Iz[k][c] r[k][j][i]
  {
    const int q = tid / N2, p = tid - q * N2, dx = q & 1, dy = q >> 1;
    if (q < 4 && dx < rx && dy < ry) {
      const int cx = rx * px + dx, cy = ry * py + dy;
      T v[2][N];
#pragma unroll
      for (int dz = 0; dz < 2; ++dz)
#pragma unroll
        for (int l = 0; l < N; ++l) {
          const int64_t ef = cx + x.nf[0] * (cy + (int64_t)x.nf[1] * (rz * pz + (dz < rz ? dz : 0)));
          v[dz][l] = dz < rz ? rf[ef * N3 + l * N2 + p] : T(0);
        }
      T a = 0;
      if (rz == 1) {
#pragma unroll
        for (int l = 0; l < N; ++l) a = l == c ? v[0][l] : a;
      } else {
#pragma unroll
        for (int dz = 0; dz < 2; ++dz)
#pragma unroll
          for (int l = 0; l < N; ++l) a += sI[dz * N2 + l * N + c] * v[dz][l];
      }
      sz[q * N2 + p] = a;
    }
  }
  __syncthreads();
  // sy[dx][b][i] = sum over the children along y of sum_j Iy[j][b] sz[dy][dx][j][i]
  if (tid < rx * N2) {
    const int dx = tid / N2, p = tid - dx * N2, b = p / N, i = p - b * N;
    T a = 0;
    if (ry == 1) {
      a = sz[dx * N2 + p];
    } else {
#pragma unroll
      for (int dy = 0; dy < 2; ++dy)
#pragma unroll
        for (int l = 0; l < N; ++l) a += sI[dy * N2 + l * N + b] * sz[(2 * dy + dx) * N2 + l * N + i];
    }
    sy[tid] = a;
  }
  __syncthreads();
  // along x
  if (tid < N2) {
    const int b = tid / N, i = tid - b * N;
    T a = 0;
    if (rx == 1) {
      a = sy[tid];
    } else {
#pragma unroll
      for (int dx = 0; dx < 2; ++dx)
#pragma unroll
        for (int l = 0; l < N; ++l) a += sI[dx * N2 + l * N + i] * sy[dx * N2 + b * N + l];
    }
    bc[(int64_t)ec * N3 + c * N2 + tid] = a;
    // the coarse level's first smoothing step starts from u = 0: its residual is b
    if (rS) gather_point<N, T>(sg, rec, a, rS, ec, c * N2 + tid);
  }
}

template <typename T>
void launch_prolongate_add(int N, const int nf[3], const int nc[3], const T* Ilo, const T* Ihi, const T* uc, T* uf,
                           cudaStream_t s) {
  XferGeom x{{nf[0], nf[1], nf[2]}, {nc[0], nc[1], nc[2]}};
  const int E = nf[0] * nf[1] * nf[2];
  switch (N) {
#define DG_CASE(NN) \
  case NN: launch_pdl(prolongate_kernel<NN, T>, dim3(E), dim3(XferShape<NN>::threads), 0, s, x, Ilo, Ihi, uc, uf); break;
    DG_CASE(2) DG_CASE(3) DG_CASE(4) DG_CASE(5) DG_CASE(6) DG_CASE(7) DG_CASE(8) DG_CASE(9) DG_CASE(10)
#undef DG_CASE
    default: fail(DG_ERR_INVALID_ARG, "unsupported N");
  }
  DG_LAUNCHED(1);
}

template <typename T>
void launch_restrict(int N, const int nf[3], const int nc[3], const T* Ilo, const T* Ihi, const T* rf, T* bc,
                     const SubdomainGeom* sg, const int4* rec, T* rS, cudaStream_t s) {
  XferGeom x{{nf[0], nf[1], nf[2]}, {nc[0], nc[1], nc[2]}};
  const int E = nc[0] * nc[1] * nc[2];
  const SubdomainGeom g = sg ? *sg : SubdomainGeom{};
  switch (N) {
#define DG_CASE(NN)                                                                                                \
  case NN:                                                                                                         \
    launch_pdl(restrict_kernel<NN, T>, dim3(E * NN), dim3(RestrictShape<NN>::threads), 0, s, x, Ilo, Ihi, rf, bc, g, \
               rec, rS);                                                                                           \
    break;
    DG_CASE(2) DG_CASE(3) DG_CASE(4) DG_CASE(5) DG_CASE(6) DG_CASE(7) DG_CASE(8) DG_CASE(9) DG_CASE(10)
#undef DG_CASE
    default: fail(DG_ERR_INVALID_ARG, "unsupported N");
  }
  DG_LAUNCHED(1);
}

template void launch_prolongate_add<double>(int, const int*, const int*, const double*, const double*, const double*,
                                            double*, cudaStream_t);
template void launch_prolongate_add<float>(int, const int*, const int*, const float*, const float*, const float*,
                                           float*, cudaStream_t);
template void launch_restrict<double>(int, const int*, const int*, const double*, const double*, const double*,
                                      double*, const SubdomainGeom*, const int4*, double*, cudaStream_t);
template void launch_restrict<float>(int, const int*, const int*, const float*, const float*, const float*, float*,
                                     const SubdomainGeom*, const int4*, float*, cudaStream_t);

}  // namespace dg
