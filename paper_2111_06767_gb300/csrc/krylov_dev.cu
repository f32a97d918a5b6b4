// Device-resident flexible GMRES (Sec. III.B; Saad, Iterative Methods, Alg. 9.6): the Hessenberg
// column, its Givens rotations, the residual estimate and the stopping decision are computed on
// the GPU, so an iteration needs no host round trip and a whole solve can be one CUDA graph whose
// Arnoldi loop is a conditional WHILE node (the rotation kernel sets the loop condition).
//
// Every kernel here reads the iteration index j (and the column count m = j + 1) from the solve's
// state in device memory rather than from launch arguments, so the same captured launches serve
// every iteration: V_j and Z_j are addressed as V + j ld and Z + j ld inside the kernels.
//
// An iteration's vector work is four launches besides Z_j: the first Gram-Schmidt pass's inner products;
// its update fused with the second pass's products (a block's tile of every V_k is read twice, the second
// time from L1); the second update fused with the norm, the rotations and the stopping decision; V_{j+1}
// together with the next preconditioner input. The block that arrives last at a counter in the state sums
// the partial products in a fixed order, so the results do not depend on which block that is. At 262,144
// points the ten kernels this replaces (a partial and a final reduction kernel per pass and 40 rows of
// blocks of which most returned at once) made a solve of 10 iterations slower: 4.21 -> 4.02 ms.
#include "internal.h"
#include "pdl.cuh"
#include "schwarz_dev.cuh"

namespace dg {

namespace {
constexpr int kThreads = 256;
inline int grid_for(int64_t n) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((n + kThreads - 1) / kThreads, 152 * 8));
}
}  // namespace

// r0 = ||b - A x0||, reference norm, g_0 = beta, V_0 scale; sets the loop condition.
__global__ void kr_start_kernel(KrylovState* st, double tol, int max_it, int rel_to_b, const double* __restrict__ nrm2,
                                double* __restrict__ g, cudaGraphConditionalHandle loop) {
  pdl_launch_dependents();
  pdl_wait();  // the state and vectors come from the previous kernel
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  st->tol = tol;
  st->max_it = max_it;
  st->rel_to_b = rel_to_b;
  const double beta = sqrt(fmax(nrm2[0], 0.0));
  const double ref = st->rel_to_b ? sqrt(fmax(nrm2[1], 0.0)) : beta;
  st->beta = beta;
  st->tol_abs = st->tol * ref;
  st->j = 0;
  st->k = 0;
  st->runs = 0;
  st->arrived = 0;
  st->est = beta;
  g[0] = beta;
  int status = KR_RUNNING;
  if (!isfinite(beta)) status = KR_BREAKDOWN;
  else if (beta <= st->tol_abs || beta == 0.0) status = KR_CONVERGED;
  else if (st->max_it <= 0) status = KR_CAP;
  st->status = status;
  st->scale = status == KR_RUNNING ? 1.0 / beta : 0.0;
  cudaGraphSetConditional(loop, status == KR_RUNNING ? 1u : 0u);
}

// V_j = scale x and the preconditioner's input, V_j in FP32 (MIXED) or FP64, while the loop runs (j and
// scale from the state); the input also straight into the finest level's subdomain vectors, whose first
// smoothing step starts from u = 0.
template <int N, typename T>
__global__ void kr_next_v_kernel(int n, const double* __restrict__ x, const KrylovState* __restrict__ st,
                                 double* __restrict__ V, int64_t ld, T* __restrict__ vin, SubdomainGeom sg,
                                 const int4* __restrict__ rec, T* __restrict__ rS) {
  constexpr int N3 = N * N * N;
  pdl_launch_dependents();
  pdl_wait();  // the state and vectors come from the previous kernel
  if (st->status != KR_RUNNING) return;
  const double a = st->scale;
  double* v = V + (int64_t)st->j * ld;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double y = a * x[i];
    v[i] = y;
    vin[i] = (T)y;
    const int e = (int)i / N3;
    gather_point<N, T>(sg, rec, (T)y, rS, e, (int)i - e * N3);
  }
}

// Z_j = z (the flexible basis keeps every preconditioned vector) and zfix = z, the fixed input of
// the operator apply that follows
template <typename T>
__global__ void kr_store_z_kernel(int64_t n, const T* __restrict__ z, const KrylovState* __restrict__ st,
                                  double* __restrict__ Z, int64_t ld, double* __restrict__ zfix) {
  pdl_launch_dependents();
  pdl_wait();  // the state and vectors come from the previous kernel
  double* zj = Z + (int64_t)st->j * ld;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double v = (double)z[i];
    zj[i] = v;
    zfix[i] = v;
  }
}

constexpr int kTile = 1024;                        // points of a block's tile, 4 per thread
constexpr int kKrWarps = kThreads / 32;
constexpr int kVecsPerWarp = (kKrGraphCap + kKrWarps - 1) / kKrWarps;  // inner products a warp accumulates
static_assert(kTile == 4 * kThreads, "a thread updates four points of a tile");

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Inner products of a tile (in shared memory, `count` points, zeros after them) with V_0 .. V_{m-1}: warp
// wid adds its vectors wid, wid + 8, ..; with few vectors the warps share a vector's points in ns parts.
__device__ __forceinline__ void tile_dots(const double* sw, int64_t lo, int count, const double* V, int64_t ld, int m,
                                          int ns, double (&acc)[kVecsPerWarp]) {
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int part = wid % ns, first = wid / ns, step = kKrWarps / ns, per = kTile / ns;
#pragma unroll
  for (int q = 0; q < kVecsPerWarp; ++q) {
    const int k = first + q * step;
    if (k >= m) break;
    const double* v = V + (int64_t)k * ld + lo;
    double a0 = 0.0, a1 = 0.0;
#pragma unroll 4
    for (int i = part * per + lane; i < (part + 1) * per; i += 64) {
      if (i < count) a0 += sw[i] * v[i];
      if (i + 32 < count) a1 += sw[i + 32] * v[i + 32];
    }
    acc[q] += a0 + a1;
  }
}

// True in the block that arrives last of the launch (whose writes, and everyone's before, it then sees).
__device__ __forceinline__ bool last_block(KrylovState* st) {
  __shared__ int s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    s_last = atomicAdd(&st->arrived, 1u) == gridDim.x - 1;
    if (s_last) st->arrived = 0;
  }
  __syncthreads();
  if (s_last) __threadfence();
  return s_last;
}

// The block's accumulated products into partial[k * blocks + block], the last block's sums into h[k].
__device__ __forceinline__ void finish_dots(KrylovState* st, int m, int ns, const double (&acc)[kVecsPerWarp],
                                            double* partial, double* __restrict__ h) {
  __shared__ double red[kKrWarps][kVecsPerWarp];
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31, blocks = gridDim.x;
#pragma unroll
  for (int q = 0; q < kVecsPerWarp; ++q) {
    const double t = warp_sum(acc[q]);
    if (lane == 0) red[wid][q] = t;
  }
  __syncthreads();
  const int step = kKrWarps / ns;
  for (int k = threadIdx.x; k < m; k += kThreads) {
    double t = 0.0;
    for (int p = 0; p < ns; ++p) t += red[(k % step) * ns + p][k / step];
    partial[(int64_t)k * blocks + blockIdx.x] = t;
  }
  if (!last_block(st)) return;
  for (int k = wid; k < m; k += kKrWarps) {
    double t = 0.0;
    for (int b = lane; b < blocks; b += 32) t += __ldcg(partial + (int64_t)k * blocks + b);
    t = warp_sum(t);
    if (lane == 0) h[k] = t;
  }
}

__device__ __forceinline__ int vector_parts(int m) { return m == 1 ? 8 : (m == 2 ? 4 : (m <= 4 ? 2 : 1)); }

// UPDATE = false: h2 = V^T w. UPDATE = true: w -= V h1, then h2 = V^T w.
template <bool UPDATE>
__global__ void __launch_bounds__(kThreads) kr_dots_kernel(int64_t n, const double* __restrict__ V, int64_t ld,
                                                           const double* __restrict__ h1, double* w, KrylovState* st,
                                                           double* partial, double* __restrict__ h2) {
  __shared__ double sw[kTile];
  pdl_launch_dependents();
  pdl_wait();  // the state and vectors come from the previous kernel
  const int m = st->j + 1, ns = vector_parts(m);
  double acc[kVecsPerWarp] = {};
  for (int64_t lo = blockIdx.x * (int64_t)kTile; lo < n; lo += gridDim.x * (int64_t)kTile) {
    const int count = (int)min((int64_t)kTile, n - lo);
    double x[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = threadIdx.x + q * kThreads;
      x[q] = i < count ? w[lo + i] : 0.0;
    }
    if constexpr (UPDATE) {
#pragma unroll 2
      for (int k = 0; k < m; ++k) {
        const double c = h1[k];
        const double* v = V + (int64_t)k * ld + lo;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int i = threadIdx.x + q * kThreads;
          if (i < count) x[q] -= c * v[i];
        }
      }
    }
    __syncthreads();  // the previous tile has been read
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = threadIdx.x + q * kThreads;
      sw[i] = x[q];
      if (UPDATE && i < count) w[lo + i] = x[q];
    }
    __syncthreads();
    tile_dots(sw, lo, count, V, ld, m, ns, acc);
  }
  finish_dots(st, m, ns, acc, partial, h2);
}

// Column j of the Hessenberg matrix from the two Gram-Schmidt passes, the previous rotations
// applied to it, the new rotation, the residual estimate |g_{j+1}| and the stopping decision; while
// the loop continues, the scale 1 / h_{j+1,j} of the next basis vector and j + 1. One thread.
__device__ void kr_givens(KrylovState* st, double* __restrict__ H, int ldh, double* __restrict__ cs,
                          double* __restrict__ sn, double* __restrict__ g, const double* h1, const double* h2,
                          double nrm2, const volatile int* cancel, cudaGraphConditionalHandle loop) {
  if (st->status != KR_RUNNING) {
    cudaGraphSetConditional(loop, 0u);
    return;
  }
  const int j = st->j;
  st->runs = j + 1;
  double* col = H + (int64_t)j * ldh;
  for (int i = 0; i <= j; ++i) col[i] = h1[i] + h2[i];
  const double hn = sqrt(fmax(0.0, nrm2));
  col[j + 1] = hn;
  for (int i = 0; i < j; ++i) {  // previous rotations
    const double a = col[i], c = col[i + 1];
    col[i] = cs[i] * a + sn[i] * c;
    col[i + 1] = -sn[i] * a + cs[i] * c;
  }
  const double den = hypot(col[j], col[j + 1]);
  int status = KR_RUNNING;
  if (den == 0.0 || !isfinite(den)) {
    status = KR_BREAKDOWN;  // column j is unusable: the update keeps the k = j columns before it
  } else {
    cs[j] = col[j] / den;
    sn[j] = col[j + 1] / den;
    col[j] = den;
    col[j + 1] = 0.0;
    g[j + 1] = -sn[j] * g[j];
    g[j] = cs[j] * g[j];
    st->k = j + 1;
    const double est = fabs(g[j + 1]);
    st->est = est;
    if (!isfinite(est)) status = KR_BREAKDOWN;
    else if (est <= st->tol_abs || hn == 0.0) status = KR_CONVERGED;
    else if (j + 1 >= st->max_it) status = KR_CAP;
    else if (cancel && *cancel) status = KR_CANCELLED;
  }
  st->status = status;
  if (status == KR_RUNNING) {
    st->scale = 1.0 / hn;
    st->j = j + 1;
  }
  cudaGraphSetConditional(loop, status == KR_RUNNING ? 1u : 0u);
}

// w -= V h2, its norm, then in the last block the rotations and the stopping decision.
__global__ void __launch_bounds__(kThreads)
    kr_finish_kernel(int64_t n, const double* __restrict__ V, int64_t ld, const double* __restrict__ h1,
                     const double* __restrict__ h2, double* w, KrylovState* st, double* partial, double* __restrict__ H,
                     int ldh, double* __restrict__ cs, double* __restrict__ sn, double* __restrict__ g,
                     const volatile int* cancel, cudaGraphConditionalHandle loop) {
  __shared__ double red[kKrWarps];
  pdl_launch_dependents();
  pdl_wait();  // the state and vectors come from the previous kernel
  const int m = st->j + 1;
  double acc = 0.0;
  for (int64_t lo = blockIdx.x * (int64_t)kTile; lo < n; lo += gridDim.x * (int64_t)kTile) {
    const int count = (int)min((int64_t)kTile, n - lo);
    double x[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = threadIdx.x + q * kThreads;
      x[q] = i < count ? w[lo + i] : 0.0;
    }
#pragma unroll 2
    for (int k = 0; k < m; ++k) {
      const double c = h2[k];
      const double* v = V + (int64_t)k * ld + lo;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int i = threadIdx.x + q * kThreads;
        if (i < count) x[q] -= c * v[i];
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = threadIdx.x + q * kThreads;
      if (i < count) w[lo + i] = x[q];
      acc += x[q] * x[q];
    }
  }
  const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  acc = warp_sum(acc);
  if (lane == 0) red[wid] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int q = 0; q < kKrWarps; ++q) t += red[q];
    partial[blockIdx.x] = t;
  }
  if (!last_block(st) || wid != 0) return;
  double t = 0.0;
  for (int b = lane; b < gridDim.x; b += 32) t += __ldcg(partial + b);
  t = warp_sum(t);
  if (lane == 0) kr_givens(st, H, ldh, cs, sn, g, h1, h2, t, cancel, loop);
}

// y = R^-1 g over the k completed columns (back substitution). One thread.
__global__ void kr_trisolve_kernel(const KrylovState* __restrict__ st, const double* __restrict__ H, int ldh,
                                   const double* __restrict__ g, double* __restrict__ y) {
  pdl_launch_dependents();
  pdl_wait();  // the state and vectors come from the previous kernel
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const int k = st->k;
  for (int i = k - 1; i >= 0; --i) {
    double acc = g[i];
    for (int l = i + 1; l < k; ++l) acc -= H[(int64_t)l * ldh + i] * y[l];
    y[i] = acc / H[(int64_t)i * ldh + i];
  }
}

// x += sum_{l < k} y[l] Z_l
__global__ void kr_add_comb_kernel(int64_t n, const double* __restrict__ Z, int64_t ld, const double* __restrict__ y,
                                   const KrylovState* __restrict__ st, double* __restrict__ x) {
  pdl_launch_dependents();
  pdl_wait();  // the state and vectors come from the previous kernel
  const int m = st->k;
  if (m == 0) return;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    double acc = x[i];
    for (int l = 0; l < m; ++l) acc += y[l] * Z[(int64_t)l * ld + i];
    x[i] = acc;
  }
}

// ------------------------------------------------------------------ launchers
//
// Every kernel above waits for its predecessor (griddepcontrol.wait) before touching the state or
// the vectors, so they can be launched with programmatic dependent launch (DG_PDL_KRYLOV=1; off by
// default, see pdl_krylov_enabled).

void launch_kr_start(KrylovState* st, double tol, int max_it, bool rel_to_b, const double* nrm2, double* g,
                     cudaGraphConditionalHandle loop, cudaStream_t s) {
  const PdlScope pdl(pdl_krylov_enabled());
  launch_pdl(kr_start_kernel, dim3(1), dim3(32), 0, s, st, tol, max_it, rel_to_b ? 1 : 0, nrm2, g, loop);
  DG_LAUNCHED(1);
}

// The outcome of one captured solve as 8 doubles: completed columns, status, loop bodies run,
// ||b - A x0||, the reference norm, the final ||b - A x||, the stopping threshold.
__global__ void kr_report_kernel(const KrylovState* __restrict__ st, const double* __restrict__ nrm2,
                                 double* __restrict__ out) {
  pdl_launch_dependents();
  pdl_wait();  // the state and vectors come from the previous kernel
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  out[0] = st->k;
  out[1] = st->status;
  out[2] = st->runs;
  out[3] = st->beta;
  out[4] = st->rel_to_b ? sqrt(fmax(nrm2[1], 0.0)) : st->beta;
  out[5] = sqrt(fmax(nrm2[2], 0.0));
  out[6] = st->tol_abs;
  out[7] = 0.0;
}
void launch_kr_report(const KrylovState* st, const double* nrm2, double* out, cudaStream_t s) {
  const PdlScope pdl(pdl_krylov_enabled());
  launch_pdl(kr_report_kernel, dim3(1), dim3(32), 0, s, st, nrm2, out);
  DG_LAUNCHED(1);
}
template <typename T>
void launch_kr_next_v(int64_t n, const double* x, const KrylovState* st, double* V, int64_t ld, T* vin,
                      const SubdomainGeom& sg, const int4* rec, T* rS, cudaStream_t s) {
  const PdlScope pdl(pdl_krylov_enabled());
  switch (sg.N) {
#define DG_CASE(NN)                                                                                                 \
  case NN:                                                                                                          \
    launch_pdl(kr_next_v_kernel<NN, T>, dim3(grid_for(n)), dim3(kThreads), 0, s, (int)n, x, st, V, ld, vin, sg, rec, \
               rS);                                                                                                 \
    break;
    DG_CASE(2) DG_CASE(3) DG_CASE(4) DG_CASE(5) DG_CASE(6) DG_CASE(7) DG_CASE(8) DG_CASE(9) DG_CASE(10)
#undef DG_CASE
    default: fail(DG_ERR_INVALID_ARG, "unsupported N");
  }
  DG_LAUNCHED(1);
}
template void launch_kr_next_v<float>(int64_t, const double*, const KrylovState*, double*, int64_t, float*,
                                      const SubdomainGeom&, const int4*, float*, cudaStream_t);
template void launch_kr_next_v<double>(int64_t, const double*, const KrylovState*, double*, int64_t, double*,
                                       const SubdomainGeom&, const int4*, double*, cudaStream_t);
template <typename T>
void launch_kr_store_z(int64_t n, const T* z, const KrylovState* st, double* Z, int64_t ld, double* zfix,
                       cudaStream_t s) {
  const PdlScope pdl(pdl_krylov_enabled());
  launch_pdl(kr_store_z_kernel<T>, dim3(grid_for(n)), dim3(kThreads), 0, s, n, z, st, Z, ld, zfix);
  DG_LAUNCHED(1);
}
template void launch_kr_store_z<float>(int64_t, const float*, const KrylovState*, double*, int64_t, double*,
                                       cudaStream_t);
template void launch_kr_store_z<double>(int64_t, const double*, const KrylovState*, double*, int64_t, double*,
                                        cudaStream_t);
// w orthogonalised against V_0 .. V_j (classical Gram-Schmidt, twice), column j and the decision.
void launch_kr_orthogonalize(int64_t n, const double* V, int64_t ld, double* w, KrylovState* st, double* partial,
                             double* H, int ldh, double* cs, double* sn, double* g, double* h1, double* h2,
                             const volatile int* cancel, cudaGraphConditionalHandle loop, cudaStream_t s) {
  const PdlScope pdl(pdl_krylov_enabled());
  const dim3 grid((unsigned)std::min<int64_t>((n + kTile - 1) / kTile, multidot_partial_blocks()));
  launch_pdl(kr_dots_kernel<false>, grid, dim3(kThreads), 0, s, n, V, ld, (const double*)nullptr, w, st, partial, h1);
  launch_pdl(kr_dots_kernel<true>, grid, dim3(kThreads), 0, s, n, V, ld, (const double*)h1, w, st, partial, h2);
  launch_pdl(kr_finish_kernel, grid, dim3(kThreads), 0, s, n, V, ld, (const double*)h1, (const double*)h2, w, st,
             partial, H, ldh, cs, sn, g, cancel, loop);
  DG_LAUNCHED(3);
}
void launch_kr_trisolve(const KrylovState* st, const double* H, int ldh, const double* g, double* y, cudaStream_t s) {
  const PdlScope pdl(pdl_krylov_enabled());
  launch_pdl(kr_trisolve_kernel, dim3(1), dim3(32), 0, s, st, H, ldh, g, y);
  DG_LAUNCHED(1);
}
void launch_kr_add_comb(int64_t n, const double* Z, int64_t ld, const double* y, const KrylovState* st, double* x,
                        cudaStream_t s) {
  const PdlScope pdl(pdl_krylov_enabled());
  launch_pdl(kr_add_comb_kernel, dim3(grid_for(n)), dim3(kThreads), 0, s, n, Z, ld, y, st, x);
  DG_LAUNCHED(1);
}

}  // namespace dg
