// Device building blocks of the Schwarz data movement (Sec. III.D.5), shared by the per-step
// kernels of schwarz.cu, the operator's subdomain output and the fused coarse-level smoother: where a
// point lies in the subdomain vectors, its residual's way in and its weighted correction's way out.
#pragma once

#include "bounds.cuh"
#include "internal.h"
#include "pdl.cuh"

namespace dg {

// Face neighbour of element e across face f (-1 at the domain boundary).
__device__ __forceinline__ int nbr_elem(const SubdomainGeom& g, int e, int f) {
  const int c0 = e % g.n[0], c1 = (e / g.n[0]) % g.n[1], c2 = e / (g.n[0] * g.n[1]);
  int c[3] = {c0, c1, c2};
  const int d = f >> 1;
  c[d] += (f & 1) ? 1 : -1;
  if (c[d] < 0 || c[d] >= g.n[d]) return -1;
  return c[0] + g.n[0] * (c[1] + g.n[1] * c[2]);
}

// Index of the node at position idx_d along d and (a1, a2) along the other two dimensions in
// increasing order (the face layout shared by neighbours across a face of normal d).
template <int N>
__device__ __forceinline__ int node_of(int d, int idx_d, int a1, int a2) {
  int c0, c1, c2;
  if (d == 0) { c0 = idx_d; c1 = a1; c2 = a2; }
  else if (d == 1) { c0 = a1; c1 = idx_d; c2 = a2; }
  else { c0 = a1; c1 = a2; c2 = idx_d; }
  return (c2 * N + c1) * N + c0;
}

// Subdomain row of point p of slot s (0 centre, 1 + f the neighbour across face f) in the
// unreflected point order, or -1 if outside S.
template <int N>
__device__ __forceinline__ int subdomain_row(int s, int p, int ov) {
  if (s == 0) return p;
  const int f = s - 1, d = f >> 1, side = f & 1;
  const int c[3] = {p % N, (p / N) % N, p / (N * N)};
  const int depth = side ? c[d] : N - 1 - c[d];
  if (depth >= ov) return -1;
  const int a1 = d == 0 ? c[1] : c[0];
  const int a2 = d == 2 ? c[1] : c[2];
  return N * N * N + f * ov * N * N + (depth * N + a2) * N + a1;
}

// A level's subdomain records, one per element and slot (0: the element's own subdomain, 1 + f: that of
// the neighbour across face f): (column of the subdomain or -1, row of point (0, 0, 0), row strides along
// i | j << 16, along k | existing-neighbour pattern << 16 in slot 0). The row of a point is affine in its
// indices for every slot and orientation, so one 16-byte record replaces a table look-up per point.
__device__ __forceinline__ int record_row(const int4& r, int i, int j, int k) {
  return r.y + (int)(short)(r.z & 0xFFFF) * i + (r.z >> 16) * j + (int)(short)(r.w & 0xFFFF) * k;
}

// Does the subdomain of slot sl contain point (i, j, k)? (A neighbour's reaches ov layers of its face.)
template <int N>
__device__ __forceinline__ bool slot_covers(int sl, int i, int j, int k, int ov) {
  if (sl == 0) return true;
  const int f = sl - 1, c = f < 2 ? i : (f < 4 ? j : k);
  return ((f & 1) ? N - 1 - c : c) < ov;
}

// r_S rows of point p of element e = val, in every subdomain that contains it (each row is one point's).
template <int N, typename T>
__device__ __forceinline__ void gather_point(const SubdomainGeom& g, const int4* __restrict__ rec, T val,
                                             T* __restrict__ rS, int e, int p) {
  const int i = p % N, j = (p / N) % N, k = p / (N * N);
#pragma unroll
  for (int sl = 0; sl < 7; ++sl) {
    if (!slot_covers<N>(sl, i, j, k, g.ov)) continue;
    const int4 r = __ldg(rec + e * 7 + sl);
    const int row = record_row(r, i, j, k);
    if (r.x >= 0 && DG_IN_BOUNDS(r.x, g.E) && DG_IN_BOUNDS(row, g.ld)) rS[(int64_t)r.x * g.ld + row] = val;
  }
}

// The static part of a point's scatter: its place in the subdomain vectors (-1: not in that slot) and
// the weight of each ([64 patterns][7][N^3] shares). SL = 7: every slot. SL = 4 where 2 ov <= N, so that a
// point lies in the overlap of at most one side per dimension: its own subdomain and one candidate along
// x, y and z (the same terms in the same order, with fewer registers and predicates).
template <int N, int SL, typename T>
__device__ __forceinline__ void scatter_look_up(const SubdomainGeom& g, const int4* __restrict__ rec,
                                                const T* __restrict__ shares, int e, int p, int64_t (&idx)[SL],
                                                int (&col)[SL], T (&w)[SL]) {
  constexpr int N3 = N * N * N;
  const int c[3] = {p % N, (p / N) % N, p / (N * N)};
  const int4 r0 = __ldg(rec + e * 7);
  const T* sh = shares + (size_t)(r0.w >> 16) * 7 * N3 + p;
#pragma unroll
  for (int q = 0; q < SL; ++q) {
    idx[q] = -1;
    col[q] = 0;
    w[q] = T(0);
    int sl = q;
    if constexpr (SL == 4) {
      if (q > 0) {
        const int cd = c[q - 1];
        if (cd < g.ov) sl = 2 * q - 1;
        else if (N - 1 - cd < g.ov) sl = 2 * q;
        else continue;
      }
    } else {
      if (!slot_covers<N>(sl, c[0], c[1], c[2], g.ov)) continue;
    }
    const int4 r = q == 0 ? r0 : __ldg(rec + e * 7 + sl);
    const int row = record_row(r, c[0], c[1], c[2]);
    if (r.x < 0 || !DG_IN_BOUNDS(r.x, g.E) || !DG_IN_BOUNDS(row, g.ld)) continue;
    idx[q] = (int64_t)r.x * g.ld + row;
    col[q] = r.x;
    w[q] = sh[sl * N3];
  }
}

}  // namespace dg
