// ig_tiles64.cuh -- the two passes of an FP64 conjugate-gradient iteration over the rows of one tile, on the
// kBlock threads of a CTA: for the loop kernels (ig_pcg.cu) and for solves in one launch that have fewer
// CTAs than tiles (ig_resident.cu).
#pragma once

#include "ig_device.cuh"

namespace ig {
namespace {

// ------------------------------------------------------------------------------- spmv
// The search direction and its product with A in one pass, for the rows of one tile (t0..t1):
// p = z + beta p and q = A p = A z + beta q (z = D^-1 r from the update kernel; A z gathers z),
// and the tile's sums p.q. Carrying q = A p by this recurrence removes the separate p-update
// pass of the textbook iteration (its p = z + beta p happens here), so an iteration is two
// kernels. beta = 0 at the start of a solve (p = q = 0 there), so the first pass is q = A z.
template <int K>
__device__ __forceinline__ void spmv_tile(const MeshDev& md, int tile, const ScalSnap& sn, double* red,
                                          double* out) {
  const long nn = md.n;
  const long t0 = (long)tile * md.tile_rows;
  const long t1 = t0 + md.tile_rows < nn ? t0 + md.tile_rows : nn;
  const double* __restrict__ A = md.A;
  const double* __restrict__ z = md.z;
  double* __restrict__ p = md.p;
  double* __restrict__ q = md.q;
  double pq[K];
#pragma unroll
  for (int c = 0; c < K; ++c) pq[c] = 0.0;
  for (long row = t0 + threadIdx.x; row < t1; row += kBlock) {
    double w[K];
    row_product<K>(md, A, row, GatherP64<K>{z}, w);
    double zi[K], pi[K], qi[K];
    load_row<K>(z, row, zi);
    load_row<K>(p, row, pi);
#pragma unroll
    for (int c = 0; c < K; ++c) qi[c] = q[c * nn + row];
#pragma unroll
    for (int c = 0; c < K; ++c) {
      const double b = sn.beta[c];
      const double pn = fma(b, pi[c], zi[c]);
      const double qn = fma(b, qi[c], w[c]);
      pi[c] = pn;
      q[c * nn + row] = qn;
      pq[c] = fma(pn, qn, pq[c]);
    }
    store_row<K>(p, row, pi);
  }
  tile_reduce<K, kFixed>(pq, red, out);
}

// ------------------------------------------------------------------------------- update
// x += alpha p, r -= alpha q, z = D^-1 r (rows padded like p, for the next SpMV's gathers) and the
// tile's sums r.z, r.r; a row's loads are issued before its stores. Rows are taken one at a time:
// FP64 arithmetic bounds this kernel, and unrolling the row loop only spills at 64 registers.
template <int K>
__device__ __forceinline__ void update_tile(const MeshDev& md, int tile, const ScalSnap& sn, double* red,
                                            double* out) {
  const int nn = md.n;
  const int t0 = tile * md.tile_rows;
  const int t1 = t0 + md.tile_rows < nn ? t0 + md.tile_rows : nn;
  double acc[2 * K];
#pragma unroll
  for (int i = 0; i < 2 * K; ++i) acc[i] = 0.0;
  const double* __restrict__ Dinv = md.Dinv;
  const double* __restrict__ p = md.p;
  const double* __restrict__ q = md.q;
  double* __restrict__ zv = md.z;
  double* __restrict__ x = md.x;
  double* __restrict__ r = md.r;
#pragma unroll 1
  for (int row = t0 + threadIdx.x; row < t1; row += kBlock) {
    double pi[K], xs[K], qs[K], rs[K];
    const double d = Dinv[row];
    load_row<K>(p, row, pi);
#pragma unroll
    for (int c = 0; c < K; ++c) {
      xs[c] = x[(long)c * nn + row];
      qs[c] = q[(long)c * nn + row];
      rs[c] = r[(long)c * nn + row];
    }
    double zo[K];
#pragma unroll
    for (int c = 0; c < K; ++c) {
      const double a = sn.alpha[c];
      const double rn = fma(-a, qs[c], rs[c]);
      zo[c] = d * rn;
      x[(long)c * nn + row] = fma(a, pi[c], xs[c]);
      r[(long)c * nn + row] = rn;
      acc[c] = fma(rn, zo[c], acc[c]);
      acc[K + c] = fma(rn, rn, acc[K + c]);
    }
    store_row<K>(zv, row, zo);
  }
  tile_reduce<2 * K, kFixed>(acc, red, out);
}

}  // namespace
}  // namespace ig
