// Pole sums by local expansion: R+(x) = sum_n (A_n + B_n y)/(q + y^2), y = x + h n,
// for many x at once.
//
// Every pole of R+ lies a = |h mu| off the real axis, so on a cell of
// half-width c <= a/5.13 the polynomial through kCellP Chebyshev nodes
// reproduces R+ to 10.36^-16 = 6e-17 of a pole's residue over c (the Bernstein
// ellipse that touches the pole has parameter 5.13 + sqrt(1 + 5.13^2)).  The
// sum over all terms therefore runs once per node (16 per cell of width 2c,
// c = 1/2 at h = 1/2) instead of once per orbit, and an orbit evaluates its
// cell's polynomial.  The terms enter at two levels: a coarse cell of kCellK
// cells takes the terms whose poles lie more than 2.5 of its half-widths from
// its centre at kCellPC nodes (4.79^-24 = 5e-17), and only the terms nearer
// than that (160 at h = 1/2, of 4067 at tau rho = 1000) are summed at the
// nodes of the cells themselves.  No term is dropped: each one is in exactly
// one of the two sums.
//
// c is a power of two, cell centres are odd multiples of c and the nodes are
// rounded to 2^-24 of the cell, so node positions, centres and the local
// variable t = (x - centre)/c are exact in FP64; the interpolation matrices
// belong to the rounded nodes.  Node values -> Chebyshev coefficients ->
// monomials (coefficients fall off like 10.36^-k, faster than the 2.41^k by
// which the change of basis can amplify), then Horner's rule.
#pragma once

#include "internal.h"
#include "pole_common.cuh"

namespace rexi {

// First index of the table's terms (n ascending, |n| in [tb, te)) with n >= v.
__device__ __forceinline__ int cell_term_at(const CellGeom& g, double v) {
  // tb = 0: n = -(te - 1)..te - 1; tb > 0: the two runs -(te - 1)..-tb and tb..te - 1
  const double n = fmin(fmax(ceil(v), -(double)g.te), (double)g.te);
  const int ni = (int)n;
  if (g.tb == 0) return min(max(ni + g.te - 1, 0), g.nterms);
  const int run = g.te - g.tb;
  if (ni <= -g.tb) return max(ni + g.te - 1, 0);
  if (ni <= g.tb) return run;
  return min(run + ni - g.tb, g.nterms);
}

// Terms summed at the cells of coarse cell cc themselves: [lo, hi).
__device__ __forceinline__ void cell_near(const CellGeom& g, int cc, int& lo, int& hi) {
  if (!g.two_level) {
    lo = 0;
    hi = g.nterms;
    return;
  }
  const double C = kCellK * g.c, Xc = (double)(g.k0 + cc * kCellK) * g.w + C;
  lo = cell_term_at(g, (-Xc - 2.5 * C) * g.inv_h);
  hi = max(lo, cell_term_at(g, (-Xc + 2.5 * C) * g.inv_h));
}

// Sum of the table's terms first, first + stride, ... below `end` at x.
template <int FORM>  // 0 FP64, 1 double-float with h n on the split grid, 2 double-float otherwise
__device__ __forceinline__ void cell_terms(const CellGeom& g, const void* table, double x, int first, int end,
                                           int stride, double& re, double& im) {
  if (FORM == 0) {
    const double2* tb = static_cast<const double2*>(table);
#pragma unroll 2
    for (int t = first; t < end; t += stride) fp64_term(tb + 3 * (size_t)t, x, g.q, re, im);
  } else {
    const float4* tb = static_cast<const float4*>(table);
    const double xg = rint(x * g.inv_grid) * g.grid;
    const float Xh = (float)xg, Xl = (float)(x - xg), Xl2 = (float)((x - xg) - (double)Xl);
    float arh = 0.f, arl = 0.f, aih = 0.f, ail = 0.f;
    int k = 0;
#pragma unroll 2
    for (int t = first; t < end; t += stride) {
      df_term<FORM == 1>(tb + 3 * (size_t)t, Xh, Xl, Xl2, g.q_hi, g.q_lo, arh, arl, aih, ail);
      if ((++k & (kRenorm - 1)) == 0) {
        df_renorm(arh, arl);
        df_renorm(aih, ail);
      }
    }
    re += (double)arh + (double)arl;
    im += (double)aih + (double)ail;
  }
}

// Far terms of coarse cell cc at its node j, one warp: far[cc kCellPC + j].
template <int FORM>
__device__ __forceinline__ void cell_far_node(const CellGeom& g, const void* table, const CellTables& T, int cc, int j,
                                              double2* far) {
  const int lane = threadIdx.x & 31;
  const double C = kCellK * g.c, Xc = (double)(g.k0 + cc * kCellK) * g.w + C;
  const double x = fma(C, T.coarse_t[j], Xc);
  int lo, hi;
  cell_near(g, cc, lo, hi);
  double re = 0.0, im = 0.0;
  // the two far runs as one sequence, so that the lanes share them evenly
  const int nfar = lo + g.nterms - hi, skip = hi - lo;
  const int cut = lo > lane ? (lo - lane + 31) / 32 * 32 + lane : lane;  // first of this lane's indices >= lo
  cell_terms<FORM>(g, table, x, lane, lo, 32, re, im);
  cell_terms<FORM>(g, table, x, cut + skip, nfar + skip, 32, re, im);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    re += __shfl_xor_sync(0xffffffffu, re, o);
    im += __shfl_xor_sync(0xffffffffu, im, o);
  }
  if (lane == 0) far[(size_t)cc * kCellPC + j] = make_double2(re, im);
}

// Polynomial of one cell, a block of kCellP x 16 threads: 16 lanes per node
// share the near terms, then the same 16 lanes form the two matrix products.
template <int FORM>
__device__ __forceinline__ void cell_poly(const CellGeom& g, const void* table, const CellTables& T, int cell,
                                          const double2* far, double2* poly, double2* sh /* 2 kCellP */) {
  const int lane = threadIdx.x & 15, node = threadIdx.x >> 4;
  const int cc = cell / kCellK, in = cell - cc * kCellK;
  const double x = fma(g.c, T.node_t[node], ((double)(g.k0 + cell) + 0.5) * g.w);
  int lo, hi;
  cell_near(g, cc, lo, hi);
  double re = 0.0, im = 0.0;
  cell_terms<FORM>(g, table, x, lo + lane, hi, 16, re, im);
  if (g.two_level) {
    const double* row = T.spread + (size_t)(in * kCellP + node) * kCellPC;
    const double2* F = far + (size_t)cc * kCellPC;
#pragma unroll
    for (int j = lane; j < kCellPC; j += 16) {
      const double2 v = F[j];
      re = fma(row[j], v.x, re);
      im = fma(row[j], v.y, im);
    }
  }
  auto sum16 = [](double& a, double& b) {
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {
      a += __shfl_xor_sync(0xffffffffu, a, o);
      b += __shfl_xor_sync(0xffffffffu, b, o);
    }
  };
  sum16(re, im);
  if (lane == 0) sh[node] = make_double2(re, im);
  __syncthreads();
  {  // Chebyshev coefficient `node`
    const double m = T.to_cheb[node * kCellP + lane];
    const double2 v = sh[lane];
    re = m * v.x;
    im = m * v.y;
    sum16(re, im);
    if (lane == 0) sh[kCellP + node] = make_double2(re, im);
  }
  __syncthreads();
  {  // coefficient of t^node
    const double m = T.to_mono[node * kCellP + lane];
    const double2 v = sh[kCellP + lane];
    re = m * v.x;
    im = m * v.y;
    sum16(re, im);
    if (lane == 0) poly[(size_t)cell * kCellP + node] = make_double2(re, im);
  }
}

// R+(x) from its cell's polynomial.
__device__ __forceinline__ double2 cell_eval(const CellGeom& g, const double2* __restrict__ poly, double x) {
  int k = (int)floor(x * g.inv_w) - g.k0;
  k = min(max(k, 0), g.ncell - 1);  // x beyond the range by rounding: the edge cell's polynomial
  const double t = (x - ((double)(g.k0 + k) + 0.5) * g.w) * g.inv_c;
  const double2* p = poly + (size_t)k * kCellP;
  double2 a = p[kCellP - 1];
#pragma unroll
  for (int i = kCellP - 2; i >= 0; --i) {
    const double2 v = p[i];
    a.x = fma(a.x, t, v.x);
    a.y = fma(a.y, t, v.y);
  }
  return a;
}

}  // namespace rexi
