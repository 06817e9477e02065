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
__device__ __forceinline__ int cell_term_at(const CellGeom& g, float v) {
  // tb = 0: n = -(te - 1)..te - 1; tb > 0: the two runs -(te - 1)..-tb and tb..te - 1
  const int ni = (int)fminf(fmaxf(ceilf(v), -(float)g.te), (float)g.te);
  if (g.tb == 0) return min(max(ni + g.te - 1, 0), g.nterms);
  const int run = g.te - g.tb;
  if (ni <= -g.tb) return max(ni + g.te - 1, 0);
  if (ni <= g.tb) return run;
  return min(run + ni - g.tb, g.nterms);
}

// Terms summed at the cells of coarse cell cc themselves: [lo, hi).  FP32
// (FP64 instructions are dear here): the far and the cell kernel call the same
// function, so a boundary term that rounds either way is still in exactly one sum.
__device__ __forceinline__ void cell_near(const CellGeom& g, int cc, int& lo, int& hi) {
  if (!g.two_level) {
    lo = 0;
    hi = g.nterms;
    return;
  }
  const float C = kCellK * (float)g.c, Xc = (float)(g.k0 + cc * kCellK) * (float)g.w + C;
  lo = cell_term_at(g, (-Xc - 2.5f * C) * (float)g.inv_h);
  hi = max(lo, cell_term_at(g, (-Xc + 2.5f * C) * (float)g.inv_h));
}

// Partial sums of R+ in the form's arithmetic.
template <int FORM>  // 0 FP64, 1 double-float with h n on the split grid, 2 double-float otherwise
struct CellAcc {
  float2 re = {0.f, 0.f}, im = {0.f, 0.f};
};
template <>
struct CellAcc<0> {
  double re = 0.0, im = 0.0;
};
__device__ __forceinline__ double cell_add(double a, double b) { return a + b; }
__device__ __forceinline__ float2 cell_add(float2 a, float2 b) { return f_add(a.x, a.y, b.x, b.y); }
__device__ __forceinline__ double cell_xor(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ float2 cell_xor(float2 v, int o) {
  return make_float2(__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o));
}
__device__ __forceinline__ double cell_f64(double v) { return v; }
__device__ __forceinline__ double cell_f64(float2 v) { return df_to_double(v); }

// x as the form's terms take it: FP64, or X_hi on the split grid + X_lo + X_lo2.
template <int FORM>
struct CellX {
  float h, l, l2;
};
template <>
struct CellX<0> {
  double x;
};
template <int FORM>
__device__ __forceinline__ CellX<FORM> cell_x(const CellGeom& g, double x) {
  if constexpr (FORM == 0) {
    return {x};
  } else {
    const double xg = rint(x * g.inv_grid) * g.grid, r = x - xg;
    const float l = (float)r;
    return {(float)xg, l, (float)(r - (double)l)};
  }
}

// acc += the table's terms first, first + stride, ... below `end` at X.
template <int FORM>
__device__ __forceinline__ void cell_terms(const CellGeom& g, const void* table, const CellX<FORM>& X, int first,
                                           int end, int stride, CellAcc<FORM>& acc) {
  if constexpr (FORM == 0) {
    const double2* tb = static_cast<const double2*>(table);
#pragma unroll 2
    for (int t = first; t < end; t += stride) fp64_term(tb + 3 * (size_t)t, X.x, g.q, acc.re, acc.im);
  } else {
    const float4* tb = static_cast<const float4*>(table);
    int k = 0;
#pragma unroll 2
    for (int t = first; t < end; t += stride) {
      df_term<FORM == 1>(tb + 3 * (size_t)t, X.h, X.l, X.l2, g.q_hi, g.q_lo, acc.re.x, acc.re.y, acc.im.x, acc.im.y);
      if ((++k & (kRenorm - 1)) == 0) {
        df_renorm(acc.re.x, acc.re.y);
        df_renorm(acc.im.x, acc.im.y);
      }
    }
    df_renorm(acc.re.x, acc.re.y);
    df_renorm(acc.im.x, acc.im.y);
  }
}

// Far terms of coarse cell cc at its node j, one block of kFarThreads:
// far[cc kCellPC + j].  `red`: one double2 per warp.
constexpr int kFarThreads = 128;
template <int FORM>
__device__ __forceinline__ void cell_far_node(const CellGeom& g, const void* table, const CellTables& T, int cc, int j,
                                              double2* far, double2* red) {
  const int tid = threadIdx.x;
  const double C = kCellK * g.c, Xc = (double)(g.k0 + cc * kCellK) * g.w + C;
  const CellX<FORM> x = cell_x<FORM>(g, fma(C, T.coarse_t[j], Xc));
  int lo, hi;
  cell_near(g, cc, lo, hi);
  CellAcc<FORM> acc;
  // the two far runs as one sequence, so that the threads share them evenly
  const int nfar = lo + g.nterms - hi, skip = hi - lo;
  const int cut = lo > tid ? (lo - tid + kFarThreads - 1) / kFarThreads * kFarThreads + tid : tid;  // first index >= lo
  cell_terms<FORM>(g, table, x, tid, lo, kFarThreads, acc);
  cell_terms<FORM>(g, table, x, cut + skip, nfar + skip, kFarThreads, acc);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    acc.re = cell_add(acc.re, cell_xor(acc.re, o));
    acc.im = cell_add(acc.im, cell_xor(acc.im, o));
  }
  if ((tid & 31) == 0) red[tid >> 5] = make_double2(cell_f64(acc.re), cell_f64(acc.im));
  __syncthreads();
  if (tid == 0) {
    double2 s = red[0];
#pragma unroll
    for (int w = 1; w < kFarThreads / 32; ++w) s = make_double2(s.x + red[w].x, s.y + red[w].y);
    far[(size_t)cc * kCellPC + j] = s;
  }
}

// Polynomial of one cell, a block of LANES kCellP threads: the LANES lanes of a
// node share its near terms; then one warp, (node, re/im) per thread, adds the
// far values and forms the two matrix products.  That part is in FP64, so it
// is kept to one warp's instructions (about 80; at 50 in each of the block's
// warps it took as long as the terms).  DF: coefficients as double-float pairs
// (float4), else double2.
template <int FORM>
struct CellShared {
  CellX<FORM> x[kCellP];
  double near[2 * kCellP], f[2 * kCellP], ch[2 * kCellP];
};
template <int FORM, bool DF, int LANES>
__device__ __forceinline__ void cell_poly(const CellGeom& g, const void* table, const CellTables& T, int cell,
                                          const double2* far, void* poly, CellShared<FORM>& sh) {
  const int tid = threadIdx.x, node = tid / LANES, lane = tid % LANES;
  const int cc = cell / kCellK, in = cell - cc * kCellK;
  if (tid < kCellP)
    sh.x[tid] = cell_x<FORM>(g, fma(g.c, T.node_t[tid], ((double)(g.k0 + cell) + 0.5) * g.w));
  int lo, hi;
  cell_near(g, cc, lo, hi);
  __syncthreads();
  CellAcc<FORM> acc;
  cell_terms<FORM>(g, table, sh.x[node], lo + lane, hi, LANES, acc);
  // lanes with bit 2 set keep the imaginary part, the others the real part
  const int comp = (lane >> 2) & 1;
  auto mine = comp ? acc.im : acc.re;
  mine = cell_add(mine, cell_xor(comp ? acc.re : acc.im, 4));
  mine = cell_add(mine, cell_xor(mine, 1));
  mine = cell_add(mine, cell_xor(mine, 2));
#pragma unroll
  for (int o = 8; o < LANES; o *= 2) mine = cell_add(mine, cell_xor(mine, o));
  if (lane == 0 || lane == 4) {
    if constexpr (FORM == 0)
      sh.near[2 * node + comp] = mine;
    else
      reinterpret_cast<float2*>(sh.near)[2 * node + comp] = mine;
  }
  __syncthreads();
  if (tid >= 32) return;
  const int i = tid >> 1, re_im = tid & 1;
  double a = 0.0, b = 0.0;
  if constexpr (FORM == 0)
    a = sh.near[tid];
  else
    a = df_to_double(reinterpret_cast<const float2*>(sh.near)[tid]);
  if (g.two_level) {
    const double2* row = reinterpret_cast<const double2*>(T.spread + (size_t)(in * kCellP + i) * kCellPC);
    const double* F = reinterpret_cast<const double*>(far + (size_t)cc * kCellPC) + re_im;
#pragma unroll
    for (int j = 0; j < kCellPC / 2; ++j) {
      const double2 m = row[j];
      a = fma(m.x, F[4 * j], a);
      b = fma(m.y, F[4 * j + 2], b);
    }
  }
  sh.f[tid] = a + b;
  __syncwarp();
  // Chebyshev coefficient i, then the coefficient of t^i
#pragma unroll
  for (int step = 0; step < 2; ++step) {
    const double2* m = reinterpret_cast<const double2*>((step == 0 ? T.to_cheb : T.to_mono) + i * kCellP);
    const double* f = (step == 0 ? sh.f : sh.ch) + re_im;
    a = b = 0.0;
#pragma unroll
    for (int j = 0; j < kCellP / 2; ++j) {
      const double2 mj = m[j];
      a = fma(mj.x, f[4 * j], a);
      b = fma(mj.y, f[4 * j + 2], b);
    }
    a += b;
    if (step == 0) {
      sh.ch[tid] = a;
      __syncwarp();
    }
  }
  if (DF)
    static_cast<float2*>(poly)[(size_t)cell * 2 * kCellP + tid] = df_from_double(a);
  else
    static_cast<double*>(poly)[(size_t)cell * 2 * kCellP + tid] = a;
}

// omega and 1 / omega (0 and 0 at omega = 0) of orbit o.  On the C grid from
// omega^2 by sqrt_rsqrt64, whose chain is shorter than a library root's and a
// division's (both sides measured in pole_cells.cu).
template <bool CGRID>
__device__ __forceinline__ double2 orbit_omega(const SymbolParams& sp, const OrbitParams& op, int o) {
  int a, b;
  orbit_rep(op, o, a, b);
  if (CGRID) {
    const double2 hx = sp.half_x[a], hy = sp.half_y[b];
    const double ax = hx.y * (2.0 * sp.inv_dx), ay = hy.y * (2.0 * sp.inv_dy);
    const double fc = sp.f * hx.x * hy.x;
    const double w2 = fma(sp.g * sp.H, fma(ax, ax, ay * ay), fc * fc);
    if (w2 > 1e-280 && w2 < 1e280) return sqrt_rsqrt64(w2);
  }
  const double w = symbol_at(sp, a, b).omega;
  return make_double2(w, w > 0.0 ? 1.0 / w : 0.0);
}

// The cell of x and the local variable t in [-1, 1] (exact: w is a power of two).
__device__ __forceinline__ int cell_of(const CellGeom& g, double x, double& t) {
  const double magic = 6755399441055744.0;  // 1.5 2^52: the sum's low bits are the nearest integer
  const double v = fma(x, g.inv_w, -0.5);
  const double r = v + magic;
  double kf = r - magic;
  int k = __double2loint(r) - g.k0;
  if (k < 0 || k >= g.ncell) {  // beyond the range by rounding: the edge cell's polynomial
    k = k < 0 ? 0 : g.ncell - 1;
    kf = (double)(g.k0 + k);
  }
  t = 2.0 * (v - kf);
  return k;
}

// Value at t of a cell's polynomial in double-float, real and imaginary part.  Every
// coefficient is a pair, as the terms of a direct sum are: monomial coefficient i
// falls off only like (c/a)^i, 5.13^-i at worst (an FP32 upper half, i >= 8, leaves
// 1.5e-13 of a single pole's value there, pairs 8e-15; at h = 2 it is 5.6e-11 of the
// whole sum against 7e-14).
__device__ __forceinline__ void cell_horner(const float4* __restrict__ p, double t, float2& ar, float2& ai) {
  const float2 td = df_from_double(t);
  const float4 top = p[kCellP - 1];
  ar = make_float2(top.x, top.y);
  ai = make_float2(top.z, top.w);
#pragma unroll
  for (int i = kCellP - 2; i >= 0; --i) {
    const float4 v = p[i];
    const float2 pr = f_mul(ar.x, ar.y, td.x, td.y), pi = f_mul(ai.x, ai.y, td.x, td.y);
    ar = f_add(v.x, v.y, pr.x, pr.y);
    ai = f_add(v.z, v.w, pi.x, pi.y);
  }
}

// fin[o] of orbit o from its cell's polynomial.
template <int KIND, bool CGRID>
__device__ __forceinline__ void cell_orbit(const CellGeom& g, const void* __restrict__ poly, const SymbolParams& sp,
                                           const OrbitParams& op, double tau, double2 R0, int o, void* fin) {
  const double2 om = orbit_omega<CGRID>(sp, op, o);
  double t;
  const int k = cell_of(g, tau * om.x, t);
  if (KIND == kOrbitDf) {
    float2 ar, ai;
    cell_horner(static_cast<const float4*>(poly) + (size_t)k * kCellP, t, ar, ai);
    const float2 iw = df_from_double(om.y);
    const float2 d = f_subf(df_from_double(R0.x), ar);
    OrbitScalarsDF out;
    out.s1 = f_mulf(ai, iw);
    out.s2 = f_mulf(f_mulf(d, iw), iw);
    static_cast<OrbitScalarsDF*>(fin)[o] = out;
    return;
  }
  const double2* p = static_cast<const double2*>(poly) + (size_t)k * kCellP;
  double2 a = p[kCellP - 1];
#pragma unroll
  for (int i = kCellP - 2; i >= 0; --i) {
    const double2 v = p[i];
    a.x = fma(a.x, t, v.x);
    a.y = fma(a.y, t, v.y);
  }
  if (KIND == kOrbitRaw) {
    static_cast<double2*>(fin)[o] = a;
    return;
  }
  OrbitScalars out;
  out.s1 = a.y * om.y;
  out.s2re = (R0.x - a.x) * om.y * om.y;
  out.s2im = R0.y * om.y * om.y;
  out.pad = 0.0;
  static_cast<OrbitScalars*>(fin)[o] = out;
}

}  // namespace rexi
