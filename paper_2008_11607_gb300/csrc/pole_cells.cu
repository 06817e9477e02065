// Kernels and dispatch of the pole sum by local expansion (pole_cells.cuh).
//
// What bounds it, and the split.  Direct sums cost orbits x terms evaluations
// of 62 FP32 operations (mixed) or 9 FP64 instructions; the cells cost nodes
// x near terms + coarse nodes x far terms.  The far kernel gives a warp to
// each coarse node (24 per 32 cells), the cell kernel 16 lanes to each node,
// so that both have warps for every SM and short chains; what is left is one
// polynomial per orbit in FP64, about 45 dependent operations, and the orbit's
// omega.  Measured (GB300): 2048^2, tau rho = 1000, 525,825 orbits x 4067
// terms, direct 4286 us (mixed) and 32,902 us (FP64), cells 166 us and 225 us;
// 375 x 500, tau rho = 150, FP64, 47,188 orbits x 667 terms, 521 us against
// 40 us.  Error against 64 bits as the direct sums' or smaller (shorter sums).
#include <math.h>

#include <algorithm>

#include "pole_cells.cuh"

namespace rexi {

namespace {

constexpr int kFarWarps = 4;
static_assert(kCellPC % kFarWarps == 0, "a block's warps belong to one coarse cell");
static_assert(kCellP == 16, "cell_poly's lanes");

template <int FORM>
__global__ void __launch_bounds__(kFarWarps * 32) cell_far_kernel(CellGeom g, CellTables T,
                                                                  const void* __restrict__ table, double2* far) {
  cell_far_node<FORM>(g, table, T, blockIdx.y, blockIdx.x * kFarWarps + (threadIdx.x >> 5), far);
}

template <int FORM>
__global__ void __launch_bounds__(kCellP * 16) cell_poly_kernel(CellGeom g, CellTables T,
                                                                const void* __restrict__ table,
                                                                const double2* __restrict__ far, double2* poly) {
  __shared__ double2 sh[2 * kCellP];
  cell_poly<FORM>(g, table, T, blockIdx.x, far, poly, sh);
}

template <int KIND>
__global__ void __launch_bounds__(256) cell_orbits_kernel(CellGeom g, const double2* __restrict__ poly,
                                                          SymbolParams sp, OrbitParams op, double tau, double2 R0,
                                                          void* __restrict__ fin) {
  const int o = blockIdx.x * blockDim.x + threadIdx.x;
  if (o >= op.norb) return;
  int a, b;
  orbit_rep(op, o, a, b);
  const double omega = symbol_at(sp, a, b).omega;
  orbit_store<KIND>(fin, o, omega, R0, cell_eval(g, poly, tau * omega));
}

typedef long double ld;

// Inverse of the n x n Chebyshev-Vandermonde matrix V[j][k] = T_k(x_j)
// (Gauss-Jordan with partial pivoting; its condition number is about n).
std::vector<ld> cheb_inverse(const std::vector<double>& x) {
  const int n = (int)x.size();
  std::vector<ld> V(n * n), I(n * n, 0.0L);
  for (int j = 0; j < n; ++j) {
    ld t0 = 1.0L, t1 = x[j];
    for (int k = 0; k < n; ++k) {
      V[j * n + k] = t0;
      const ld t2 = 2.0L * x[j] * t1 - t0;
      t0 = t1;
      t1 = t2;
    }
    I[j * n + j] = 1.0L;
  }
  for (int c = 0; c < n; ++c) {
    int p = c;
    for (int r = c + 1; r < n; ++r)
      if (fabsl(V[r * n + c]) > fabsl(V[p * n + c])) p = r;
    for (int k = 0; k < n; ++k) {
      std::swap(V[c * n + k], V[p * n + k]);
      std::swap(I[c * n + k], I[p * n + k]);
    }
    const ld d = 1.0L / V[c * n + c];
    for (int k = 0; k < n; ++k) {
      V[c * n + k] *= d;
      I[c * n + k] *= d;
    }
    for (int r = 0; r < n; ++r) {
      const ld f = V[r * n + c];
      if (r == c || f == 0.0L) continue;
      for (int k = 0; k < n; ++k) {
        V[r * n + k] -= f * V[c * n + k];
        I[r * n + k] -= f * I[c * n + k];
      }
    }
  }
  return I;  // I[k][j]: coefficient k from value j
}

std::vector<double> cheb_points(int n) {
  std::vector<double> x(n);
  for (int j = 0; j < n; ++j) x[j] = rint(cos(M_PI * (2 * j + 1) / (2.0 * n)) * 16777216.0) / 16777216.0;
  return x;
}

std::vector<double> build_tables() {
  const std::vector<double> t = cheb_points(kCellP), T = cheb_points(kCellPC);
  std::vector<double> out(t);
  out.insert(out.end(), T.begin(), T.end());
  const std::vector<ld> inv = cheb_inverse(t), invC = cheb_inverse(T);
  // spread[(i P + j) PC + m]: value at node j of cell i of a coarse cell from the coarse value m
  for (int i = 0; i < kCellK; ++i)
    for (int j = 0; j < kCellP; ++j) {
      const ld y = ((ld)(2 * i + 1 - kCellK) + (ld)t[j]) / kCellK;
      ld Ty[kCellPC];
      Ty[0] = 1.0L;
      Ty[1] = y;
      for (int k = 2; k < kCellPC; ++k) Ty[k] = 2.0L * y * Ty[k - 1] - Ty[k - 2];
      for (int m = 0; m < kCellPC; ++m) {
        ld s = 0.0L;
        for (int k = 0; k < kCellPC; ++k) s += Ty[k] * invC[k * kCellPC + m];
        out.push_back((double)s);
      }
    }
  for (ld v : inv) out.push_back((double)v);
  // monomial coefficients of T_k: rows i (power), columns k; integers
  std::vector<double> mono(kCellP * kCellP, 0.0);
  mono[0] = 1.0;
  mono[kCellP + 1] = 1.0;
  for (int k = 2; k < kCellP; ++k)
    for (int i = 0; i < kCellP; ++i)
      mono[i * kCellP + k] = (i > 0 ? 2.0 * mono[(i - 1) * kCellP + k - 1] : 0.0) - mono[i * kCellP + k - 2];
  out.insert(out.end(), mono.begin(), mono.end());
  return out;
}

}  // namespace

const std::vector<double>& cell_tables_host() {
  static const std::vector<double> t = build_tables();
  return t;
}

CellTables cell_tables_at(const double* dev) {
  CellTables T;
  T.node_t = dev;
  T.coarse_t = T.node_t + kCellP;
  T.spread = T.coarse_t + kCellPC;
  T.to_cheb = T.spread + kCellK * kCellP * kCellPC;
  T.to_mono = T.to_cheb + kCellP * kCellP;
  return T;
}

bool cell_geometry(int form, int norb, int nterms, int tb, int te, double h, double q, double x_lo, double x_hi,
                   double grid, CellGeom* g) {
  if (nterms < 1 || !(q > 0.0) || !(x_hi >= x_lo)) return false;
  const double a = sqrt(q);
  g->c = ldexp(1.0, (int)floor(log2(a / 5.13)));
  if (!(g->c > 1e-12) || !(std::max(fabs(x_lo), fabs(x_hi)) < 1e8)) return false;
  g->w = 2.0 * g->c;
  g->inv_c = 1.0 / g->c;
  g->inv_w = 0.5 * g->inv_c;
  g->inv_h = 1.0 / h;
  g->q = q;
  g->q_hi = (float)q;
  g->q_lo = (float)(q - (double)g->q_hi);
  g->grid = grid;
  g->inv_grid = grid > 0.0 ? 1.0 / grid : 0.0;
  g->tb = tb;
  g->te = te;
  g->nterms = nterms;
  const double k0 = floor(x_lo * g->inv_w), k1 = floor(x_hi * g->inv_w);
  if (!(k1 - k0 < 1e6) || !(fabs(k0) < 1e9)) return false;
  g->k0 = (int)k0;
  g->ncell = (int)(k1 - k0) + 1;
  g->ncoarse = (g->ncell + kCellK - 1) / kCellK;
  // Costs in term evaluations: a launch is worth about 4 us of them, a
  // polynomial 32 FP64 instructions.  The cells win as soon as the orbits
  // outnumber the nodes by enough to pay for the extra launches: 360 x 250,
  // tau rho = 120, mixed (22,806 orbits, 1936 nodes) 52 us direct, 30 us with
  // cells; 64^2, tau rho = 50 (561 orbits, 816 nodes) stays direct.
  const bool mixed = form == REXI_FORM_MIXED;
  const double launch = mixed ? 2.0e6 : 2.7e5, poly = mixed ? 27.0 : 4.0;
  const double near = std::min<double>(nterms, 5.0 * kCellK * g->c * g->inv_h);
  const double nodes = (double)g->ncell * kCellP;
  const double one = nodes * nterms;
  const double two = nodes * (near + 6.0) + (double)g->ncoarse * kCellPC * (nterms - near) + launch;
  g->two_level = two < one ? 1 : 0;
  return std::min(one, two) + poly * norb + launch < (double)norb * nterms;
}

size_t cell_scratch_values(const CellGeom& g) {
  return (size_t)g.ncell * kCellP + (size_t)g.ncoarse * kCellPC;
}

cudaError_t pole_cells(int form, const CellGeom& g, const CellTables& T, const void* table, double2* scratch,
                       const SymbolParams& sp, const OrbitParams& op, const FusedScalars& fs, OrbitOut kind,
                       void* fin, cudaStream_t s) {
  double2* poly = scratch;
  double2* far = scratch + (size_t)g.ncell * kCellP;
  const int f = form == REXI_FORM_MIXED ? (fs.exact_hn ? 1 : 2) : 0;
  cudaError_t e;
  if (g.two_level) {
    const dim3 grid(kCellPC / kFarWarps, (unsigned)g.ncoarse);
    auto k = f == 0 ? cell_far_kernel<0> : f == 1 ? cell_far_kernel<1> : cell_far_kernel<2>;
    k<<<grid, kFarWarps * 32, 0, s>>>(g, T, table, far);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  auto kp = f == 0 ? cell_poly_kernel<0> : f == 1 ? cell_poly_kernel<1> : cell_poly_kernel<2>;
  kp<<<(unsigned)g.ncell, kCellP * 16, 0, s>>>(g, T, table, far, poly);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  auto ko = kind == kOrbitFp64 ? cell_orbits_kernel<kOrbitFp64>
            : kind == kOrbitDf ? cell_orbits_kernel<kOrbitDf>
                               : cell_orbits_kernel<kOrbitRaw>;
  ko<<<(unsigned)((op.norb + 255) / 256), 256, 0, s>>>(g, poly, sp, op, fs.tau, make_double2(fs.R0re, fs.R0im), fin);
  return cudaGetLastError();
}

}  // namespace rexi
