// Kernels and dispatch of the pole sum by local expansion (pole_cells.cuh).
//
// What bounds it, and the split.  Direct sums cost orbits x terms evaluations
// of 62 FP32 operations (mixed) or 9 FP64 instructions; the cells cost nodes
// x near terms + coarse nodes x far terms.  The far kernel gives a block to
// each coarse node (24 per 32 cells), the cell kernel 8 or 32 lanes to each
// node, so that both have warps for every SM and short chains; what is left is
// one polynomial per orbit and the orbit's omega, where every FP64 instruction
// counts (one takes the time of about 60 FP32 ones).  Measured (GB300): 2048^2, tau rho = 1000, 525,825 orbits x 4067
// terms, direct 4286 us (mixed) and 32,902 us (FP64), cells 75 us and 185 us
// (166 and 225 us with 16 FP64 lanes per node and the library's root and
// division per orbit); the serving mix of 96 instances, mixed, 3088 us in the
// persistent kernel, 356 us with cells; 375 x 500, tau rho = 150, FP64, 47,188
// orbits x 667 terms, 521 us against 36 us.  Error against 64 bits as the direct sums' or smaller (shorter sums).
#include <math.h>

#include <algorithm>

#include "pole_cells.cuh"

namespace rexi {

namespace {

static_assert(kCellP == 16 && kCellPC % 2 == 0, "cell_poly's second part");
// Lanes per node: 8, or 32 up to this many cells, where a multiprocessor (152 of
// them) has less than four blocks and their chains of terms set the time (360 x 250,
// tau rho = 120, 121 cells x 547 terms).  Near the line: 400 cells (1024^2) 11.7 us
// with 32 lanes, 601 cells (512 x 384, scalar) 16.6 us with 8.
constexpr int kWideCells = 600;

template <int FORM>
__global__ void __launch_bounds__(kFarThreads) cell_far_kernel(CellGeom g, CellTables T,
                                                               const void* __restrict__ table, double2* far) {
  __shared__ double2 red[kFarThreads / 32];
  cell_far_node<FORM>(g, table, T, blockIdx.y, blockIdx.x, far, red);
}

template <int FORM, bool DF, int LANES>
__global__ void __launch_bounds__(LANES* kCellP) cell_poly_kernel(CellGeom g, CellTables T,
                                                                  const void* __restrict__ table,
                                                                  const double2* __restrict__ far, void* poly) {
  __shared__ CellShared<FORM> sh;
  cell_poly<FORM, DF, LANES>(g, table, T, blockIdx.x, far, poly, sh);
}
template <int LANES>
void launch_poly(int f, bool df, const CellGeom& g, const CellTables& T, const void* table, const double2* far,
                 void* poly, cudaStream_t s) {
  auto k = f == 0   ? (df ? cell_poly_kernel<0, true, LANES> : cell_poly_kernel<0, false, LANES>)
           : f == 1 ? (df ? cell_poly_kernel<1, true, LANES> : cell_poly_kernel<1, false, LANES>)
                    : (df ? cell_poly_kernel<2, true, LANES> : cell_poly_kernel<2, false, LANES>);
  k<<<(unsigned)g.ncell, LANES * kCellP, 0, s>>>(g, T, table, far, poly);
}

template <int KIND, bool CGRID>
__global__ void __launch_bounds__(256) cell_orbits_kernel(CellGeom g, const void* __restrict__ poly, SymbolParams sp,
                                                          OrbitParams op, double tau, double2 R0,
                                                          void* __restrict__ fin) {
  const int o = blockIdx.x * blockDim.x + threadIdx.x;
  if (o < op.norb) cell_orbit<KIND, CGRID>(g, poly, sp, op, tau, R0, o, fin);
}

// The same over the instances of a batch: a block looks its (instance, cell)
// up in a flat list.
template <bool MIXED>
__global__ void __launch_bounds__(kFarThreads) batch_far_kernel(const CellInst* __restrict__ inst,
                                                                const int2* __restrict__ list, CellTables T,
                                                                double2* scratch) {
  __shared__ double2 red[kFarThreads / 32];
  const int2 e = list[blockIdx.y];
  const CellInst& I = inst[e.x];
  double2* far = scratch + I.scratch_off + (size_t)I.g.ncell * kCellP;
  if (!MIXED)
    cell_far_node<0>(I.g, I.table, T, e.y, blockIdx.x, far, red);
  else if (I.exact_hn)
    cell_far_node<1>(I.g, I.table, T, e.y, blockIdx.x, far, red);
  else
    cell_far_node<2>(I.g, I.table, T, e.y, blockIdx.x, far, red);
}
template <bool MIXED>
__global__ void __launch_bounds__(8 * kCellP) batch_poly_kernel(const CellInst* __restrict__ inst,
                                                                const int2* __restrict__ list, CellTables T,
                                                                double2* scratch, int df) {
  const int2 e = list[blockIdx.x];
  const CellInst& I = inst[e.x];
  double2* poly = scratch + I.scratch_off;
  const double2* far = poly + (size_t)I.g.ncell * kCellP;
  const bool pairs = df && I.half_ok;
  if constexpr (!MIXED) {
    __shared__ CellShared<0> sh;
    cell_poly<0, false, 8>(I.g, I.table, T, e.y, far, poly, sh);
  } else if (I.exact_hn) {
    __shared__ CellShared<1> sh;
    if (pairs)
      cell_poly<1, true, 8>(I.g, I.table, T, e.y, far, poly, sh);
    else
      cell_poly<1, false, 8>(I.g, I.table, T, e.y, far, poly, sh);
  } else {
    __shared__ CellShared<2> sh;
    if (pairs)
      cell_poly<2, true, 8>(I.g, I.table, T, e.y, far, poly, sh);
    else
      cell_poly<2, false, 8>(I.g, I.table, T, e.y, far, poly, sh);
  }
}
__global__ void __launch_bounds__(256) batch_orbits_kernel(const CellInst* __restrict__ inst,
                                                           const int2* __restrict__ list,
                                                           const double2* __restrict__ scratch,
                                                           OrbitScalars* __restrict__ orb, int df) {
  const int2 e = list[blockIdx.x];
  const CellInst& I = inst[e.x];
  const int o = e.y + threadIdx.x;
  if (o >= I.op.norb) return;
  void* fin = orb + I.orb_off;
  if (df && I.half_ok)
    cell_orbit<kOrbitDf, true>(I.g, scratch + I.scratch_off, I.sp, I.op, I.tau, I.R0, o, fin);
  else
    cell_orbit<kOrbitFp64, true>(I.g, scratch + I.scratch_off, I.sp, I.op, I.tau, I.R0, o, fin);
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
                   double grid, int shared_launches, CellGeom* g) {
  if (nterms < 1 || !(q > 0.0) || !(x_hi >= x_lo)) return false;
  const double a = sqrt(q);
  g->c = ldexp(1.0, (int)floor(log2(a / 5.13)));
  if (!(g->c > 1e-12) || !(std::max(fabs(x_lo), fabs(x_hi)) < 1e8)) return false;
  g->w = 2.0 * g->c;
  g->inv_w = 1.0 / g->w;
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
  // Costs in term evaluations: a launch is worth about 4 us of them, a fiftieth of
  // that per instance of a batch (the mix of 96 shares each launch; small batches
  // gain too: two of 128^2, tau rho = 50, mixed 75 -> 52 us a step, two of 64^2 stay
  // direct; no batch of 1 to 8 instances tried was slower).  The cells win as soon as the orbits
  // outnumber the nodes by enough to pay for the extra launches: 360 x 250,
  // tau rho = 120, mixed (22,806 orbits, 1936 nodes) 52 us direct, 22 us with
  // cells; 64^2, tau rho = 50 (561 orbits, 816 nodes) stays direct.
  const bool mixed = form == REXI_FORM_MIXED;
  const double launch = (mixed ? 2.0e6 : 2.7e5) * (shared_launches ? 0.02 : 1.0);
  const double poly = mixed ? 12.0 : 6.0;  // an orbit's omega and polynomial
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
    auto k = f == 0 ? cell_far_kernel<0> : f == 1 ? cell_far_kernel<1> : cell_far_kernel<2>;
    k<<<dim3(kCellPC, (unsigned)g.ncoarse), kFarThreads, 0, s>>>(g, T, table, far);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  const bool df = kind == kOrbitDf;
  if (g.ncell <= kWideCells)
    launch_poly<32>(f, df, g, T, table, far, poly, s);
  else
    launch_poly<8>(f, df, g, T, table, far, poly, s);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const bool cgrid = sp.spectral == 0;
  auto ko = kind == kOrbitDf     ? cell_orbits_kernel<kOrbitDf, true>
            : kind == kOrbitRaw  ? cell_orbits_kernel<kOrbitRaw, false>
            : cgrid              ? cell_orbits_kernel<kOrbitFp64, true>
                                 : cell_orbits_kernel<kOrbitFp64, false>;
  ko<<<(unsigned)((op.norb + 255) / 256), 256, 0, s>>>(g, poly, sp, op, fs.tau, make_double2(fs.R0re, fs.R0im), fin);
  return cudaGetLastError();
}

cudaError_t pole_cells_batch(int form, const CellBatch& b, const CellTables& T, double2* scratch, void* orb, int df,
                             cudaStream_t s) {
  const bool mixed = form == REXI_FORM_MIXED;
  cudaError_t e;
  if (b.n_far > 0) {
    auto k = mixed ? batch_far_kernel<true> : batch_far_kernel<false>;
    k<<<dim3(kCellPC, (unsigned)b.n_far), kFarThreads, 0, s>>>(b.inst, b.far, T, scratch);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  auto k = mixed ? batch_poly_kernel<true> : batch_poly_kernel<false>;
  k<<<(unsigned)b.n_cell, 8 * kCellP, 0, s>>>(b.inst, b.cell, T, scratch, df);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  batch_orbits_kernel<<<(unsigned)b.n_orbit, 256, 0, s>>>(b.inst, b.orbit, scratch, static_cast<OrbitScalars*>(orb),
                                                          df);
  return cudaGetLastError();
}

}  // namespace rexi
