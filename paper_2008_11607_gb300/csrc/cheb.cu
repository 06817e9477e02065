// Variable-depth path, shared-Krylov method: the basis of span{f, A f, A^2 f,
// ...} taken as Chebyshev polynomials.
//
// K = -i dt A is self-adjoint in the energy inner product with spectrum in
// [-Lh, Lh], Lh = |dt| rho, and the step applies the scalar function r(ix) of
// the pole sum to it, so
//   r(dt A) f = sum_k c_k T_k(K / Lh) f,
// with c_k the Chebyshev coefficients of r(ix) on that interval: all poles
// together, in one basis that needs no inner products.  The tail sum_{k > K}
// |c_k| bounds the relative error in the energy norm.  r approximates e^{ix},
// whose coefficients 2 J_k(Lh) fall off super-exponentially beyond k = Lh: the
// degree K is Lh + O(Lh^(1/3)), the step count of the Lanczos recurrence, and
// is known on the host before the first launch.  With B = dt A / Lh,
// T_k(K / Lh) f = (-i)^k P_k with the real recurrence
//   P_{k+1} = 2 B P_k + P_{k-1},   P_0 = f, P_1 = B f,
// and d_k = (-i)^k c_k is real (r(-ix) = conj r(ix) over the full term set), so
// real input stays real and complex input is two real problems.  The sum runs
// as a Clenshaw recurrence,
//   b_k = d_k f + 2 B b_{k+1} + b_{k+2},  r(dt A) f = d_0 f + B b_1 + b_2,
// which keeps two vectors (b_k overwrites b_{k+2}), stores no basis and needs
// no second pass.  Against the Lanczos form: 13.9 -> 6.7 ms at 1024^2, tau rho =
// 400 (double-float), 4.35 -> 1.08 ms at 380 x 310, tau rho = 100 (FP64).
//
// Depth gradient: with mu_k the Clenshaw vectors of W^{-1} G for -dt (B^T = -W
// B W^{-1}), dL = sum_k c'_k <W mu_{k+1}, dB P_k> (c'_0 = 1, else 2), and H
// enters B only through its eta row, (dB P)_eta = -dH div P dt / Lh:
//   dL/dH = -w sum_k' mu_{k+1,eta} s_k,   s_k = (2 dt / Lh) div P_k (k = 0 halved):
// one pass forward that stores the scalar field s_k per step and one Clenshaw
// pass that consumes them, O(K nk) work where the two-sided Lanczos form
// contracts K x K pairs of basis vectors (8 steps with gradients at 512^2, tau
// rho = 200: 269 -> 47 ms).
//
// Unknowns are scaled, U = (2 dt / (Lh dx)) u, V = (2 dt / (Lh dy)) v, so that
// the divergence needs no products and each momentum row two.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "cheb.h"
#include "dfloat.cuh"

namespace rexi {
namespace {

constexpr int TX = 32, ROWS = 2, TYT = 8, TY = ROWS * TYT, THREADS = TX * TYT;

// ---- arithmetic: FP64, and double-float as unevaluated (hi, lo) pairs ------
// Sums of double-floats stay unnormalised inside a point's update (TwoSum of
// the high parts, low parts added in FP32); one FastTwoSum at its end.
__device__ __forceinline__ float2 u_add(float2 a, float2 b) {
  const float s = a.x + b.x, bb = s - a.x;
  return make_float2(s, ((a.x - (s - bb)) + (b.x - bb)) + (a.y + b.y));
}
__device__ __forceinline__ double u_add(double a, double b) { return a + b; }
__device__ __forceinline__ float2 u_sub(float2 a, float2 b) { return u_add(a, make_float2(-b.x, -b.y)); }
__device__ __forceinline__ double u_sub(double a, double b) { return a - b; }
// acc + x c
__device__ __forceinline__ float2 u_madd(float2 acc, float2 x, float2 c) {
  return u_add(acc, f_mul(x.x, x.y, c.x, c.y));
}
__device__ __forceinline__ double u_madd(double acc, double x, double c) { return fma(x, c, acc); }
__device__ __forceinline__ float2 u_norm(float2 a) { return f_fast(a.x, a.y); }
__device__ __forceinline__ double u_norm(double a) { return a; }
__device__ __forceinline__ float2 u_neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ double u_neg(double a) { return -a; }
__device__ __forceinline__ float2 u_half(float2 a) { return make_float2(0.5f * a.x, 0.5f * a.y); }
__device__ __forceinline__ double u_half(double a) { return 0.5 * a; }
__device__ __forceinline__ double u_to_double(float2 a) { return df_to_double(a); }
__device__ __forceinline__ double u_to_double(double a) { return a; }
template <typename T>
__device__ __forceinline__ T u_from(double v);
template <>
__device__ __forceinline__ double u_from<double>(double v) {
  return v;
}
template <>
__device__ __forceinline__ float2 u_from<float2>(double v) {
  return df_from_double(v);
}
inline float2 h_pair(double v, float2) { return df_split_host(v); }
inline double h_pair(double v, double) { return v; }

template <typename T>
struct Geom {
  int nx, ny;
  size_t nk;
  T cu, gu, cv, gv;  // momentum rows: U <- cu V4 - gu dx(eta), V <- -(cv U4) - gv dy(eta)
  double su, sv;     // U = su u, V = sv v
  double isu, isv;
};

__device__ __forceinline__ int wrap(int i, int n, int t) {
  return n > t ? (i < 0 ? i + n : (i >= n ? i - n : i)) : (i + n) % n;
}
__device__ __forceinline__ void cp_async8(void* smem, const void* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ---- coefficients ----------------------------------------------------------

// 1 / x for normal FP64 x: hardware seed, r0 (1 + e + e^2) with e = 1 - x r0.
__device__ __forceinline__ double rcp64(double x) {
  double r0;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r0) : "d"(x));
  const double e = fma(-x, r0, 1.0);
  return fma(r0, fma(e, e, e), r0);
}

constexpr int NT = 128;

struct Term {
  double x, y, z, w;
};

// r(ix) at the nodes x_j = Lh cos((j + 1/2) pi / n) >= 0, j < n / 2, one block
// per node.  terms[m] = (c1 h mu, c2) of term m >= 0; term -m has (conj c1, -conj c2).
__global__ void __launch_bounds__(NT) cheb_nodes(const Term* terms, int N, double h, double hmu, double Lh, int n,
                                                 double2* val) {
  __shared__ double2 red[NT / 32];
  const int j = blockIdx.x;
  const double x = Lh * cospi((j + 0.5) / n), q = hmu * hmu;
  double re = 0.0, im = 0.0;
  for (int m = threadIdx.x; m <= N; m += NT) {
    const Term t = terms[m];
    const double y = fma(h, (double)m, x), r = rcp64(fma(y, y, q));
    re = fma(fma(t.z, y, t.x), r, re);
    im = fma(fma(t.w, y, t.y), r, im);
    if (m) {
      const double z = fma(-h, (double)m, x), p = rcp64(fma(z, z, q));
      re = fma(fma(-t.z, z, t.x), p, re);
      im = fma(fma(t.w, z, -t.y), p, im);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    re += __shfl_down_sync(0xffffffffu, re, o);
    im += __shfl_down_sync(0xffffffffu, im, o);
  }
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = make_double2(re, im);
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < NT / 32; ++i) {
      re += red[i].x;
      im += red[i].y;
    }
    val[j] = make_double2(re, im);
  }
}

// d_k = (-1)^(k/2) (4/n) sum_{j < n/2} v_j cos(k (j + 1/2) pi / n), v the real
// part of r for even k and the imaginary part for odd k (halved at k = 0).
__global__ void __launch_bounds__(NT) cheb_coeffs(const double2* val, int n, double* d, float2* d_df) {
  __shared__ double red[NT / 32];
  const int k = blockIdx.x;
  double a = 0.0;
  for (int j = threadIdx.x; j < n / 2; j += NT) {
    const long long m = (long long)k * (2 * j + 1) % (4 * n);
    a = fma((k & 1) ? val[j].y : val[j].x, cospi((double)m / (2.0 * n)), a);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = a;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < NT / 32; ++i) a += red[i];
    a *= ((k >> 1) & 1 ? -1.0 : 1.0) * (k ? 4.0 : 2.0) / n;
    d[k] = a;
    d_df[k] = df_from_double(a);
  }
}

// report = (sum_{K < k < n} |d_k|, high word of the largest |input|)
__global__ void __launch_bounds__(32) cheb_report(const double* d, int K, int n, const unsigned* maxbits,
                                                  double* report) {
  double a = 0.0;
  for (int k = K + 1 + threadIdx.x; k < n; k += 32) a += fabs(d[k]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
  if (threadIdx.x == 0) {
    report[0] = a;
    report[1] = (double)*maxbits;
  }
}

// ---- vectors ---------------------------------------------------------------

// F = in in scaled unknowns (eta / w for the adjoint); bK = d_K F when bK is
// given; maxbits = high word of the largest |value| (integer maximum: infinities
// and NaN come out above every finite value).  blockIdx.y: real part, imaginary part.
template <typename T>
__global__ void __launch_bounds__(256) cheb_init(Geom<T> G, const double2* in, const double* w, int adjoint, T* F, T* bK,
                                                 const T* dK, unsigned* maxbits) {
  const size_t i = (size_t)blockIdx.x * 256 + threadIdx.x;
  unsigned hi = 0u;
  if (i < 3 * G.nk) {
    const double2 z = in[i];
    double v = blockIdx.y ? z.y : z.x;
    const int c = i < G.nk ? 0 : (i < 2 * G.nk ? 1 : 2);
    if (c == 0) {
      if (adjoint) v /= w[i];
    } else {
      v *= c == 1 ? G.su : G.sv;
    }
    hi = (unsigned)__double2hiint(v) & 0x7fffffffu;
    const T f = u_from<T>(v);
    const size_t o = i + blockIdx.y * 3 * G.nk;
    F[o] = f;
    if (bK) bK[o] = u_norm(u_madd(T{}, f, *dK));
  }
  hi = __reduce_max_sync(0xffffffffu, hi);
  if ((threadIdx.x & 31) == 0 && hi) atomicMax(maxbits, hi);
}

enum StepMode { kSum = 0, kSumLast, kGrad, kGradLast, kForward, kForwardFirst };

template <typename T>
struct StepArgs {
  const T *b1, *b2;  // b_{k+1}, b_{k+2} (null: zero); forward: P_k, P_{k-1}
  T* bout;           // may be b2
  const T* F;
  const T* H;
  const T* d;        // d_k of this step
  T* s;              // forward: s_k out; gradient: s_k in
  T* acc;            // gradient: sum of mu_{k+1,eta} s_k (first: starts it)
  int first;
  double2* out;      // last: the step's output
  double* grad;      // last: the depth gradient
  const double* w;
  int adjoint, real_out;
};

// One step of the recurrence on a tile of TX x TY points, two rows per thread.
// The tile and the halo sides that the stencil reads go to shared memory by
// asynchronous copies; pair sums of the Coriolis averages and the row's eta are
// carried in registers from one row to the next.  Point-wise operands that no
// running launch writes (F, H, s, and b2, two launches old) are loaded before the
// wait for the previous step.
template <typename T, int MODE>
__global__ void __launch_bounds__(THREADS, 4) cheb_step_kernel(Geom<T> G, StepArgs<T> A) {
  constexpr bool LAST = MODE == kSumLast || MODE == kGradLast, FWD = MODE == kForward || MODE == kForwardFirst;
  constexpr bool GRAD = MODE == kGrad || MODE == kGradLast, HALF = LAST || MODE == kForwardFirst;
  __shared__ T E[TY + 1][TX + 1], U[TY + 1][TX + 1], V[TY + 1][TX + 1];
  const size_t nk = G.nk, set = (size_t)blockIdx.z * 3 * nk;
  const int i0 = blockIdx.x * TX, j0 = blockIdx.y * TY;
  const int tx = threadIdx.x % TX, ty = threadIdx.x / TX;
  const int i = i0 + tx;
  T pb[ROWS][3], pf[ROWS][3], pH[ROWS], ps[ROWS];
#pragma unroll
  for (int r = 0; r < ROWS; ++r) {
    const int j = j0 + ty * ROWS + r;
    const bool live = i < G.nx && j < G.ny;
    const size_t id = live ? (size_t)j * G.nx + i : 0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      pb[r][c] = A.b2 ? A.b2[set + id + c * nk] : T{};
      if (!FWD) pf[r][c] = A.F[set + id + c * nk];
    }
    pH[r] = A.H[id];
    if (GRAD) ps[r] = A.s[id];
  }
  pdl_wait();
  pdl_release();
  const T* b1 = A.b1 + set;
  for (int q = threadIdx.x; q < (TY + 1) * (TX + 1); q += THREADS) {
    const int c = q % (TX + 1), r = q / (TX + 1);
    const size_t row = (size_t)wrap(j0 + r, G.ny, TY) * G.nx, rowm = (size_t)wrap(j0 + r - 1, G.ny, TY) * G.nx;
    const int ic = wrap(i0 + c, G.nx, TX), im = wrap(i0 + c - 1, G.nx, TX);
    cp_async8(&E[r][c], b1 + row + ic);
    cp_async8(&U[r][c], b1 + nk + row + im);
    cp_async8(&V[r][c], b1 + 2 * nk + rowm + ic);
  }
  T dk = T{};
  if (!FWD) dk = *A.d;
  cp_async_wait_all();
  __syncthreads();
  const T cu = HALF ? u_half(G.cu) : G.cu, gu = HALF ? u_half(G.gu) : G.gu;
  const T cv = HALF ? u_half(G.cv) : G.cv, gv = HALF ? u_half(G.gv) : G.gv;
  const int r0 = ty * ROWS;
  T e = E[r0][tx], u = U[r0][tx + 1], vs = V[r0][tx];
  T du = u_sub(u, U[r0][tx]), su = u_add(u, U[r0][tx]);  // of row j
  T sv = u_add(vs, V[r0][tx + 1]);                       // of row j - 1
#pragma unroll
  for (int r = 0; r < ROWS; ++r) {
    const int j = j0 + r0 + r;
    const T en = E[r0 + r + 1][tx], un = U[r0 + r + 1][tx + 1], unw = U[r0 + r + 1][tx];
    const T v = V[r0 + r + 1][tx];
    const T svn = u_add(v, V[r0 + r + 1][tx + 1]);
    const T s = u_add(du, u_sub(v, vs));
    T a0 = pb[r][0], a1 = pb[r][1], a2 = pb[r][2];
    if (!FWD) {
      a0 = u_madd(a0, pf[r][0], dk);
      a1 = u_madd(a1, pf[r][1], dk);
      a2 = u_madd(a2, pf[r][2], dk);
    }
    a0 = u_norm(u_madd(a0, s, u_neg(HALF ? u_half(pH[r]) : pH[r])));
    a1 = u_madd(a1, u_add(sv, svn), cu);
    a1 = u_norm(u_madd(a1, u_sub(E[r0 + r][tx + 1], e), u_neg(gu)));
    const T sun = u_add(un, unw);
    a2 = u_madd(a2, u_add(su, sun), u_neg(cv));
    a2 = u_norm(u_madd(a2, u_sub(en, e), u_neg(gv)));
    if (i < G.nx && j < G.ny) {
      const size_t id = (size_t)j * G.nx + i, o = set + id;
      if (!LAST) {
        A.bout[o] = a0;
        A.bout[o + nk] = a1;
        A.bout[o + 2 * nk] = a2;
      }
      if (FWD) A.s[id] = u_norm(s);
      if (GRAD) {
        const T es = LAST ? u_half(e) : e;
        const T t = u_norm(u_madd(A.first ? T{} : A.acc[id], es, ps[r]));
        if (MODE == kGrad)
          A.acc[id] = t;
        else
          A.grad[id] -= A.w[id] * u_to_double(t);
      }
      if (MODE == kSumLast || (MODE == kGradLast && A.out)) {
        double o0 = u_to_double(a0), o1 = u_to_double(a1) * G.isu, o2 = u_to_double(a2) * G.isv;
        if (A.adjoint) o0 *= A.w[id];
        if (A.real_out) {
          A.out[id] = make_double2(o0, 0.0);
          A.out[id + nk] = make_double2(o1, 0.0);
          A.out[id + 2 * nk] = make_double2(o2, 0.0);
        } else {
          double* p = reinterpret_cast<double*>(A.out) + blockIdx.z;
          p[2 * id] = o0;
          p[2 * (id + nk)] = o1;
          p[2 * (id + 2 * nk)] = o2;
        }
      }
    }
    e = en;
    du = u_sub(un, unw);
    su = sun;
    sv = svn;
    vs = v;
  }
}

// Launch that may overlap the previous step's tail (see pdl_wait); an error is
// left for the caller's cudaGetLastError.
template <typename T, int MODE>
void launch_step(const Geom<T>& G, const StepArgs<T>& A, int nset, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((G.nx + TX - 1) / TX, (G.ny + TY - 1) / TY, nset);
  cfg.blockDim = dim3(THREADS);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, cheb_step_kernel<T, MODE>, G, A);
}

// Smallest K with 2 sum_{k > K} |J_k(x)| <= target: Miller's downward
// recurrence, normalised by J_0 + 2 sum J_2m = 1.
int bessel_degree(double x, double target) {
  const int top = (int)std::ceil(x + 30.0 + 16.0 * std::cbrt(x));
  std::vector<double> J(top + 2, 0.0);
  J[top] = 1e-280;
  for (int k = top; k > 0; --k) {
    J[k - 1] = 2.0 * k / x * J[k] - J[k + 1];
    if (std::fabs(J[k - 1]) > 1e200)
      for (int m = k - 1; m <= top; ++m) J[m] *= 1e-250;
  }
  double norm = J[0];
  for (int k = 2; k <= top; k += 2) norm += 2.0 * J[k];
  double tail = 0.0;
  int K = top;
  for (; K > 2; --K) {
    tail += 2.0 * std::fabs(J[K] / norm);
    if (tail > target) break;
  }
  return K;
}

struct Scratch {
  Term* terms;
  double2* val;
  double* d;
  float2* d_df;
  double* report;
  unsigned* maxbits;
};
size_t al(size_t v) { return (v + 255) / 256 * 256; }
size_t carve(const ChebPlan& p, int N, char* base, Scratch* S) {
  size_t o = 0;
  auto take = [&](size_t bytes) {
    char* at = base + o;
    o += al(bytes);
    return at;
  };
  S->terms = reinterpret_cast<Term*>(take((size_t)(N + 1) * sizeof(Term)));
  S->val = reinterpret_cast<double2*>(take((size_t)p.n / 2 * sizeof(double2)));
  S->d = reinterpret_cast<double*>(take((size_t)p.n * sizeof(double)));
  S->d_df = reinterpret_cast<float2*>(take((size_t)p.n * sizeof(float2)));
  S->report = reinterpret_cast<double*>(take(2 * sizeof(double)));
  S->maxbits = reinterpret_cast<unsigned*>(take(sizeof(unsigned)));
  return o;
}

inline const double* coeff_table(const Scratch& S, double) { return S.d; }
inline const float2* coeff_table(const Scratch& S, float2) { return S.d_df; }
inline const double* depth_table(const KrylovSettings* k, double) { return k->depth; }
inline const float2* depth_table(const KrylovSettings* k, float2) { return k->Hdf; }

cudaError_t coefficients(const ChebPlan& p, double h, int M, const Scratch& S, cudaStream_t s, int64_t* launches) {
  TermSet ts;
  rexii_terms(M, h, &ts);
  const int N = ts.N;
  const double hmu = h * ts.mu;
  std::vector<Term> t(N + 1);
  for (int m = 0; m <= N; ++m)
    t[m] = Term{ts.c1re[N + m] * hmu, ts.c1im[N + m] * hmu, ts.c2re[N + m], ts.c2im[N + m]};
  cudaError_t e = cudaMemcpyAsync(S.terms, t.data(), t.size() * sizeof(Term), cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return e;
  cheb_nodes<<<p.n / 2, NT, 0, s>>>(S.terms, N, h, hmu, p.Lh, p.n, S.val);
  cheb_coeffs<<<p.n, NT, 0, s>>>(S.val, p.n, S.d, S.d_df);
  *launches += 2;
  return cudaGetLastError();
}

template <typename T>
Geom<T> make_geom(const KrylovSettings* k, double tau, const ChebPlan& p) {
  Geom<T> G;
  G.nx = k->nx;
  G.ny = k->ny;
  G.nk = (size_t)k->nx * k->ny;
  const double idx = k->nx / k->Lx, idy = k->ny / k->Ly, t2 = std::copysign(p.t2, tau);
  G.su = t2 * idx;
  G.sv = t2 * idy;
  G.isu = 1.0 / G.su;
  G.isv = 1.0 / G.sv;
  G.cu = h_pair(0.25 * t2 * k->f * (idx / idy), T{});
  G.cv = h_pair(0.25 * t2 * k->f * (idy / idx), T{});
  G.gu = h_pair(k->g * G.su * G.su, T{});
  G.gv = h_pair(k->g * G.sv * G.sv, T{});
  return G;
}

template <typename T>
cudaError_t init(const Geom<T>& G, const KrylovSettings* k, const void* in, int adjoint, T* F, T* bK, const T* dK,
                 const Scratch& S, int nset, cudaStream_t s, int64_t* launches) {
  cudaError_t e = cudaMemsetAsync(S.maxbits, 0, sizeof(unsigned), s);
  if (e != cudaSuccess) return e;
  cheb_init<T><<<dim3((unsigned)((3 * G.nk + 255) / 256), nset), 256, 0, s>>>(
      G, static_cast<const double2*>(in), k->w64, adjoint, F, bK, dK, S.maxbits);
  ++*launches;
  return cudaGetLastError();
}
cudaError_t report(KrylovSettings* k, const ChebPlan& p, const Scratch& S, int slot, cudaStream_t s,
                   int64_t* launches) {
  cheb_report<<<1, 32, 0, s>>>(S.d, p.K, p.n, S.maxbits, S.report);
  ++*launches;
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(k->pinned + 2 * slot, S.report, 2 * sizeof(double), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaEventRecord(k->ev[slot], s);
  return e;
}
// Whether the expansion stands: tail within rtol, and the input zero or of a
// size that the arithmetic holds with room on both sides (exponents of +-64 for
// double-float, +-900 for FP64).  Other input, NaN and infinities included, is
// left to the Lanczos form, which normalises its vectors and reports what is
// not finite.
cudaError_t accepted(KrylovSettings* k, int df, int slot, bool* ok, double* bound) {
  const cudaError_t e = cudaEventSynchronize(k->ev[slot]);
  if (e != cudaSuccess) return e;
  const double tail = k->pinned[2 * slot];
  const unsigned hi = (unsigned)k->pinned[2 * slot + 1];
  const int room = df ? 64 : 900, ex = (int)(hi >> 20) - 1023;
  *ok = tail <= k->rtol && (hi == 0u || (ex >= -room && ex <= room));
  *bound = std::max(*bound, tail);
  return cudaSuccess;
}
rexi_status failed(cudaError_t e) {
  set_last_error(cudaGetErrorString(e));
  return REXI_ECUDA;
}

// The Clenshaw steps k = K - 1 .. 1 on F with b_K in bA; the two newest
// vectors are left in *b1 (b_1) and *b2 (b_2, null when K = 1).
template <typename T, int MODE>
void clenshaw(const Geom<T>& G, StepArgs<T> A, int K, const T* d, T* bA, T* bB, const T* sfield, int nset,
              cudaStream_t s, const T** b1, const T** b2) {
  T *cur = bA, *old = bB;
  bool have_old = false;
  for (int k = K - 1; k >= 1; --k) {
    A.b1 = cur;
    A.b2 = have_old ? old : nullptr;
    A.bout = old;
    A.d = d + k;
    if (MODE == kGrad) A.s = const_cast<T*>(sfield) + (size_t)k * G.nk;
    launch_step<T, MODE>(G, A, nset, s);
    A.first = 0;
    std::swap(cur, old);
    have_old = true;
  }
  *b1 = cur;
  *b2 = have_old ? old : nullptr;
}

template <typename T>
rexi_status step_impl(KrylovSettings* k, const ChebPlan& p, double h, int M, const void* in, void* out, double dt,
                      int real_input, bool adjoint, const ChebBuffers& b, cudaStream_t s, const KrylovHooks& hooks,
                      double* bound) {
  auto mark = [&](int i) {
    if (hooks.mark) hooks.mark(hooks.ctx, i, s);
  };
  int64_t launches = 0;
  const int nset = real_input ? 1 : 2;
  const Geom<T> G = make_geom<T>(k, adjoint ? -dt : dt, p);
  Scratch S;
  carve(p, M + kL, static_cast<char*>(b.scratch), &S);
  T *F = static_cast<T*>(b.f0), *bA = static_cast<T*>(b.bA), *bB = static_cast<T*>(b.bB);
  const T* d = coeff_table(S, T{});
  mark(0);
  cudaError_t e = coefficients(p, h, M, S, s, &launches);
  mark(1);
  if (e == cudaSuccess) e = init(G, k, in, adjoint ? 1 : 0, F, bA, d + p.K, S, nset, s, &launches);
  if (e == cudaSuccess) e = report(k, p, S, 0, s, &launches);
  if (e != cudaSuccess) return failed(e);
  StepArgs<T> A = {};
  A.F = F;
  A.H = depth_table(k, T{});
  const T *b1, *b2;
  clenshaw<T, kSum>(G, A, p.K, d, bA, bB, nullptr, nset, s, &b1, &b2);
  launches += p.K - 1;
  mark(2);
  mark(3);
  // the host looks at the tail and the input while the steps run; `out` is
  // written by the last step only
  bool ok = false;
  e = accepted(k, std::is_same<T, float2>::value, 0, &ok, bound);
  if (e != cudaSuccess) return failed(e);
  if (ok) {
    A.b1 = b1;
    A.b2 = b2;
    A.d = d;
    A.out = static_cast<double2*>(out);
    A.w = k->w64;
    A.adjoint = adjoint ? 1 : 0;
    A.real_out = real_input;
    launch_step<T, kSumLast>(G, A, nset, s);
    ++launches;
  }
  mark(4);
  if (hooks.launches) *hooks.launches += launches;
  e = cudaGetLastError();
  if (e != cudaSuccess) return failed(e);
  return ok ? REXI_OK : REXI_EUNSUPPORTED;
}

template <typename T>
rexi_status grad_impl(KrylovSettings* k, const ChebPlan& p, double h, int M, const void* f_in, const void* g_out,
                      double* grad_depth, double dt, const ChebGradBuffers& b, cudaStream_t s,
                      const KrylovHooks& hooks, double* bound) {
  auto mark = [&](int i) {
    if (hooks.mark) hooks.mark(hooks.ctx, i, s);
  };
  int64_t launches = 0;
  Scratch S;
  carve(p, M + kL, static_cast<char*>(b.scratch), &S);
  T *F = static_cast<T*>(b.f0), *bA = static_cast<T*>(b.bA), *bB = static_cast<T*>(b.bB);
  T* sf = static_cast<T*>(b.div);
  const T* d = coeff_table(S, T{});
  const int df = std::is_same<T, double>::value ? 0 : 1;
  mark(0);
  cudaError_t e = coefficients(p, h, M, S, s, &launches);
  mark(1);
  // forward: P_0 in bA, P_1 in bB, then each P_{k+1} over P_{k-1}; s_k for k < K
  Geom<T> G = make_geom<T>(k, dt, p);
  if (e == cudaSuccess) e = init(G, k, f_in, 0, bA, static_cast<T*>(nullptr), d, S, 1, s, &launches);
  if (e == cudaSuccess) e = report(k, p, S, 0, s, &launches);
  if (e != cudaSuccess) return failed(e);
  {
    StepArgs<T> A = {};
    A.H = depth_table(k, T{});
    T *cur = bA, *old = bB;
    for (int j = 0; j < p.K; ++j) {
      A.b1 = cur;
      A.b2 = j ? old : nullptr;
      A.bout = old;
      A.s = sf + (size_t)j * G.nk;
      if (j == 0)
        launch_step<T, kForwardFirst>(G, A, 1, s);
      else
        launch_step<T, kForward>(G, A, 1, s);
      std::swap(cur, old);
    }
  }
  launches += p.K;
  // backward: the Clenshaw vectors of W^{-1} G under -dt, each step taking its s_k
  G = make_geom<T>(k, -dt, p);
  e = init(G, k, g_out, 1, F, bA, d + p.K, S, 1, s, &launches);
  if (e == cudaSuccess) e = report(k, p, S, 1, s, &launches);
  if (e != cudaSuccess) return failed(e);
  StepArgs<T> A = {};
  A.F = F;
  A.H = depth_table(k, T{});
  A.acc = static_cast<T*>(b.acc);
  A.first = 1;
  const T *b1, *b2;
  clenshaw<T, kGrad>(G, A, p.K, d, bA, bB, sf, 1, s, &b1, &b2);
  launches += p.K - 1;
  mark(2);
  mark(3);
  bool okf = false, okg = false;
  e = accepted(k, df, 0, &okf, bound);
  if (e == cudaSuccess) e = accepted(k, df, 1, &okg, bound);
  if (e != cudaSuccess) return failed(e);
  if (okf && okg) {
    A.first = 0;
    A.b1 = b1;
    A.b2 = b2;
    A.d = d;
    A.s = sf;
    A.grad = grad_depth;
    A.w = k->w64;
    launch_step<T, kGradLast>(G, A, 1, s);
    ++launches;
  }
  mark(4);
  if (hooks.launches) *hooks.launches += launches;
  e = cudaGetLastError();
  if (e != cudaSuccess) return failed(e);
  return okf && okg ? REXI_OK : REXI_EUNSUPPORTED;
}

}  // namespace

// The expansion replaces the Lanczos form where its degree is that of e^{ix}:
//  - the bound rho holds for the plan's operator (an overridden rho may not),
//  - the tolerance is one that FP64 coefficients reach (their sum carries
//    rounding of 1e-14),
//  - the spacing h makes r a smooth multiple of e^{ix}: the pole sum's alias
//    e^{i (1 - 2 pi / h) x} has amplitude e^{h^2 - (2 pi - h)^2} (4e-15 at
//    h = 0.5, 6e-7 at h = 2), whose coefficients reach up to 2 pi / h times Lh,
//  - the degree keeps to the caller's step cap.
// The coefficients found on the device are checked again (accepted()).  Partial
// sums of terms have single poles' convergence, (1 + h |mu| / Lh)^-k, and stay
// with the Lanczos form.
bool cheb_plan(const KrylovSettings* k, double h, int M, double dt, double target, ChebPlan* p) {
  if (!(k->rho_op > 0.0)) return false;
  // 2 / rho cut to 12 bits (the interval grows by 5e-4 at most): on unit-square
  // grids the scaled stencil's constants are then exact in double-float too, and
  // a small change of the depth leaves them and the coefficients as they are
  // (differences of nearby problems see no rounding of theirs)
  int ex;
  p->t2 = std::frexp(2.0 / k->rho_op, &ex);
  p->t2 = std::ldexp(std::floor(std::ldexp(p->t2, 12)), ex - 12);
  const double Lh = 2.0 * std::fabs(dt) / p->t2;
  if (k->rho_bound < k->rho_op || !(Lh >= 1e-6) || Lh > 1e6) return false;
  if (k->rtol < 1e-13 || std::exp(h * h - (2.0 * M_PI - h) * (2.0 * M_PI - h)) > 0.05 * k->rtol) return false;
  if (M * h < std::fabs(dt) * k->rho_op) return false;
  p->Lh = Lh;
  p->K = std::max(2, bessel_degree(Lh, target));
  if (p->K > k->max_iters) return false;
  p->n = (p->K + 1 + 32 + p->K / 16 + 1) / 2 * 2;
  return true;
}

size_t cheb_scratch_bytes(const ChebPlan& p, int N) {
  Scratch S;
  return carve(p, N, nullptr, &S);
}

rexi_status cheb_step(KrylovSettings* k, const ChebPlan& p, int df, double h, int M, const void* in, void* out,
                      double dt, int real_input, bool adjoint, const ChebBuffers& b, cudaStream_t s,
                      const KrylovHooks& hooks, double* bound) {
  *bound = 0.0;
  return df ? step_impl<float2>(k, p, h, M, in, out, dt, real_input, adjoint, b, s, hooks, bound)
            : step_impl<double>(k, p, h, M, in, out, dt, real_input, adjoint, b, s, hooks, bound);
}

rexi_status cheb_grad(KrylovSettings* k, const ChebPlan& p, int df, double h, int M, const void* f_in,
                      const void* g_out, double* grad_depth, double dt, const ChebGradBuffers& b, cudaStream_t s,
                      const KrylovHooks& hooks, double* bound) {
  *bound = 0.0;
  return df ? grad_impl<float2>(k, p, h, M, f_in, g_out, grad_depth, dt, b, s, hooks, bound)
            : grad_impl<double>(k, p, h, M, f_in, g_out, grad_depth, dt, b, s, hooks, bound);
}

}  // namespace rexi
