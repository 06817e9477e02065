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
// 400 (double-float), 4.35 -> 0.77 ms at 380 x 310, tau rho = 100 (FP64).
//
// Depth gradient: with mu_k the Clenshaw vectors of W^{-1} G for -dt (B^T = -W
// B W^{-1}), dL = sum_k c'_k <W mu_{k+1}, dB P_k> (c'_0 = 1, else 2), and H
// enters B only through its eta row, (dB P)_eta = -dH div P dt / Lh:
//   dL/dH = -w sum_k' mu_{k+1,eta} s_k,   s_k = (2 dt / Lh) div P_k (k = 0 halved):
// one pass forward that stores the scalar field s_k per step and one Clenshaw
// pass that consumes them, O(K nk) work where the two-sided Lanczos form
// contracts K x K pairs of basis vectors (8 steps with gradients at 512^2, tau
// rho = 200: 269 -> 27 ms).
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
#include "recip.cuh"

namespace rexi {
namespace {

constexpr int TX = 32, ROWS = 2, TYT = 8, TY = ROWS * TYT, THREADS = TX * TYT;

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

// report = (sum_{K < k < n} |d_k|, whether the expansion stands), *declined = 1 where
// it does not.  It stands with a tail within rtol and input that is zero or of a
// size that the arithmetic holds with room on both sides (exponents of +-room: 64
// for double-float, 900 for FP64).  Other input, NaN and infinities included, is
// left to the Lanczos form, which normalises its vectors and reports what is not
// finite.
__global__ void __launch_bounds__(32) cheb_report(const double* d, int K, int n, const unsigned* maxbits, double rtol,
                                                  int room, double* report, unsigned* declined) {
  double a = 0.0;
  for (int k = K + 1 + threadIdx.x; k < n; k += 32) a += fabs(d[k]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
  if (threadIdx.x == 0) {
    const unsigned hi = *maxbits;  // high word of the largest |input|
    const int ex = (int)(hi >> 20) - 1023;
    const bool ok = a <= rtol && (hi == 0u || (ex >= -room && ex <= room));
    report[0] = a;
    report[1] = ok ? 1.0 : 0.0;
    if (!ok) *declined = 1u;
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
  const unsigned* bad;  // last: nonzero where an earlier launch gave up: out is NaN, grad untouched
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
  const bool gone = LAST && A.bad && *A.bad;
  if (gone) dk = u_from<T>(nan(""));
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
        else if (!gone)
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

// Launch that may overlap the previous step's tail (see pdl_wait; not behind a
// launch of many steps, which wrote what this one loads early).  An error is
// left for the caller's cudaGetLastError.
template <typename T, int MODE>
void launch_step(const Geom<T>& G, const StepArgs<T>& A, int nset, cudaStream_t s, bool overlap = true) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((G.nx + TX - 1) / TX, (G.ny + TY - 1) / TY, nset);
  cfg.blockDim = dim3(THREADS);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = overlap ? 1 : 0;
  cudaLaunchKernelEx(&cfg, cheb_step_kernel<T, MODE>, G, A);
}

// ---- many steps in one launch ------------------------------------------------
//
// Steps on grids whose vectors fit the multiprocessors' shared memory: every
// block keeps a tile (b_{k+1}, b_{k+2}, F, H with a halo) there for all steps and
// passes only its edge values to its neighbours.  An edge value travels through
// L2 as two 64-bit words, each 32 bits of it and the step's number, so that the
// reader polls the value itself: no flag and no fence on the way.  The tile's
// edge is computed first; while the compute warps work on the interior, the
// last kCommWarps warps publish the edge, poll the neighbours' and fill the next
// step's halo, so a step costs the longer of the two.  Two slots per edge
// value, by the parity of the step: a block overwrites a slot only after it has
// the next step's edges of every reader (west / east, south / north and the two
// corners that the Coriolis averages touch are neighbours in both directions).
// A launch per step costs 2.2 us however small the grid, and moves 13 values per
// point through L2.  Per step, one launch each -> tiles: 512^2 double-float 4.93
// -> 2.54 us, 256^2 2.47 -> 1.73, 96 x 80 2.56 -> 1.7; 380 x 310 FP64 7.36 -> 5.2
// (FP64 pipe: 3.8 us at its peak rate), 100 x 90 4.49 -> 2.4.  What is left at
// 512^2 is issue (3.15 of 4 instructions per cycle, 224 of 332 per point on the
// FMA pipe before a task took two rows); below 256^2 it is the way of an edge
// value through L2, 1.2 us.
struct Exchange {
  ulonglong2* col;        // [parity][set][3][strip][ny], then rows [parity][set][3][group][nx]
  unsigned* bad;          // a wait ran out
  unsigned* host_bad;     // the same for the host (KrylovSettings::gave_up)
  int polls;              // of one wait before a warp gives up
};
enum { kColE = 0, kColV = 1, kColU = 2, kRowE = 0, kRowU = 1, kRowV = 2 };

__device__ __forceinline__ ulonglong2 pack(float2 v, unsigned flag) {
  const unsigned long long f = (unsigned long long)flag << 32;
  return make_ulonglong2(f | __float_as_uint(v.x), f | __float_as_uint(v.y));
}
__device__ __forceinline__ ulonglong2 pack(double v, unsigned flag) {
  const unsigned long long f = (unsigned long long)flag << 32;
  return make_ulonglong2(f | (unsigned)__double2loint(v), f | (unsigned)__double2hiint(v));
}
template <typename T>
__device__ __forceinline__ T unpack(ulonglong2 w);
template <>
__device__ __forceinline__ float2 unpack<float2>(ulonglong2 w) {
  return make_float2(__uint_as_float((unsigned)w.x), __uint_as_float((unsigned)w.y));
}
template <>
__device__ __forceinline__ double unpack<double>(ulonglong2 w) {
  return __hiloint2double((int)(unsigned)w.y, (int)(unsigned)w.x);
}
__device__ __forceinline__ void st_edge(ulonglong2* p, ulonglong2 w) {
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(w.x), "l"(w.y) : "memory");
}
__device__ __forceinline__ ulonglong2 ld_edge(const ulonglong2* p) {
  ulonglong2 w;
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(w.x), "=l"(w.y) : "l"(p) : "memory");
  return w;
}
__device__ __forceinline__ bool arrived(ulonglong2 w, unsigned flag) {
  return (unsigned)(w.x >> 32) == flag && (unsigned)(w.y >> 32) == flag;
}
// Out of line: its stores inside the poll loop cost 0.8% of a 512^2 step.
__device__ __noinline__ void give_up(const Exchange& X, unsigned* dead) {
  *(volatile unsigned*)X.bad = 1u;
  *(volatile unsigned*)X.host_bad = 1u;
  *(volatile unsigned*)dead = 1u;
}

template <typename T>
struct ManyArgs {
  const T *b1, *b2;  // newest vectors (b2 null: zero)
  T *o1, *o2;        // where the newest two go at the end (null: nowhere)
  const T *F, *H, *d;  // d: coefficient of the first step, descending
  T* s;              // kForward: s of the first step, ascending; kGrad: of the first step, descending
  T* acc;            // kGrad: sum of mu_eta s (written)
  int steps, nset, ns, ng, seg_shift;
  unsigned flag0;    // flags of earlier launches on this exchange buffer end here
  const unsigned* declined;  // nonzero: the expansion does not stand (cheb_report), nothing to do
  Exchange X;
};

constexpr int kCommWarps = 4, kComm = 32 * kCommWarps, kSlots = 4;  // edge values per communicating thread
constexpr int kMaxComputeWarps = 16;

// A block's tile: W columns by rows rows; a field is kept with pitch P, E and U
// with rows 0 .. rows, V with rows -1 .. rows - 1, columns -1 .. W.
struct Tile {
  int W, rows, P, fs;
  __device__ int at(int x, int y) const { return y * P + x + 1; }        // in a field of E or U
  __device__ int atv(int x, int y) const { return 2 * fs + (y + 1) * P + x + 1; }  // V in a vector
};
__host__ __device__ inline int tile_pitch(int W) { return (W + 2) | 1; }
__host__ __device__ inline size_t tile_values(int W, int rows, bool grad) {
  return (size_t)tile_pitch(W) * (6 * (rows + 1) + (grad ? 5 : 4) * rows);
}

template <typename T, int MODE>
__global__ void __launch_bounds__(32 * (kMaxComputeWarps + kCommWarps), 1) cheb_many_kernel(Geom<T> G, ManyArgs<T> A) {
  constexpr bool FWD = MODE == kForward, GRAD = MODE == kGrad;
  extern __shared__ double smem_raw[];
  __shared__ unsigned dead;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nc = (blockDim.x >> 5) - kCommWarps;  // compute warps
  const int per_set = A.ns * A.ng;
  const int set = blockIdx.x / per_set, strip = blockIdx.x % per_set / A.ng, grp = blockIdx.x % A.ng;
  const int nx = G.nx, ny = G.ny;
  // columns [i0, i0 + W), rows [j0, j0 + rows)
  const int wq = nx / A.ns, wr = nx % A.ns, hq = ny / A.ng, hr = ny % A.ng;
  const int i0 = strip * wq + min(strip, wr), j0 = grp * hq + min(grp, hr);
  Tile t;
  t.W = wq + (strip < wr);
  t.rows = hq + (grp < hr);
  t.P = tile_pitch(t.W);
  t.fs = (t.rows + 1) * t.P;
  const int W = t.W, rows = t.rows, fs = t.fs;
  T* cur = reinterpret_cast<T*>(smem_raw);
  T* old = cur + 3 * fs;
  T* sF = old + 3 * fs;            // 3 fields of rows x P
  T* sH = sF + 3 * rows * t.P;
  T* sA = sH + rows * t.P;         // the gradient's sum
  const size_t nk = G.nk, so = (size_t)set * 3 * nk;
  const size_t id0 = (size_t)j0 * nx + i0;
  for (int q = threadIdx.x; q < W * rows; q += blockDim.x) {
    const int x = q % W, y = q / W, a = t.at(x, y), av = t.atv(x, y), f = y * t.P + x;
    const size_t o = so + id0 + (size_t)y * nx + x;
    cur[a] = A.b1[o];
    cur[fs + a] = A.b1[o + nk];
    cur[av] = A.b1[o + 2 * nk];
    old[a] = A.b2 ? A.b2[o] : T{};
    old[fs + a] = A.b2 ? A.b2[o + nk] : T{};
    old[av] = A.b2 ? A.b2[o + 2 * nk] : T{};
    if (!FWD) {
      sF[f] = A.F[o];
      sF[rows * t.P + f] = A.F[o + nk];
      sF[2 * rows * t.P + f] = A.F[o + 2 * nk];
    }
    sH[f] = u_neg(A.H[o - so]);
    if (GRAD) sA[f] = T{};
  }
  if (threadIdx.x == 0) dead = 0u;
  const unsigned declined = *A.declined;
  __syncthreads();
  if (declined) return;

  if (warp >= nc) {
    // ---- edges
    const size_t ncol = (size_t)3 * A.ns * ny, nrow = (size_t)3 * A.ng * nx;
    const size_t pcol = A.nset * ncol, prow = A.nset * nrow;
    const int strip_w = strip ? strip - 1 : A.ns - 1, strip_e = strip + 1 < A.ns ? strip + 1 : 0;
    const int grp_s = grp ? grp - 1 : A.ng - 1, grp_n = grp + 1 < A.ng ? grp + 1 : 0;
    const int jn = j0 + rows < ny ? j0 + rows : 0, js = j0 ? j0 - 1 : ny - 1;
    // slot of a column (row) edge value at an even step; an odd step's is a parity
    // stride further on (odd: the stride, in units of a slot)
    auto col_slot = [&](int kind, int st, int j) { return (unsigned)(set * ncol + ((size_t)kind * A.ns + st) * ny + j); };
    auto row_slot = [&](int kind, int g, int i) {
      return (unsigned)(2 * pcol + set * nrow + ((size_t)kind * A.ng + g) * nx + i);
    };
    int src[kSlots], dst[kSlots];            // tile offsets, -1: none
    unsigned put[kSlots], get[kSlots], podd[kSlots], godd[kSlots];
#pragma unroll
    for (int m = 0; m < kSlots; ++m) {
      const int c = threadIdx.x - 32 * nc;
      int q = c + kComm * m;
      src[m] = dst[m] = -1;
      put[m] = get[m] = 0u;
      podd[m] = godd[m] = (unsigned)(q < 3 * W ? prow : pcol);
      if (q < 3 * W) {
        const int k = q / W, x = q % W;
        src[m] = k == kRowE ? t.at(x, 0) : (k == kRowU ? fs + t.at(x, 0) : t.atv(x, rows - 1));
        put[m] = row_slot(k, grp, i0 + x);
        dst[m] = k == kRowE ? t.at(x, rows) : (k == kRowU ? fs + t.at(x, rows) : t.atv(x, -1));
        get[m] = row_slot(k, k == kRowV ? grp_s : grp_n, i0 + x);
        continue;
      }
      q -= 3 * W;
      const int qp = q;
      if (qp < 3 * rows) {
        const int k = qp / rows, y = qp % rows;
        src[m] = k == kColE ? t.at(0, y) : (k == kColV ? t.atv(0, y) : fs + t.at(W - 1, y));
        put[m] = col_slot(k, strip, j0 + y);
      }
      // E rows 0 .., V rows -1 .. of the east strip, U rows 0 .. rows of the west strip
      if (q < rows) {
        dst[m] = t.at(W, q);
        get[m] = col_slot(kColE, strip_e, j0 + q);
      } else if ((q -= rows) <= rows) {
        dst[m] = t.atv(W, q - 1);
        get[m] = col_slot(kColV, strip_e, q ? j0 + q - 1 : js);
      } else if ((q -= rows + 1) <= rows) {
        dst[m] = fs + t.at(-1, q);
        get[m] = col_slot(kColU, strip_w, q < rows ? j0 + q : jn);
      }
    }
    ulonglong2* X = A.X.col;
    // sends the edge of b under `flag` and fills b's halo with the neighbours'
    auto exchange = [&](T* b, unsigned flag) {
#pragma unroll
      for (int m = 0; m < kSlots; ++m)
        if (src[m] >= 0) st_edge(X + put[m] + ((flag & 1) ? podd[m] : 0u), pack(b[src[m]], flag));
      unsigned left = 0;
#pragma unroll
      for (int m = 0; m < kSlots; ++m)
        if (dst[m] >= 0) left |= 1u << m;
      for (int n = 0; left; ++n) {
        ulonglong2 w[kSlots];
#pragma unroll
        for (int m = 0; m < kSlots; ++m)
          if (left >> m & 1) w[m] = ld_edge(X + get[m] + ((flag & 1) ? godd[m] : 0u));
#pragma unroll
        for (int m = 0; m < kSlots; ++m)
          if ((left >> m & 1) && arrived(w[m], flag)) {
            b[dst[m]] = unpack<T>(w[m]);
            left &= ~(1u << m);
          }
        if (n >= A.X.polls || ((n & 1023) == 1023 && *(volatile unsigned*)A.X.bad)) {
          give_up(A.X, &dead);
          return;
        }
      }
    };
    exchange(cur, A.flag0 + 1);
    __syncthreads();
    for (int step = 0; step < A.steps; ++step) {
      if (*(volatile unsigned*)&dead) return;
      asm volatile("bar.sync 1, %0;" ::"r"(blockDim.x) : "memory");  // the edge is computed
      if (step + 1 < A.steps) exchange(old, A.flag0 + 2 + step);
      T* x = cur;
      cur = old;
      old = x;
      __syncthreads();
    }
    return;
  }

  // ---- points: the first and last row, then the outer columns, then the rest
  const int sh = A.seg_shift, seg = 1 << sh, inner = max(rows - 2, 0);  // seg: warps to a row of the widest tile
  const int t_row = (rows > 1 ? 2 : 1) * seg, t_col = (2 * inner + 31) / 32, t_all = t_row + t_col + (inner + 1) / 2 * seg;
  __syncthreads();
  for (int step = 0; step < A.steps; ++step) {
    if (*(volatile unsigned*)&dead) return;
    T dk = T{};
    if (!FWD) dk = A.d[-step];
    bool told = false;
    for (int k = warp; k < t_all; k += nc) {
      if (!told && k >= t_row + t_col) {
        told = true;
        asm volatile("bar.arrive 1, %0;" ::"r"(blockDim.x) : "memory");
      }
      int x, y;
      bool live, two = false;
      if (k < t_row) {
        x = (k & (seg - 1)) * 32 + lane;
        y = k < seg ? 0 : rows - 1;
        live = x < W;
      } else if (k < t_row + t_col) {
        const int q = (k - t_row) * 32 + lane;
        live = q < 2 * inner;
        x = q < inner ? 0 : W - 1;
        y = 1 + (q < inner ? q : q - inner);
      } else {
        const int q = k - t_row - t_col;
        x = (q & (seg - 1)) * 32 + lane;
        y = 1 + 2 * (q >> sh);
        two = y + 1 < rows - 1;
        live = x > 0 && x < W - 1;
      }
      if (!live) x = y = 0;
      const T* c = cur + t.at(x, y);
      const T* v = cur + t.atv(x, y);
      T* b = old + t.at(x, y);
      T* bv = old + t.atv(x, y);
      int f = y * t.P + x;
      size_t o = id0 + (size_t)y * nx + x;
      // carried from row to row: E, U's difference and pair sum, V below and its pair sum
      T e = c[0], u = c[fs], w = c[fs - 1], vs = v[-t.P];
      T ps[2] = {};
      if (GRAD) {
        const T* sp = A.s - (size_t)step * nk + o;
        ps[0] = sp[0];
        if (two) ps[1] = sp[nx];
      }
      T du = u_sub(u, w), su = u_add(u, w), sv = u_add(vs, v[1 - t.P]);
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        if (r == 1 && !two) break;
        const T vo = v[0], svn = u_add(vo, v[1]), en = c[t.P];
        u = c[fs + t.P];
        w = c[fs + t.P - 1];
        T a0 = b[0], a1 = b[fs], a2 = bv[0];
        if (!FWD) {
          a0 = u_madd(a0, sF[f], dk);
          a1 = u_madd(a1, sF[rows * t.P + f], dk);
          a2 = u_madd(a2, sF[2 * rows * t.P + f], dk);
        }
        const T s = u_add(du, u_sub(vo, vs)), sun = u_add(u, w);
        a0 = u_norm(u_madd(a0, s, sH[f]));
        a1 = u_madd(a1, u_add(sv, svn), G.cu);
        a1 = u_norm(u_madd(a1, u_sub(c[1], e), u_neg(G.gu)));
        a2 = u_madd(a2, u_add(su, sun), u_neg(G.cv));
        a2 = u_norm(u_madd(a2, u_sub(en, e), u_neg(G.gv)));
        if (live) {
          b[0] = a0;
          b[fs] = a1;
          bv[0] = a2;
          if (FWD) A.s[o + (size_t)step * nk] = u_norm(s);
          if (GRAD) sA[f] = u_norm(u_madd(sA[f], e, ps[r]));
        }
        if (r == 0) {
          e = en;
          du = u_sub(u, w);
          su = sun;
          sv = svn;
          vs = vo;
          c += t.P;
          v += t.P;
          b += t.P;
          bv += t.P;
          f += t.P;
          o += nx;
        }
      }
    }
    if (!told) asm volatile("bar.arrive 1, %0;" ::"r"(blockDim.x) : "memory");
    T* x = cur;
    cur = old;
    old = x;
    __syncthreads();
  }
  for (int q = threadIdx.x; q < W * rows; q += 32 * nc) {
    const int x = q % W, y = q / W, a = t.at(x, y), av = t.atv(x, y);
    const size_t o = so + id0 + (size_t)y * nx + x;
    if (A.o1) {
      A.o1[o] = cur[a];
      A.o1[o + nk] = cur[fs + a];
      A.o1[o + 2 * nk] = cur[av];
      A.o2[o] = old[a];
      A.o2[o + nk] = old[fs + a];
      A.o2[o + 2 * nk] = old[av];
    }
    if (GRAD) A.acc[o - so] = sA[y * t.P + x];
  }
}

size_t exchange_bytes(int ns, int ng, int nx, int ny, int nset) {
  return 256 + (size_t)2 * nset * 3 * ((size_t)ns * ny + (size_t)ng * nx) * sizeof(ulonglong2);
}
// The tiles for a grid, one block per multiprocessor, or blocks == 0 where they do
// not fit: of the ways to cut the grid into ns strips of ng tiles, the one
// whose blocks have the fewest warp-rows to compute, then the fewest edge values.
struct ManyPlan {
  int ns = 0, ng = 0, blocks = 0, warps = 0, seg_shift = 0;  // warps: compute warps; 2^seg_shift warps to a row
  size_t smem = 0;
};
ManyPlan many_plan(int nx, int ny, int nset, int sms, bool grad, size_t exchange) {
  ManyPlan p;
  long long best = 1ll << 62;
  for (int ns = 1; ns * nset <= sms && 2 * ns <= nx; ++ns) {
    const int top = std::min(sms / (ns * nset), ny), W = (nx + ns - 1) / ns, H = (ny + top - 1) / top;
    const int ng = (ny + H - 1) / H;  // no more tiles than rows of height H need
    int sh = 0;
    while (32 << sh < W) ++sh;
    const int seg = 1 << sh, inner = std::max(H - 2, 0);
    const int edge = (H > 1 ? 2 : 1) * seg + (2 * inner + 31) / 32, tasks = edge + (inner + 1) / 2 * seg;
    const int work = seg * H + (2 * inner + 31) / 32;
    const size_t smem = tile_values(W, H, grad) * 8;
    if (3 * W + 3 * H + 2 > kComm * kSlots || smem > 226 * 1024 || exchange_bytes(ns, ng, nx, ny, nset) > exchange)
      continue;
    const long long c = (long long)work * 4096 + W + H;
    if (c >= best) continue;
    best = c;
    p.ns = ns;
    p.ng = ng;
    p.blocks = ns * ng * nset;
    // two turns or more where most of the work is inside, so that the edge is not
    // computed in step with the rest (256^2: 2.10 -> 1.73 us per step)
    const int turns = std::max(2 * edge <= tasks ? 2 : 1, (tasks + kMaxComputeWarps - 1) / kMaxComputeWarps);
    p.warps = (tasks + turns - 1) / turns;
    p.seg_shift = sh;
    p.smem = smem;
  }
  return p;
}
cudaError_t exchange_at(const ManyPlan& p, const KrylovSettings* k, int nset, void* base, Exchange* X,
                        cudaStream_t s) {
  const int nx = k->nx, ny = k->ny;
  char* b = static_cast<char*>(base);
  X->host_bad = k->gave_up;
  X->polls = k->edge_polls;
  X->bad = reinterpret_cast<unsigned*>(b);
  X->col = reinterpret_cast<ulonglong2*>(b + 256);
  return cudaMemsetAsync(b, 0, exchange_bytes(p.ns, p.ng, nx, ny, nset), s);
}
template <typename T, int MODE>
cudaError_t launch_many(const Geom<T>& G, ManyArgs<T> A, const ManyPlan& p, int nset, cudaStream_t s, bool* launched) {
  A.nset = nset;
  A.ns = p.ns;
  A.ng = p.ng;
  A.seg_shift = p.seg_shift;
  auto kern = cheb_many_kernel<T, MODE>;
  Geom<T> geom = G;
  void* args[] = {&geom, &A};
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.smem);
  if (e == cudaSuccess)
    e = cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(kern), dim3(p.blocks),
                                    dim3(32 * (p.warps + kCommWarps)), args, p.smem, s);
  // a device that cannot hold the grid at once (part of it set aside): one
  // launch per step
  *launched = e == cudaSuccess;
  if (e == cudaErrorCooperativeLaunchTooLarge) {
    cudaGetLastError();
    return cudaSuccess;
  }
  return e;
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
  unsigned *maxbits, *declined;
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
  S->maxbits = reinterpret_cast<unsigned*>(take(2 * sizeof(unsigned)));
  S->declined = S->maxbits + 1;
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

// slot: 0 and 1 for a call's first and second input, of which either declines.
template <typename T>
cudaError_t init(const Geom<T>& G, const KrylovSettings* k, const void* in, int adjoint, T* F, T* bK, const T* dK,
                 const Scratch& S, int nset, int slot, cudaStream_t s, int64_t* launches) {
  cudaError_t e = cudaMemsetAsync(S.maxbits, 0, (slot == 0 ? 2 : 1) * sizeof(unsigned), s);
  if (e != cudaSuccess) return e;
  cheb_init<T><<<dim3((unsigned)((3 * G.nk + 255) / 256), nset), 256, 0, s>>>(
      G, static_cast<const double2*>(in), k->w64, adjoint, F, bK, dK, S.maxbits);
  ++*launches;
  return cudaGetLastError();
}
cudaError_t report(KrylovSettings* k, const ChebPlan& p, const Scratch& S, int df, int slot, cudaStream_t s,
                   int64_t* launches) {
  cheb_report<<<1, 32, 0, s>>>(S.d, p.K, p.n, S.maxbits, k->rtol, df ? 64 : 900, S.report, S.declined);
  ++*launches;
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(k->pinned + 2 * slot, S.report, 2 * sizeof(double), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaEventRecord(k->ev[slot], s);
  return e;
}
cudaError_t accepted(KrylovSettings* k, int slot, bool* ok, double* bound) {
  const cudaError_t e = cudaEventSynchronize(k->ev[slot]);
  if (e != cudaSuccess) return e;
  *ok = k->pinned[2 * slot + 1] != 0.0;
  *bound = std::max(*bound, k->pinned[2 * slot]);
  return cudaSuccess;
}
// Whether the input of a slot up to `slot` is declined, asked before the step that
// follows kAhead launches of one step each: enough of them that the stream does not
// run dry while the host learns it, and all that declined input costs.
constexpr int kAhead = 16;
bool known_declined(KrylovSettings* k, int slot, int launched) {
  if (launched != kAhead) return false;
  for (int i = 0; i <= slot; ++i)
    if (cudaEventSynchronize(k->ev[i]) == cudaSuccess && k->pinned[2 * i + 1] == 0.0) return true;
  return false;
}
rexi_status failed(cudaError_t e) {
  set_last_error(cudaGetErrorString(e));
  return REXI_ECUDA;
}

// The Clenshaw steps k = K - 1 .. 1 on F with b_K in bA; the two newest
// vectors are left in *b1 (b_1) and *b2 (b_2, null when K = 1).  The number of
// steps launched: fewer where the input is declined.
template <typename T, int MODE>
int clenshaw(const Geom<T>& G, StepArgs<T> A, KrylovSettings* ks, int slot, int K, const T* d, T* bA, T* bB,
             const T* sfield, int nset, cudaStream_t s, const T** b1, const T** b2) {
  T *cur = bA, *old = bB;
  bool have_old = false;
  int n = 0;
  for (int k = K - 1; k >= 1; --k, ++n) {
    if (known_declined(ks, slot, n)) break;
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
  return n;
}

template <typename T>
rexi_status step_impl(KrylovSettings* k, const ChebPlan& p, double h, int M, const void* in, void* out, double dt,
                      int real_input, bool adjoint, const ChebBuffers& b, cudaStream_t s, const KrylovHooks& hooks,
                      double* bound) {
  auto mark = [&](int i) {
    if (hooks.mark) hooks.mark(hooks.ctx, i, s);
  };
  int64_t launches = 0;
  const int nset = real_input ? 1 : 2, df = std::is_same<T, double>::value ? 0 : 1;
  const Geom<T> G = make_geom<T>(k, adjoint ? -dt : dt, p);
  Scratch S;
  carve(p, M + kL, static_cast<char*>(b.scratch), &S);
  T *F = static_cast<T*>(b.f0), *bA = static_cast<T*>(b.bA), *bB = static_cast<T*>(b.bB);
  const T* d = coeff_table(S, T{});
  mark(0);
  cudaError_t e = coefficients(p, h, M, S, s, &launches);
  mark(1);
  if (e == cudaSuccess) e = init(G, k, in, adjoint ? 1 : 0, F, bA, d + p.K, S, nset, 0, s, &launches);
  if (e == cudaSuccess) e = report(k, p, S, df, 0, s, &launches);
  if (e != cudaSuccess) return failed(e);
  StepArgs<T> A = {};
  A.F = F;
  A.H = depth_table(k, T{});
  const T *b1, *b2;
  const ManyPlan mp = many_plan(k->nx, k->ny, nset, k->sms, false, b.exchange_bytes);
  bool many = mp.blocks && p.K > 2;
  if (many) {
    ManyArgs<T> Q = {};
    e = exchange_at(mp, k, nset, b.exchange, &Q.X, s);
    Q.b1 = bA;
    Q.o1 = bA;
    Q.o2 = bB;
    Q.F = F;
    Q.H = A.H;
    Q.d = d + p.K - 1;
    Q.steps = p.K - 1;
    Q.declined = S.declined;
    if (e == cudaSuccess) e = launch_many<T, kSum>(G, Q, mp, nset, s, &many);
    if (e != cudaSuccess) return failed(e);
    b1 = bA;
    b2 = bB;
    A.bad = Q.X.bad;
    launches += many;
  }
  if (!many) {
    A.bad = nullptr;
    launches += clenshaw<T, kSum>(G, A, k, 0, p.K, d, bA, bB, nullptr, nset, s, &b1, &b2);
  }
  mark(2);
  mark(3);
  // the host looks at the tail and the input while the steps run; `out` is
  // written by the last step only
  bool ok = false;
  e = accepted(k, 0, &ok, bound);
  if (e != cudaSuccess) return failed(e);
  if (ok) {
    A.b1 = b1;
    A.b2 = b2;
    A.d = d;
    A.out = static_cast<double2*>(out);
    A.w = k->w64;
    A.adjoint = adjoint ? 1 : 0;
    A.real_out = real_input;
    launch_step<T, kSumLast>(G, A, nset, s, !many);
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
                      double* grad_depth, void* grad_in, double dt, const ChebGradBuffers& b, cudaStream_t s,
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
  const ManyPlan mp = many_plan(k->nx, k->ny, 1, k->sms, true, b.exchange_bytes);
  bool many = mp.blocks && p.K > 2;
  ManyArgs<T> Q = {};
  Q.H = depth_table(k, T{});
  Q.steps = p.K - 1;
  Q.declined = S.declined;
  if (many && e == cudaSuccess) e = exchange_at(mp, k, 1, b.exchange, &Q.X, s);
  // forward: P_0 in bA, P_1 in bB, then each P_{k+1} over P_{k-1}; s_k for k < K
  Geom<T> G = make_geom<T>(k, dt, p);
  if (e == cudaSuccess) e = init(G, k, f_in, 0, bA, static_cast<T*>(nullptr), d, S, 1, 0, s, &launches);
  if (e == cudaSuccess) e = report(k, p, S, df, 0, s, &launches);
  if (e != cudaSuccess) return failed(e);
  {
    StepArgs<T> A = {};
    A.H = depth_table(k, T{});
    T *cur = bA, *old = bB;
    for (int j = 0; j < p.K; ++j) {
      if (known_declined(k, 0, j)) break;
      A.b1 = cur;
      A.b2 = j ? old : nullptr;
      A.bout = old;
      A.s = sf + (size_t)j * G.nk;
      if (j == 0)
        launch_step<T, kForwardFirst>(G, A, 1, s);
      else
        launch_step<T, kForward>(G, A, 1, s);
      ++launches;
      std::swap(cur, old);
      if (j == 0 && many) {
        Q.b1 = cur;
        Q.b2 = old;
        Q.s = sf + G.nk;
        e = launch_many<T, kForward>(G, Q, mp, 1, s, &many);
        if (e != cudaSuccess) return failed(e);
        launches += many;
        if (many) break;
      }
    }
  }
  // backward: the Clenshaw vectors of W^{-1} G under -dt, each step taking its s_k
  G = make_geom<T>(k, -dt, p);
  e = init(G, k, g_out, 1, F, bA, d + p.K, S, 1, 1, s, &launches);
  if (e == cudaSuccess) e = report(k, p, S, df, 1, s, &launches);
  if (e != cudaSuccess) return failed(e);
  StepArgs<T> A = {};
  A.F = F;
  A.H = depth_table(k, T{});
  A.acc = static_cast<T*>(b.acc);
  A.first = 1;
  A.bad = Q.X.bad;  // of either launch of many steps (null: no exchange was set up)
  const T *b1, *b2;
  if (many) {
    Q.b1 = bA;
    Q.b2 = nullptr;
    Q.o1 = bA;
    Q.o2 = bB;
    Q.F = F;
    Q.d = d + p.K - 1;
    Q.s = sf + (size_t)(p.K - 1) * G.nk;
    Q.acc = A.acc;
    Q.flag0 = p.K;
    e = launch_many<T, kGrad>(G, Q, mp, 1, s, &many);
    if (e != cudaSuccess) return failed(e);
    b1 = bA;
    b2 = bB;
    launches += many;
  }
  if (!many) {
    launches += clenshaw<T, kGrad>(G, A, k, 1, p.K, d, bA, bB, sf, 1, s, &b1, &b2);
  }
  mark(2);
  mark(3);
  bool okf = false, okg = false;
  e = accepted(k, 0, &okf, bound);
  if (e == cudaSuccess) e = accepted(k, 1, &okg, bound);
  if (e != cudaSuccess) return failed(e);
  if (okf && okg) {
    A.first = 0;
    A.b1 = b1;
    A.b2 = b2;
    A.d = d;
    A.s = sf;
    A.grad = grad_depth;
    A.w = k->w64;
    A.out = static_cast<double2*>(grad_in);
    A.adjoint = A.real_out = 1;
    launch_step<T, kGradLast>(G, A, 1, s, !many);
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
  // 2 / rho cut to 12 bits (the interval grows by 5e-4 at most): a small change of
  // the depth then leaves the scaled stencil's constants and the coefficients as they
  // are, and where the spacings, g and f are short binary numbers (unit-square grids of
  // 2^m points) the constants are exact in double-float too, so that differences of
  // nearby problems see no rounding of theirs.  On other domains the constants round to
  // 48 bits, the same for both problems unless rho crosses a step of the 12 bits
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
                      const void* g_out, double* grad_depth, void* grad_in, double dt, const ChebGradBuffers& b,
                      cudaStream_t s, const KrylovHooks& hooks, double* bound) {
  *bound = 0.0;
  return df ? grad_impl<float2>(k, p, h, M, f_in, g_out, grad_depth, grad_in, dt, b, s, hooks, bound)
            : grad_impl<double>(k, p, h, M, f_in, g_out, grad_depth, grad_in, dt, b, s, hooks, bound);
}

}  // namespace rexi
