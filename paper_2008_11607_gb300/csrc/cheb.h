// Chebyshev form of the shared-Krylov method (cheb.cu), used by lanczos.cu.
#pragma once

#include <cuda_runtime.h>

#include "internal.h"
#include "krylov.h"

namespace rexi {

// Degree and node count of the expansion of r on [-Lh, Lh].
struct ChebPlan {
  int K = 0;  // degree: the last coefficient kept
  int n = 0;  // Chebyshev nodes r is sampled at (even, > K)
  double Lh = 0.0;
  double t2 = 0.0;  // 2 |dt| / Lh
};
// Whether the full sum at this dt is taken as a Chebyshev expansion with the
// coefficients beyond K summing to less than `target` (see cheb.cu), and its
// degree.
bool cheb_plan(const KrylovSettings* k, double h, int M, double dt, double target, ChebPlan* p);
// Bytes of device scratch for the coefficients (nodes, coefficients, report).
size_t cheb_scratch_bytes(const ChebPlan& p, int N);

struct ChebBuffers {
  void *f0, *bA, *bB;  // state-sized vectors (nset x 3 nk values of 8 bytes)
  void* scratch;       // cheb_scratch_bytes
  void* exchange;      // edge values between warps (any size; 256-byte aligned)
  size_t exchange_bytes;
};
// out = r(dt A) in (adjoint: r(dt A)^H), as krylov_step.  REXI_EUNSUPPORTED,
// with `out` untouched, where the input or the coefficients call for the
// Lanczos form.
rexi_status cheb_step(KrylovSettings* k, const ChebPlan& p, int df, double h, int M, const void* in, void* out,
                      double dt, int real_input, bool adjoint, const ChebBuffers& b, cudaStream_t s,
                      const KrylovHooks& hooks, double* bound);

struct ChebGradBuffers {
  void *f0, *bA, *bB;  // state-sized vectors (3 nk values of 8 bytes)
  void* acc;           // nk values of 8 bytes
  void* div;           // K nk values of 8 bytes
  void* scratch;       // cheb_scratch_bytes
  void* exchange;      // edge values between warps (any size; 256-byte aligned)
  size_t exchange_bytes;
};
// grad_depth += dL/dH for out = r(dt A(H)) f_in, G = dL/d out (real input), and,
// with grad_in, grad_in = r(dt A)^H G: the end of the same recurrence.  Same
// refusals, with both untouched.
rexi_status cheb_grad(KrylovSettings* k, const ChebPlan& p, int df, double h, int M, const void* f_in,
                      const void* g_out, double* grad_depth, void* grad_in, double dt, const ChebGradBuffers& b,
                      cudaStream_t s, const KrylovHooks& hooks, double* bound);

}  // namespace rexi
