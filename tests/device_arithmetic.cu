// Entry points that run the library's device arithmetic on arrays, for tests/test_gpu_arithmetic.py.
#include "pole_cells.cuh"

using namespace rexi;

namespace {
// out[i] = the polynomial with coefficients re, im (kCellP each) at t[i]
__global__ void horner(int n, const double* re, const double* im, const double* t, double2* out) {
  __shared__ float4 p[kCellP];
  if (threadIdx.x < kCellP) {
    const float2 a = df_from_double(re[threadIdx.x]), b = df_from_double(im[threadIdx.x]);
    p[threadIdx.x] = make_float4(a.x, a.y, b.x, b.y);
  }
  __syncthreads();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float2 ar, ai;
  cell_horner(p, t[i], ar, ai);
  out[i] = make_double2(df_to_double(ar), df_to_double(ai));
}
// out[3 i ..] = rcp64(x[i]) and sqrt_rsqrt64(x[i])
__global__ void reciprocals(int n, const double* x, double* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double2 s = sqrt_rsqrt64(x[i]);
  out[3 * i] = rcp64(x[i]);
  out[3 * i + 1] = s.x;
  out[3 * i + 2] = s.y;
}
}  // namespace

extern "C" int device_reciprocals(int n, const double* x, double* out) {
  reciprocals<<<(n + 127) / 128, 128>>>(n, x, out);
  return (int)cudaDeviceSynchronize();
}
extern "C" int device_horner(int n, const double* re, const double* im, const double* t, void* out) {
  horner<<<(n + 127) / 128, 128>>>(n, re, im, t, static_cast<double2*>(out));
  return (int)cudaDeviceSynchronize();
}
