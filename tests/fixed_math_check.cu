// Test harness: the fixed-point elementary functions, element by element.
#include "fixmath.cuh"

using namespace gps;

__global__ void k_fixed_log(const double* __restrict__ x, double* __restrict__ out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = fx_log(x[i]);
}

extern "C" int run_fixed_log(const double* x, double* out, int n) {
  if (n <= 0) return 0;
  k_fixed_log<<<(n + 255) / 256, 256>>>(x, out, n);
  return (int)cudaDeviceSynchronize();
}

__global__ void k_fixed_divide(const double* __restrict__ a, const double* __restrict__ b, double* __restrict__ out,
                               int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = fx_div(a[i], fx_divisor(b[i]));
}

extern "C" int run_fixed_divide(const double* a, const double* b, double* out, int n) {
  if (n <= 0) return 0;
  k_fixed_divide<<<(n + 255) / 256, 256>>>(a, b, out, n);
  return (int)cudaDeviceSynchronize();
}
