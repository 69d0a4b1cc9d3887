// Test harness: scalar device functions of the library's headers, one thread per argument.
#include "gks_step.cuh"

#include <cmath>

namespace {

__global__ void quotient_kernel(long n, const double* a, const double* b, double* q) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) q[i] = gks::g_quot<double>(a[i], b[i]);
}

__global__ void physical_kernel(long n, const double* w, int* ok) {  // w: [n][4]
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) ok[i] = gks::physical<2, double>(1.4, w + 4 * i);
}

__global__ void rsqrt_kernel(long n, const double* x, double* y) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = gks::g_rsqrt<double>(x[i]);
}

// the library's erfc(x) and exp(-x^2), and CUDA's
__global__ void gauss_kernel(long n, const double* x, double* c, double* e, double* cc, double* ce) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  gks::g_gauss<double>(x[i], c[i], e[i]);
  cc[i] = erfc(x[i]);
  ce[i] = exp(-x[i] * x[i]);
}

unsigned blocks(long n) { return (unsigned)((n + 255) / 256); }

}  // namespace

// device pointers; the default stream
extern "C" int dev_quotient(long n, const double* a, const double* b, double* q) {
  quotient_kernel<<<blocks(n), 256>>>(n, a, b, q);
  return (int)cudaDeviceSynchronize();
}
extern "C" int dev_physical(long n, const double* w, int* ok) {
  physical_kernel<<<blocks(n), 256>>>(n, w, ok);
  return (int)cudaDeviceSynchronize();
}
extern "C" int dev_rsqrt(long n, const double* x, double* y) {
  rsqrt_kernel<<<blocks(n), 256>>>(n, x, y);
  return (int)cudaDeviceSynchronize();
}
extern "C" int dev_gauss(long n, const double* x, double* c, double* e, double* cc, double* ce) {
  gauss_kernel<<<blocks(n), 256>>>(n, x, c, e, cc, ce);
  return (int)cudaDeviceSynchronize();
}
// erfc in the host's extended precision, as a sum of two doubles
extern "C" void host_erfc(long n, const double* x, double* hi, double* lo) {
  for (long i = 0; i < n; ++i) {
    const long double v = erfcl((long double)x[i]);
    hi[i] = (double)v;
    lo[i] = (double)(v - hi[i]);
  }
}
