// Test harness: scalar device functions of the library's headers, one thread per argument.
#include "gks_step.cuh"

namespace {

__global__ void quotient_kernel(long n, const double* a, const double* b, double* q) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) q[i] = gks::g_quot<double>(a[i], b[i]);
}

__global__ void physical_kernel(long n, const double* w, int* ok) {  // w: [n][4]
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) ok[i] = gks::physical<2, double>(1.4, w + 4 * i);
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
