// Test harness: scalar device functions of the library's headers, one thread per argument.
#include "gks_step.cuh"

namespace {

__global__ void quotient_kernel(long n, const double* a, const double* b, double* q) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) q[i] = gks::g_quot<double>(a[i], b[i]);
}

unsigned blocks(long n) { return (unsigned)((n + 255) / 256); }

}  // namespace

// device pointers; the default stream
extern "C" int dev_quotient(long n, const double* a, const double* b, double* q) {
  quotient_kernel<<<blocks(n), 256>>>(n, a, b, q);
  return (int)cudaDeviceSynchronize();
}
