// Stateless per-face flux evaluation (gks_face_flux).
#include "gks_dispatch.h"
#include "gks_flux.cuh"
#include "gks_step.cuh"

namespace gks {

constexpr int kFaceT = 64;  // faces (threads) per CTA: 27 KB of 3D records, six CTAs per SM

// double -> float, rounded to nearest even as the conversion instruction does, on the integer pipe:
// this part converts at the FP64 rate (2 per clock per SM), and the 53 values of a 3D record took 76% of that pipe.
// Values outside the normal single-precision range (but zero) go through the instruction.
__device__ __forceinline__ float d2f_rn(double x) {
  const unsigned int H = (unsigned int)__double2hiint(x), L = (unsigned int)__double2loint(x);
  const unsigned long long r = (((unsigned long long)H << 32) | L) + 0x0fffffffull + ((L >> 29) & 1u);
  const unsigned int h = (unsigned int)(r >> 32), l = (unsigned int)r;
  const unsigned int e = (h >> 20) & 0x7ffu;
  float f = __uint_as_float(((__funnelshift_r(l, h, 29) + 0x40000000u) & 0x7fffffffu) | (h & 0x80000000u));
  if (e - 897u >= 254u) f = ((H << 1) | L) == 0u ? __uint_as_float(H) : (float)x;
  return f;
}
__device__ __forceinline__ void to_arith(double x, float& o) { o = d2f_rn(x); }
__device__ __forceinline__ void to_arith(double x, double& o) { o = x; }

// One face per thread.  A CTA's records are contiguous: they are staged in shared memory by 16-byte asynchronous
// copies and read back by record (21, 35 and 53 doubles: an odd stride, no bank conflicts), and the fluxes go
// out the same way, so that the kernel moves its bytes in full lines; bound by HBM in single precision and by
// the FP64 pipe in double.  400k 3D records in single precision (181 MB): 74.1 -> 53.5 us per
// call with the conversions of the outputs (one thread reading its record from global memory before).
template <int D, class R, bool MULTID, bool RAR>
__global__ void __launch_bounds__(kFaceT) face_kernel(int abar_t0, Gas<double> gas_d, double dt, const double* faces,
                                                      long nfaces, double* Fout, double* tout) {
  constexpr int nv = D + 2;
  constexpr int len = 6 * nv + 2 * (D - 1) * nv + 3;
  __shared__ __align__(16) double rec[kFaceT * len];
  const int tid = threadIdx.x;
  const long f0 = (long)blockIdx.x * kFaceT;
  const int nf = (int)min((long)kFaceT, nfaces - f0), nd = nf * len;
  const double* src = faces + f0 * len;
  if ((size_t)src % 16 == 0) {
    for (int i = tid; i < nd / 2; i += kFaceT) cp_async<16>(&rec[2 * i], src + 2 * i);
    if (nd % 2 && tid == 0) cp_async<8>(&rec[nd - 1], src + nd - 1);
  } else {
    for (int i = tid; i < nd; i += kFaceT) cp_async<8>(&rec[i], src + i);
  }
  cp_async_wait_all();
  __syncthreads();
  R F[nv], tau = R(0);
  const double* r = rec + (tid < nf ? tid : 0) * len;
  R wl[nv], wr[nv], cl[nv], cr[nv], sl[nv], sr[nv], tl[Dims<D>::nt][nv], tr[Dims<D>::nt][nv], dxl, dxr, tau_t, dtr;
#pragma unroll
  for (int v = 0; v < nv; ++v) {
    to_arith(r[v], wl[v]);
    to_arith(r[nv + v], wr[v]);
    to_arith(r[2 * nv + v], cl[v]);
    to_arith(r[3 * nv + v], cr[v]);
    to_arith(r[4 * nv + v], sl[v]);
    to_arith(r[5 * nv + v], sr[v]);
  }
  if (MULTID) {
#pragma unroll
    for (int s = 0; s < D - 1; ++s)
#pragma unroll
      for (int v = 0; v < nv; ++v) {
        to_arith(r[6 * nv + s * nv + v], tl[s][v]);
        to_arith(r[6 * nv + (D - 1) * nv + s * nv + v], tr[s][v]);
      }
  }
  to_arith(r[len - 3], dxl);
  to_arith(r[len - 2], dxr);
  to_arith(r[len - 1], tau_t);
  to_arith(dt, dtr);
  __syncthreads();  // every record is read: its space takes the fluxes
  Gas<R> gas;
  to_arith(gas_d.bK, gas.bK);
  to_arith(gas_d.ibK, gas.ibK);
  to_arith(gas_d.K, gas.K);
  to_arith(gas_d.mu, gas.mu);
  to_arith(gas_d.C_a, gas.C_a);
  // the distances are the caller's: infinity stands for a side without a gradient, and its reciprocal is zero
  const R idxl = g_div_full(R(1), dxl), idxr = g_div_full(R(1), dxr);
  // the same flux code as the step kernels: in single precision the two sides
  // of the face on the paired FP32 instructions
  if constexpr (std::is_same<R, float>::value)
    face_flux_ps_inv<D, MULTID, RAR>(wl, wr, cl, cr, sl, sr, tl, tr, idxl, idxr, tau_t, dtr, gas, abar_t0, F, &tau);
  else
    face_flux_inv<D, R, MULTID, RAR>(wl, wr, cl, cr, sl, sr, tl, tr, idxl, idxr, tau_t, dtr, gas, abar_t0, F, &tau);
  if (tid < nf) {
#pragma unroll
    for (int v = 0; v < nv; ++v) rec[tid * nv + v] = (double)F[v];
    if (tout) tout[f0 + tid] = (double)tau;
  }
  __syncthreads();
  for (int i = tid; i < nf * nv; i += kFaceT) Fout[f0 * nv + i] = rec[i];
}

template <int D, class R, bool M>
static void go(bool rar, int abar_t0, double gamma, double mu, double C_a, double dt, const double* faces, long n,
               double* F, double* tau, cudaStream_t s) {
  const unsigned blocks = (unsigned)((n + kFaceT - 1) / kFaceT);
  const Gas<double> gas{2.0 / (gamma - 1.0), (gamma - 1.0) / 2.0, 2.0 / (gamma - 1.0) - D, mu, C_a};
  if (rar)
    face_kernel<D, R, M, true><<<blocks, kFaceT, 0, s>>>(abar_t0, gas, dt, faces, n, F, tau);
  else
    face_kernel<D, R, M, false><<<blocks, kFaceT, 0, s>>>(abar_t0, gas, dt, faces, n, F, tau);
}

void launch_face_flux(int D, int prec, bool multid, int abar_t0, int rar, double gamma, double mu, double C_a,
                      double dt, const double* faces, long n, double* F, double* tau, cudaStream_t s) {
  const bool f64 = prec == 0, r = rar != 0;
  if (D == 1) {
    if (f64) go<1, double, false>(r, abar_t0, gamma, mu, C_a, dt, faces, n, F, tau, s);
    else go<1, float, false>(r, abar_t0, gamma, mu, C_a, dt, faces, n, F, tau, s);
  } else if (D == 2) {
    if (f64) {
      if (multid) go<2, double, true>(r, abar_t0, gamma, mu, C_a, dt, faces, n, F, tau, s);
      else go<2, double, false>(r, abar_t0, gamma, mu, C_a, dt, faces, n, F, tau, s);
    } else {
      if (multid) go<2, float, true>(r, abar_t0, gamma, mu, C_a, dt, faces, n, F, tau, s);
      else go<2, float, false>(r, abar_t0, gamma, mu, C_a, dt, faces, n, F, tau, s);
    }
  } else {
    if (f64) {
      if (multid) go<3, double, true>(r, abar_t0, gamma, mu, C_a, dt, faces, n, F, tau, s);
      else go<3, double, false>(r, abar_t0, gamma, mu, C_a, dt, faces, n, F, tau, s);
    } else {
      if (multid) go<3, float, true>(r, abar_t0, gamma, mu, C_a, dt, faces, n, F, tau, s);
      else go<3, float, false>(r, abar_t0, gamma, mu, C_a, dt, faces, n, F, tau, s);
    }
  }
}

}  // namespace gks
