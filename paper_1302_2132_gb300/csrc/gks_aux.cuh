// Kernels shared by the single-solve C ABI and the serving layer: state conversion between caller
// layouts and the stored form, the CFL rate of a stored state, and control-block parameters.
#pragma once
#include <cuda_runtime.h>

#include "gks.h"
#include "gks_step.cuh"

namespace gks {
namespace aux {

template <class Tin>
__global__ void state_in_kernel(const Tin* src, int layout, int D, long ncell, double gamma, int prec,
                                void* W, float* Wlo) {
  const long c = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= ncell) return;
  const int nv = D + 2;
  double w[5];
  for (int v = 0; v < nv; ++v) w[v] = (double)(layout == GKS_LAYOUT_AOS_CONS ? src[c * nv + v] : src[v * ncell + c]);
  if (layout == GKS_LAYOUT_SOA_PRIM) {
    const double rho = w[0], p = w[D + 1];
    double q = 0.0;
    for (int i = 0; i < D; ++i) {
      q += w[1 + i] * w[1 + i];
      w[1 + i] = rho * w[1 + i];
    }
    w[D + 1] = p / (gamma - 1.0) + 0.5 * rho * q;
  }
  for (int v = 0; v < nv; ++v) {
    if (prec == PREC_F32) {
      const float hi = (float)w[v];
      ((float*)W)[v * ncell + c] = hi;
      Wlo[v * ncell + c] = (float)(w[v] - (double)hi);
    } else {
      ((double*)W)[v * ncell + c] = w[v];
    }
  }
}

template <class Tout>
__global__ void state_out_kernel(Tout* dst, int layout, int D, long ncell, double gamma, int prec, const void* W,
                                 const float* Wlo) {
  const long c = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= ncell) return;
  const int nv = D + 2;
  double w[5];
  for (int v = 0; v < nv; ++v)
    w[v] = prec == PREC_F32 ? (double)((const float*)W)[v * ncell + c] + (double)Wlo[v * ncell + c]
                            : ((const double*)W)[v * ncell + c];
  if (layout == GKS_LAYOUT_SOA_PRIM) {
    double q = 0.0;
    for (int i = 0; i < D; ++i) q += w[1 + i] * w[1 + i];
    const double p = (gamma - 1.0) * (w[D + 1] - 0.5 * q / w[0]);
    for (int i = 0; i < D; ++i) w[1 + i] = w[1 + i] / w[0];
    w[D + 1] = p;
  }
  for (int v = 0; v < nv; ++v) {
    if (layout == GKS_LAYOUT_AOS_CONS)
      dst[c * nv + v] = (Tout)w[v];
    else
      dst[v * ncell + c] = (Tout)w[v];
  }
}

template <class Tin, class Tout>
__global__ void field_kernel(const Tin* src, Tout* dst, long n) {
  const long c = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (c < n) dst[c] = (Tout)src[c];
}

// f *= rho (scale = 1) or out = f / rho (scale = 0) with rho the density of a stored state; the
// conversions between k, omega and the transported rho k, rho omega
template <class R, class S>
__global__ void density_scale_kernel(R* f, const S* W, long n) {
  const long c = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (c < n) f[c] = f[c] * (R)W[c];
}
template <class R, class S, class O>
__global__ void density_unscale_kernel(const R* f, const S* W, O* out, long n) {
  const long c = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (c < n) out[c] = (O)(f[c] / (R)W[c]);
}

template <class T>
__global__ void copy_kernel(const T* src, T* dst, long n) {
  const long c = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (c < n) dst[c] = src[c];
}

// CFL rate of the stored state into ctrl->rate[slot] (a step computes it for its successor); a cell
// with rho <= 0 or p <= 0 sets the non-physical status bit, as the step's update does.
template <int D, int PREC>
__global__ void __launch_bounds__(kThreads) rate_kernel(const __grid_constant__ StepArgs A) {
  using R = typename PrecT<PREC>::R;
  __shared__ double red[kMaxWarps];
  const DevGrid& g = A.g;
  const Consts<R> kc = make_consts<R>(g);
  R rmax = R(0);
  int bad = 0;
  for (long c = (long)blockIdx.x * blockDim.x + threadIdx.x; c < g.ncell; c += (long)gridDim.x * blockDim.x) {
    R w[D + 2];
    load_stored<D, PREC>(A.g, A.Win, c, w);
    int pos[3];
    pos[0] = (int)(c % g.n[0]);
    pos[1] = (int)((c / g.n[0]) % g.n[1]);
    pos[2] = (int)(c / ((long)g.n[0] * g.n[1]));
    R ih[D];
    for (int d = 0; d < D; ++d) ih[d] = g_rcp((R)g.w[d][pos[d] + kWG]);
    if (!(w[0] > R(0)) || !(pressure_of<R>(D, kc.gamma, w) > R(0))) bad = 1;
    rmax = fmax(rmax, cell_rate_inv<D, R>(w, kc.gamma, ih));
  }
  const double m = block_max<double>((double)rmax, red);
  if (threadIdx.x == 0) atomic_max_nonneg(&A.ctrl->rate[A.slot], m);
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(&A.ctrl->status, 1u);
}

// Residual norms of the step that took Win to Wout: l2 += (dW/dt)^2, linf = max |dW|/dt, total += W volume (area: per
// cell, body-fitted grids; null: the product of the widths).  It runs after the last step of a call only, so the
// step kernels carry none of it.  The increment is the difference of the stored states, in double in every
// precision.  Doubles run at 1/64 of the FP32 rate on this part and bound it: four double operations per value (six of
// a float pair), dt divided out once per CTA, and a reduction in shared memory in which one warp
// adds up one quantity (T/32 + 5 additions a lane, against five per quantity in every warp).
// Accumulated inside the step kernel the norms took 115 us of that step at 1024^2 with the double state, and
// their code 5% of every other step (the 49-step call 4.82 -> 4.53 ms, 160^3 x 7 steps 7.65 -> 6.67 ms).
template <int D, int PREC>
__global__ void __launch_bounds__(kThreads) residual_kernel(const __grid_constant__ StepArgs A, const double* area) {
  using S = typename PrecT<PREC>::S;
  constexpr int NV = D + 2, T = kThreads, NW = T / 32;
  __shared__ double sums[2 * NV * T];
  __shared__ double maxs[NV * T];
  const DevGrid& g = A.g;
  const double dt = A.ctrl->last_dt;
  if (dt == 0.0) return;  // past t_end: the state was carried over
  const int tid = threadIdx.x;
  double s2[NV], tot[NV], mx[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    s2[v] = tot[v] = mx[v] = 0.0;
  }
  const S* W0 = (const S*)A.Win;
  const S* W1 = (const S*)A.Wout;
  for (long c = (long)blockIdx.x * T + tid; c < g.ncell; c += (long)gridDim.x * T) {
    double vol;
    if (area) {
      vol = area[c];
    } else {
      vol = g.w[0][(int)(c % g.n[0]) + kWG];
      if (D >= 2) vol *= g.w[1][(int)((c / g.n[0]) % g.n[1]) + kWG];
      if (D >= 3) vol *= g.w[2][(int)(c / ((long)g.n[0] * g.n[1])) + kWG];
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const long i = (long)v * g.ncell + c;
      double w, r;
      if constexpr (PREC == PREC_F32) {  // a float pair is its sum, exactly
        w = f2d(W1[i]) + f2d(A.Wout_lo[i]);
        r = w - (f2d(W0[i]) + f2d(A.Win_lo[i]));
      } else {
        w = W1[i];
        r = w - W0[i];
      }
      mx[v] = fmax(mx[v], fabs(r));
      s2[v] += r * r;
      tot[v] += w * vol;
    }
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    sums[v * T + tid] = s2[v];
    sums[(NV + v) * T + tid] = tot[v];
    maxs[v * T + tid] = mx[v];
  }
  __syncthreads();
  const int lane = tid & 31;
  for (int q = tid >> 5; q < 3 * NV; q += NW) {
    if (q < 2 * NV) {
      double s = sums[q * T + lane];
#pragma unroll
      for (int k = 1; k < NW; ++k) s += sums[q * T + lane + 32 * k];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) {
        if (q < NV)
          atomicAdd(&A.ctrl->l2[q], s / dt / dt);
        else
          atomicAdd(&A.ctrl->total[q - NV], s);
      }
    } else {
      double m = maxs[(q - 2 * NV) * T + lane];
#pragma unroll
      for (int k = 1; k < NW; ++k) m = fmax(m, maxs[(q - 2 * NV) * T + lane + 32 * k]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
      if (lane == 0) atomic_max_nonneg(&A.ctrl->linf[q - 2 * NV], m / dt);
    }
  }
}

template <int unused = 0>
__global__ void set_params_kernel(Ctrl* c, double dt_fixed, double cfl, double t_end) {
  c->dt_fixed = dt_fixed;
  c->cfl = cfl;
  c->t_end = t_end;
  for (int v = 0; v < 5; ++v) {
    c->l2[v] = 0.0;
    c->total[v] = 0.0;
    c->linf[v] = 0ull;
  }
}

}  // namespace aux
}  // namespace gks
