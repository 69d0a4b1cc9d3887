// Per-interface BGK-Navier-Stokes flux of the gas-kinetic scheme (Righi 2013 Section 2, after
// Xu 2001), device code templated on the dimension D and the arithmetic type T.
//
// All quantities are in the frame of the face: velocity index 0 is the face normal (u), indices
// 1..D-1 the tangential directions (v, w).  Moments <.> are normalised by rho.  The Maxwellian of a
// state has lambda = rho/(2p) and K = bK - D internal degrees of freedom (bK = 2/(gamma-1)).
//
// The moments are taken in closed form.  A slope a . psi of a Maxwellian is the derivative of its
// logarithm, r + c.U'/theta + theta'/(2 theta^2) (c^2 + xi^2 - bK theta), with the peculiar velocity c, theta =
// 1/(2 lambda) = p/rho and the gradients (r = rho'/rho, U', theta') of the macroscopic variables.  The time slope A is
// then the Euler equations' time derivative, the full-line moments are the Navier-Stokes fluxes of those
// gradients, and the transverse velocities average out of a half-line moment before it is taken: what
// is left on a half line are one cubic and one quadratic polynomial in the normal velocity.  890
// operations per 2D multi-dimensional face and 1193 in 3D (moment tables: 1674 and 2767).  The kernels are bound
// by their instruction count, in single precision (issue and FP32 pipe about 58% busy) and in double (FP64 pipe 88%
// busy), so the step times followed: 1024^2 with the double state 122 -> 98 us, 512^2 in FP64 1.88 -> 1.33 ms, 160^3
// 1.59 -> 1.11 ms (84 us, 1.18 ms and 0.88 ms with the changes noted where they stand).
#pragma once
#ifndef GKS_HOST_COUNT
#include <cuda_runtime.h>
#endif
#include <math.h>

#include <type_traits>
#include "gks_f2.cuh"

#ifndef GKS_FN
#define GKS_FN __device__ __forceinline__
#endif

namespace gks {

template <class T> GKS_FN T g_sqrt(T x);
#ifdef GKS_HOST_COUNT
template <> GKS_FN float g_sqrt<float>(float x) { return sqrtf(x); }
#else
// single precision: the hardware approximate square root (relative error about 2^-23, no slow-path
// branch); double precision stays IEEE
template <> GKS_FN float g_sqrt<float>(float x) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
#endif
template <> GKS_FN double g_sqrt<double>(double x) { return sqrt(x); }
// 1/sqrt(x): the hardware approximate reciprocal square root in single precision, IEEE otherwise
template <class T> GKS_FN T g_rsqrt(T x) { return T(1) / g_sqrt(x); }
#ifndef GKS_HOST_COUNT
template <> GKS_FN float g_rsqrt<float>(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
#endif
template <class T> GKS_FN T g_exp(T x);
#ifdef GKS_HOST_COUNT
template <> GKS_FN float g_exp<float>(float x) { return expf(x); }
#endif
template <> GKS_FN double g_exp<double>(double x) { return exp(x); }
template <class T> GKS_FN T g_erfc(T x);
#ifdef GKS_HOST_COUNT
template <> GKS_FN float g_erfc<float>(float x) { return erfcf(x); }
#endif
template <> GKS_FN double g_erfc<double>(double x) { return erfc(x); }
template <class T> GKS_FN T g_abs(T x) { return x < T(0) ? -x : x; }
#ifndef GKS_HOST_COUNT
template <> GKS_FN float g_abs<float>(float x) { return fabsf(x); }
template <> GKS_FN double g_abs<double>(double x) { return fabs(x); }
#endif

// Products, sums and fused multiply-adds that are rounded as written (never contracted with their
// neighbours), for values that two kernels have to agree on to the last bit.
template <class T> GKS_FN T g_mul_rn(T a, T b) { return a * b; }
template <class T> GKS_FN T g_add_rn(T a, T b) { return a + b; }
template <class T> GKS_FN T g_fma_rn(T a, T b, T c) { return a * b + c; }
#ifndef GKS_HOST_COUNT
template <> GKS_FN float g_mul_rn<float>(float a, float b) { return __fmul_rn(a, b); }
template <> GKS_FN double g_mul_rn<double>(double a, double b) { return __dmul_rn(a, b); }
template <> GKS_FN float g_add_rn<float>(float a, float b) { return __fadd_rn(a, b); }
template <> GKS_FN double g_add_rn<double>(double a, double b) { return __dadd_rn(a, b); }
template <> GKS_FN float g_fma_rn<float>(float a, float b, float c) { return __fmaf_rn(a, b, c); }
template <> GKS_FN double g_fma_rn<double>(double a, double b, double c) { return __fma_rn(a, b, c); }
#endif

// Quotient and reciprocal: IEEE in double precision (the FP64 path matches the oracle to 1e-12);
// in single precision the hardware reciprocal (about 1 ulp), which avoids the multi-instruction
// IEEE sequence and its slow-path branch.  The FP32 form's tolerances are far above this error.  The
// flush-to-zero form of it needs a normal divisor and is shorter (1024^2 with the double state 91 -> 87.5 us per
// step, WENO-5 at 603 x 501 50 -> 45.8).  g_div_full takes any divisor, for those that are a caller's data (epsilon, omega,
// the distances of gks_face_flux).
template <class T> GKS_FN T g_div(T a, T b) { return a / b; }
template <class T> GKS_FN T g_rcp(T x) { return T(1) / x; }
template <class T> GKS_FN T g_div_full(T a, T b) { return a / b; }
// a density as a divisor: at least the smallest normal number (the host's quotients take any).  On the device
// each arithmetic type has its own, so that none goes without.
#ifdef GKS_HOST_COUNT
template <class T> GKS_FN T g_normal(T x) { return x; }
#else
template <class T> GKS_FN T g_normal(T x);
template <> GKS_FN float g_rcp<float>(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
template <> GKS_FN float g_div<float>(float a, float b) { return a * g_rcp<float>(b); }
template <> GKS_FN float g_div_full<float>(float a, float b) { return __fdividef(a, b); }
template <> GKS_FN float g_normal<float>(float x) { return fmaxf(x, 1.17549435e-38f); }
template <> GKS_FN double g_normal<double>(double x) { return fmax(x, 2.2250738585072014e-308); }
template <> GKS_FN F2 g_normal<F2>(F2 x) { return F2(g_normal<float>(x.v.x), g_normal<float>(x.v.y)); }
template <> GKS_FN float g_exp<float>(float x) { return __expf(x); }
// Double reciprocal and reciprocal square root of normal positive numbers (densities, temperatures, widths,
// sums of them): the hardware's approximation and one third-order step, r (1 + e + e^2) with e = 1 - x r, and
// y (1 + h/2 + 3 h^2/8) with h = 1 - x y^2 (the binomial series; Householder's iterations).  Three and five
// double operations, with no slow path: the FP64 pipe (one warp instruction per 64 clocks and sub-partition) is
// what the FP64 kernels wait for.  The reciprocal is within 0.505 units in the last place (a division within 0.5), the
// reciprocal square root closer than 1 / sqrt(x) by two IEEE operations, over a million arguments (2^-60 to 2^60).
// Quotients that may see zero or infinity keep the IEEE form (g_div).
template <> GKS_FN double g_rcp<double>(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  double e = __fma_rn(-x, r, 1.0);
  e = __fma_rn(e, e, e);
  return __fma_rn(r, e, r);
}
template <> GKS_FN double g_rsqrt<double>(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double h = __fma_rn(-x * y, y, 1.0);
  return __fma_rn(y * h, __fma_rn(0.375, h, 0.5), y);
}

// Single-precision erfc from the Chebyshev-fitted form of Press, Teukolsky, Vetterling and Flannery
// (Numerical Recipes, 2nd ed., section 6.2): for z = |x|, t = 1/(1 + z/2),
// erfc(z) = t exp(-z^2 + P(t)) with a degree-9 polynomial P, fractional error below 1.2e-7;
// erfc(-z) = 2 - erfc(z).
GKS_FN float erfc_cheb(float x) {
  const float z = fabsf(x);
  const float t = g_rcp<float>(1.0f + 0.5f * z);
  const float c[10] = {-1.26551223f, 1.00002368f, 0.37409196f, 0.09678418f, -0.18628806f,
                       0.27886807f, -1.13520398f, 1.48851587f, -0.82215223f, 0.17087277f};
  float p = c[9];
#pragma unroll
  for (int i = 8; i >= 0; --i) p = fmaf(p, t, c[i]);
  const float r = t * __expf(p - z * z);
  return x >= 0.0f ? r : 2.0f - r;
}
template <> GKS_FN float g_erfc<float>(float x) { return erfc_cheb(x); }
#endif

// a / b from r, the reciprocal of b, for normal numbers whose quotient is normal.  In double the product is corrected by
// its exact remainder (Markstein's last step, which rounds as a division does); in single precision the product, as g_div.
template <class T> GKS_FN T g_quot_r(T a, T b, T r) {
  const T q = g_mul_rn<T>(a, r);
  if constexpr (std::is_same<T, double>::value)
    return g_fma_rn<T>(g_fma_rn<T>(-q, b, a), r, q);
  else
    return q;
}
template <class T> GKS_FN T g_quot(T a, T b) { return g_div(a, b); }
#ifndef GKS_HOST_COUNT
// (a reciprocal to 2^-40, by Newton's step, leaves the corrected quotient within 2^-28 units of the rounded one)
template <> GKS_FN double g_quot<double>(double a, double b) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(b));
  r = __fma_rn(r, __fma_rn(-b, r, 1.0), r);
  return g_quot_r<double>(a, b, r);
}
#endif

// erfc(x) and exp(-x^2) together.
template <class T> GKS_FN void g_gauss(T x, T& c, T& e) {
  c = g_erfc(x);
  e = g_exp(-x * x);
}
#ifndef GKS_HOST_COUNT
// In double one exponential serves both: for a = |x| >= 0, erfc(a) = exp(-a^2) w(a), and (1 + sqrt(pi) a) w(a), which is 1 at
// both ends, is a polynomial of degree 24 in t = (a - 3)/(a + 3) to 1.2e-17: its Chebyshev series on [-1, 1], computed
// in 60 digits (the mapping of Schonfelder and of Shepherd and Laframboise for this function), its leading coefficient
// in two parts.  The roundings of a^2, of the polynomial's last step and of the quotient are carried to first order into
// the last operation, so that of the error little more than the exponential's is left: relative error of erfc at most
// 4.0e-16 where it is normal (CUDA's 4.7e-16), 8.1e-17 in the root mean square (9.6e-17).  One exponential, the reciprocals
// above and the inverse widths in the update took the FP64 step from 1.34 to 1.13 ms at 512^2 (k-epsilon,
// multi-dimensional) and from 39.0 to 29.7 us on the 400-cell shock tube; of that the corrected quotients took back
// 23 and 0.6 us, these corrections 17 and 0.4.
template <> GKS_FN void g_gauss<double>(double x, double& c, double& e) {
  const double m0 = 1.130814990365315, m0l = 1.0122955773236472e-16;
  const double m[24] = {-0.15730767105387838, -0.0142078862510333066, 0.0978158787627484546, -0.0975498893780881991,
                        0.0577612034134763832, -0.0205803575852415208, 0.00232213762002999957, 0.00160587866420396248, -0.00068595951686176365,
                        -0.0000859074652169480687, 0.000109403210195641532, 3.47842163101718717e-6, -0.0000175723862950109043, -5.05198940975773676e-7,
                        3.0437515559732887e-6, 2.88623899544377934e-7, -5.43060517125976003e-7, -1.1920154572965122e-7, 9.02620167290913922e-8,
                        3.54129561773177263e-8, -1.1890984470997693e-8, -7.14018809267724831e-9, 8.88513573014043976e-10, 7.32248898966643554e-10};
  const double a = fabs(x), s = a * a;
  e = exp(-s);
  const double sl = __fma_rn(a, a, -s);
  const double d1 = a + 3.0, d2 = __fma_rn(1.7724538509055160273, a, 1.0);
  const double r = g_rcp(d1 * d2);
  const double rt = r * d2;  // 1 / d1
  double t = (a - 3.0) * rt;
  t = __fma_rn(__fma_rn(-t, d1, a - 3.0), rt, t);
  double p = m[23];
#pragma unroll
  for (int i = 22; i >= 0; --i) p = __fma_rn(p, t, m[i]);
  const double ph = __fma_rn(p, t, m0), pl = __fma_rn(p, t, m0 - ph) + m0l;
  const double rd = r * d1;  // 1 / d2
  const double w = ph * rd, wl = (__fma_rn(-w, d2, ph) + pl) * rd;
  // (far out the quotients are infinity times zero: erfc is zero there)
  const double q = a >= 28.0 ? 0.0 : __fma_rn(e, w, e * __fma_rn(-w, sl, wl));
  c = x >= 0.0 ? q : 2.0 - q;
}
#endif

// The same functions on two lanes (two faces per thread): reciprocals, exponentials and square roots
// per lane as in single precision, erfc from the same Chebyshev fit with paired arithmetic.
GKS_FN F2 g_rcp(F2 x) { return F2(g_rcp<float>(x.v.x), g_rcp<float>(x.v.y)); }
GKS_FN F2 g_div(F2 a, F2 b) { return F2(a * g_rcp(b)); }
GKS_FN F2 g_exp(F2 x) { return F2(g_exp<float>(x.v.x), g_exp<float>(x.v.y)); }
GKS_FN F2 g_sqrt(F2 x) { return F2(g_sqrt<float>(x.v.x), g_sqrt<float>(x.v.y)); }
GKS_FN F2 g_rsqrt(F2 x) { return F2(g_rsqrt<float>(x.v.x), g_rsqrt<float>(x.v.y)); }
GKS_FN F2 g_abs(F2 x) { return F2(fabsf(x.v.x), fabsf(x.v.y)); }
GKS_FN F2 g_erfc(F2 x) {
  const F2 z = g_abs(x);
  const F2 t = g_rcp(F2(1.0f) + F2(0.5f) * z);
  const float c[10] = {-1.26551223f, 1.00002368f, 0.37409196f, 0.09678418f, -0.18628806f,
                       0.27886807f, -1.13520398f, 1.48851587f, -0.82215223f, 0.17087277f};
  F2 p = F2(c[9]);
#pragma unroll
  for (int i = 8; i >= 0; --i) p = p * t + F2(c[i]);
  const F2 r = F2(t * g_exp(p - z * z));
  return F2(x.v.x >= 0.0f ? r.v.x : 2.0f - r.v.x, x.v.y >= 0.0f ? r.v.y : 2.0f - r.v.y);
}
// a pending product as the argument: rounded first (exact overloads, so the templates above are not
// deduced with the product type)
GKS_FN F2 g_rcp(F2Mul x) { return g_rcp(F2(x)); }
GKS_FN F2 g_div(F2Mul a, F2Mul b) { return g_div(F2(a), F2(b)); }
GKS_FN F2 g_exp(F2Mul x) { return g_exp(F2(x)); }
GKS_FN F2 g_sqrt(F2Mul x) { return g_sqrt(F2(x)); }
GKS_FN F2 g_abs(F2Mul x) { return g_abs(F2(x)); }
GKS_FN F2 g_erfc(F2Mul x) { return g_erfc(F2(x)); }

constexpr double kInvSqrtPi = 0.56418958354775628695;  // 1/sqrt(pi)

template <int D> struct Dims {
  static constexpr int nv = D + 2;
  static constexpr int nt = D > 1 ? D - 1 : 1;  // storage for tangential arrays (>= 1)
};

// Macroscopic description of one Maxwellian.
template <int D, class T> struct Maxw {
  T rho, ir, U[D];  // ir = 1/rho
  T th, it;         // theta = 1/(2 lambda) = p/rho, and 1/theta
};

// Gas constants used by every face.
template <class T> struct Gas {
  T bK;   // K + D = 2/(gamma - 1)
  T ibK;  // 1 / bK
  T K;    // internal degrees of freedom
  T mu;   // molecular viscosity (tau_mol = mu / p)
  T C_a;  // artificial-dissipation coefficient (Eq. taua)
};

// (rho, U, theta) of the Maxwellian carrying the conservative state w (Section 2: E = (u^2 + xi^2)/2,
// so rho E = rho (|U|^2 + bK theta) / 2).  Two reciprocals: 1/rho and 1/theta; ibK = 1/bK.
template <int D, class T>
GKS_FN Maxw<D, T> maxwellian(const T* w, T ibK) {
  Maxw<D, T> g;
  g.rho = w[0];
  g.ir = g_rcp(w[0]);
  T q = T(0);
#pragma unroll
  for (int i = 0; i < D; ++i) {
    g.U[i] = w[1 + i] * g.ir;
    q += g.U[i] * g.U[i];
  }
  // (2 rho E as a sum, exactly: the two-lane type would round one of two products before their difference)
  const T e2 = w[D + 1] + w[D + 1];
  g.th = (e2 - w[0] * q) * g.ir * ibK;
  g.it = g_rcp(g.th);
  return g;
}

// n eta_n = n <(u - U)^k>, k = 0..6, over u > 0 (sgn = +1) or u < 0 (sgn = -1), from the textbook half-line
// Gaussian integrals: <1> = erfc(-sgn U/sqrt(2 theta))/2, <u - U> = sgn sqrt(theta/(2 pi)) exp(-U^2/(2 theta)) =: b,
// and by parts <(u - U)^(k+2)> = (k + 1) theta <(u - U)^k> + (-U)^(k+1) b.
template <int D, class T>
GKS_FN void half_moments(const Maxw<D, T>& g, T sgn, T n, T* e) {
  T s2, z, c, x;  // sqrt(2 theta), U/sqrt(2 theta)
  if constexpr (std::is_same<T, double>::value) {
    const T y = g_rsqrt(T(2) * g.th);
    s2 = T(2) * g.th * y;
    z = g.U[0] * y;
  } else {
    s2 = g_sqrt(T(2) * g.th);
    z = T(0.5) * g.U[0] * s2 * g.it;
  }
  g_gauss(T(-sgn * z), c, x);
  e[0] = T(0.5) * n * c;
  e[1] = sgn * T(0.5 * kInvSqrtPi) * n * s2 * x;
  T b = e[1];
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    b = -g.U[0] * b;
    e[k + 2] = T(k + 1) * g.th * e[k] + b;
  }
}

// Gradients of the macroscopic variables along one direction.
template <int D, class T> struct Grad {
  T r, U[D], th;  // rho'/rho, U', theta'
};
// ... from r = W'/rho: W_E' = (rho (|U|^2 + bK theta)/2)'.
template <int D, class T>
GKS_FN void gradient(const Maxw<D, T>& g, T bK, T ibK, const T* r, Grad<D, T>& o) {
  T c = bK * g.th, UU = T(0);
#pragma unroll
  for (int i = 0; i < D; ++i) {
    c += g.U[i] * g.U[i];
    o.U[i] = r[1 + i] - g.U[i] * r[0];
    UU += g.U[i] * o.U[i];
  }
  o.r = r[0];
  o.th = (T(2) * (r[D + 1] - UU) - c * r[0]) * ibK;
}

// Minus the Euler time derivatives of (r, U, theta) from the gradients along the normal (gx) and the
// tangential axes (gs, multi-dimensional expansion only): convection, dilatation and pressure.  This is
// -A of the compatibility condition <(a u + b v + A) psi> = 0 (Eq. initialf0).
template <int D, class T, bool MULTID>
GKS_FN void euler_rate(const Maxw<D, T>& g, T ibK, const Grad<D, T>& gx, const Grad<D, T>* gs, T& S, T& div,
                       Grad<D, T>& N) {
  S = T(0);  // sum of the tangential dilatations
  div = gx.U[0];
  if (MULTID) {
#pragma unroll
    for (int q = 0; q < D - 1; ++q) S += gs[q].U[1 + q];
    div = gx.U[0] + S;
  }
  N.r = g.U[0] * gx.r + div;
  N.U[0] = g.U[0] * gx.U[0] + (g.th * gx.r + gx.th);
  N.th = g.U[0] * gx.th + T(2) * ibK * (g.th * div);
#pragma unroll
  for (int i = 1; i < D; ++i) N.U[i] = g.U[0] * gx.U[i];
  if (MULTID) {
#pragma unroll
    for (int q = 0; q < D - 1; ++q) {
      const T V = g.U[1 + q];
      N.r += V * gs[q].r;
      N.th += V * gs[q].th;
#pragma unroll
      for (int i = 0; i < D; ++i) N.U[i] += V * gs[q].U[i];
      N.U[1 + q] += g.th * gs[q].r + gs[q].th;
    }
  }
}

enum { LIM_MINMOD = 0, LIM_VANLEER = 1 };

// Slope limiter on one conservative variable: minmod(a, b) = (sgn a + sgn b)/2 min(|a|, |b|), or
// van Leer (a b + |a b|)/(a + b), zero unless a b > 0.
template <class R>
GKS_FN R limiter(int lim, R a, R b) {
  if (lim == LIM_MINMOD) {
    const R sa = R((a > R(0)) - (a < R(0))), sb = R((b > R(0)) - (b < R(0)));
    const R ma = g_abs(a), mb = g_abs(b);
    return R(0.5) * (sa + sb) * (ma < mb ? ma : mb);
  }
  return (a * b > R(0)) ? g_quot(R(2) * a * b, a + b) : R(0);
}

// Higher-order face values in index space (Section 4 lists third-order MUSCL and fifth-order
// WENO beside the second-order default).  muscl3_right(a, b, c) is cell b's value at its right face
// from cells a, b, c; muscl3_left(a, b, c) cell b's value at its left face: the kappa = 1/3 scheme
// with each one-sided difference limited by minmod against 4 times the other.
template <class R>
GKS_FN R muscl3_right(R a, R b, R c) {
  const R dm = b - a, dp = c - b;
  return b + limiter<R>(LIM_MINMOD, dm, R(4) * dp) * R(1.0 / 6.0) + limiter<R>(LIM_MINMOD, dp, R(4) * dm) * R(1.0 / 3.0);
}
template <class R>
GKS_FN R muscl3_left(R a, R b, R c) {
  const R dm = b - a, dp = c - b;
  return b - limiter<R>(LIM_MINMOD, dp, R(4) * dm) * R(1.0 / 6.0) - limiter<R>(LIM_MINMOD, dm, R(4) * dp) * R(1.0 / 3.0);
}
// Jiang and Shu's WENO-5: the value at the face to the right of c from cells a, b, c, d, e
// (candidate stencils' face values, smoothness indicators with 13/12 and 1/4, linear weights
// 1/10, 6/10, 3/10, epsilon 1e-6).
template <class R>
GKS_FN R weno5(R a, R b, R c, R d, R e) {
  const R s6 = R(1.0 / 6.0), c13 = R(13.0 / 12.0);
  const R q0 = (R(2) * a - R(7) * b + R(11) * c) * s6;
  const R q1 = (-b + R(5) * c + R(2) * d) * s6;
  const R q2 = (R(2) * c + R(5) * d - e) * s6;
  const R t0 = a - R(2) * b + c, u0 = a - R(4) * b + R(3) * c;
  const R t1 = b - R(2) * c + d, u1 = b - d;
  const R t2 = c - R(2) * d + e, u2 = R(3) * c - R(4) * d + e;
  const R b0 = c13 * t0 * t0 + R(0.25) * u0 * u0;
  const R b1 = c13 * t1 * t1 + R(0.25) * u1 * u1;
  const R b2 = c13 * t2 * t2 + R(0.25) * u2 * u2;
  const R eps = R(1e-6);
  const R a0 = g_div(R(0.1), (eps + b0) * (eps + b0));
  const R a1 = g_div(R(0.6), (eps + b1) * (eps + b1));
  const R a2 = g_div(R(0.3), (eps + b2) * (eps + b2));
  return g_div(a0 * q0 + a1 * q1 + a2 * q2, a0 + a1 + a2);
}

// Both sides of the face between c and d of the cells a..f; in single precision on the paired
// instructions (603 x 501, float pair, 45.8 -> 43.5 us per step against one side after the other).
template <class R>
GKS_FN void weno5_sides(R a, R b, R c, R d, R e, R f, R& wl, R& wr) {
  if constexpr (std::is_same<R, float>::value) {
    const F2 w = weno5<F2>(F2(a, f), F2(b, e), F2(c, d), F2(d, c), F2(e, b));
    wl = w.v.x;
    wr = w.v.y;
  } else {
    wl = weno5<R>(a, b, c, d, e);
    wr = weno5<R>(f, e, d, c, b);
  }
}

// Time integrals over [0, dt] of Eq. resultingf, e = exp(-t/tau):
//   T0 = int (1 - e), T1 = int ((tau + t) e - tau), T2 = int (t - tau + tau e), T3 = int e,
//   T4 = -int (tau + t) e, T5 = -tau int e, Dn = dt^2/2 - T2;
// the flux uses T0, T2, T3, Dn and the ratios r1 = T1/Dn, r4 = T4/Dn, r45 = (T4 - T5)/Dn (finite as
// tau -> 0).  With x = dt/tau and phi_k(x) = sum_m (-x)^m/(m+k)!: T0 = dt x phi2, T2 = dt^2 x phi3, T3 = dt phi1,
// Dn = dt^2 phi2, r1 = -x (phi2 - 2 phi3)/phi2, r4 = (e - 2 phi1)/(x phi2), r45 = -(phi1 - phi2)/phi2.
// For x < 1 phi3 is summed from its series and phi2, phi1, e by the backward recurrence
// phi_{k-1} = 1/(k-1)! - x phi_k (no cancellation), in the arithmetic type; otherwise the closed
// forms in e = exp(-x) are used.
template <class T> struct TimeCoef {
  T T0, T2, T3, Dn, r1, r4, r45;
};

// phi3 = sum_m (-x)^m / (m+3)! by Horner, then phi2, phi1 and e = exp(-x) by the backward recurrence
// phi_{k-1} = 1/(k-1)! - x phi_k.  For 0 <= x < 1 every step is free of cancellation; 18 terms
// reach double precision, 12 leave a truncation below 1e-9 (enough in single precision).
template <class T>
GKS_FN void phi_series(T x, T& p1, T& p2, T& p3, T& e) {
  T s;
  if constexpr (std::is_same<T, double>::value) {
    const double c[18] = {1.0 / 6, 1.0 / 24, 1.0 / 120, 1.0 / 720, 1.0 / 5040, 1.0 / 40320, 1.0 / 362880,
                          1.0 / 3628800, 1.0 / 39916800, 1.0 / 479001600, 1.0 / 6227020800.0,
                          1.0 / 87178291200.0, 1.0 / 1307674368000.0, 1.0 / 20922789888000.0,
                          1.0 / 355687428096000.0, 1.0 / 6402373705728000.0, 1.0 / 121645100408832000.0,
                          1.0 / 2432902008176640000.0};
    s = c[17];
#pragma unroll
    for (int m = 16; m >= 0; --m) s = c[m] - x * s;
  } else {
    // single-precision coefficients written as such, so that no double-to-float conversion (an FP64
    // pipe instruction) is left in the series
    const float c[12] = {1.0f / 6, 1.0f / 24, 1.0f / 120, 1.0f / 720, 1.0f / 5040, 1.0f / 40320, 1.0f / 362880,
                         1.0f / 3628800, 1.0f / 39916800, 1.0f / 479001600, 1.0f / 6227020800.0f,
                         1.0f / 87178291200.0f};
    s = T(c[11]);
#pragma unroll
    for (int m = 10; m >= 0; --m) s = T(c[m]) - x * s;
  }
  p3 = s;
  p2 = T(0.5) - x * p3;
  p1 = T(1) - x * p2;
  e = T(1) - x * p1;
}

template <class T>
GKS_FN void time_coeffs(T dt, T tau, TimeCoef<T>& c) {
  const T x = g_div(dt, tau);
  const T y = tau * g_rcp(g_normal(dt));
  if (x < T(1)) {
    // series branch (phi_k summed, no cancellation) in the arithmetic type
    T p1, p2, p3, e;
    phi_series<T>(x, p1, p2, p3, e);
    const T i2 = g_rcp(p2);
    c.T0 = dt * x * p2;
    c.T2 = dt * dt * x * p3;
    c.T3 = dt * p1;
    c.Dn = dt * dt * p2;
    c.r1 = -x * (p2 - T(2) * p3) * i2;
    c.r4 = (e - T(2) * p1) * i2 * y;
    c.r45 = (p2 - p1) * i2;
  } else {
    const T e = g_exp(-x);
    const T yq = y - y * e;
    const T P = T(1) - yq;
    const T inv = g_rcp(P);
    c.T0 = dt * P;
    c.Dn = tau * c.T0;
    c.T2 = T(0.5) * dt * dt - c.Dn;
    c.T3 = dt * yq;
    c.r1 = (T(2) * yq - (T(1) + e)) * inv;
    c.r4 = (e - T(2) * yq) * inv;
    c.r45 = (e - yq) * inv;
  }
}

// Two lanes: both branches of time_coeffs, each lane keeping its own (x < 1: the series).
template <>
GKS_FN void time_coeffs<F2>(F2 dt, F2 tau, TimeCoef<F2>& c) {
  TimeCoef<float> a, b;
  time_coeffs<float>(dt.v.x, tau.v.x, a);
  time_coeffs<float>(dt.v.y, tau.v.y, b);
  c.T0 = F2(a.T0, b.T0);
  c.T2 = F2(a.T2, b.T2);
  c.T3 = F2(a.T3, b.T3);
  c.Dn = F2(a.Dn, b.Dn);
  c.r1 = F2(a.r1, b.r1);
  c.r4 = F2(a.r4, b.r4);
  c.r45 = F2(a.r45, b.r45);
}

// The time coefficients with the degree of rarefaction eps in place of tau/dt (Eqs. tautautilde,
// rarefactionkepsilon, epsilonkomega): Eq. fkepsilon with alpha = eps (1 - e^{-1/eps}) and
// beta = e^{-1/eps} (Eq. alphabetakepsilon with the corrected beta):
//   T0 = dt (1 - alpha), T2 = dt (dt/2 - tau (1 - alpha)), T3 = dt alpha, Dn = dt tau (1 - alpha),
//   r1 = (2 alpha - 1 - beta)/(1 - alpha), r4 = (beta - 2 alpha)/(1 - alpha), r45 = (beta - alpha)/(1 - alpha).
// eps = tau/dt gives time_coeffs.  For eps > 1 (x = 1/eps < 1) alpha = phi1(x), 1 - alpha = x phi2,
// 2 alpha - 1 - beta = -x^2 (phi2 - 2 phi3), beta - alpha = -x (phi1 - phi2), from the cancellation-free series.
template <class T>
GKS_FN void time_coeffs_hat(T dt, T tau, T eps, TimeCoef<T>& c) {
  T a, one_a, c1, c4, c45;
  if (eps > T(1)) {
    const T x = g_rcp(eps);
    T p1, p2, p3, e;
    phi_series<T>(x, p1, p2, p3, e);
    a = p1;
    one_a = x * p2;
    c1 = -x * x * (p2 - T(2) * p3);
    c4 = e - T(2) * p1;
    c45 = x * (p2 - p1);
  } else {
    const T beta = eps > T(0) ? g_exp(-g_div(T(1), eps)) : T(0);
    a = eps * (T(1) - beta);
    one_a = T(1) - a;
    c1 = T(2) * a - T(1) - beta;
    c4 = beta - T(2) * a;
    c45 = beta - a;
  }
  const T i1 = g_rcp(one_a);
  c.T0 = dt * one_a;
  c.T2 = dt * (T(0.5) * dt - tau * one_a);
  c.T3 = dt * a;
  c.Dn = dt * tau * one_a;
  c.r1 = c1 * i1;
  c.r4 = c4 * i1;
  c.r45 = c45 * i1;
}

// One side of the initial state (Eq. initialf0): with the slopes sn (normal) and st (tangential) of its
// conservative variables and the half-line moments rho eta_n in e, the distribution
// q = r5 A + r4 (u a + v b) of the Abar condition and of the flux is, averaged over the transverse velocities,
//   <q>       = q0 + q1 c + q2 c^2 + q3 c^3,
//   <q c_k>   = k0 + k1 c + k2 c^2,                                      c = u - U, k a tangential axis,
//   <q w/2>   = (bK - 1) theta/2 <q> + e0 + e1 c,                        w = sum c_k^2 + xi^2,
// with the Euler rates N, the deviatoric strain and the heat-flux gradients as coefficients.  Returned in the
// frame moving with U0 (that of g0): its moments rhs = <q psi>, and F = Dn <u q psi> + T3 <u psi>.
// FO: a first-order face (no slopes): free transport only, rhs = 0.
template <int D, class T, bool MULTID, bool FO = false>
GKS_FN void side_terms(const Maxw<D, T>& g, const T* e, const T* sn, const T (*st)[D + 2], const T* U0, T bK, T ibK, T T3,
                       T Dn, T r4, T r45, T* rhs, T* F) {
  constexpr int nv = D + 2;
  const T k1d = bK - T(1), hk = T(0.5) * k1d * g.th;
  T m[nv], x[nv];  // moments of q psi and u q psi in the side's own frame
  if constexpr (FO) {
#pragma unroll
    for (int v = 0; v < nv; ++v) m[v] = x[v] = T(0);
  } else {
    Grad<D, T> gx, gs[Dims<D>::nt], N;
    T r[nv], S, div;
#pragma unroll
    for (int v = 0; v < nv; ++v) r[v] = sn[v] * g.ir;
    gradient<D, T>(g, bK, ibK, r, gx);
    if (MULTID) {
#pragma unroll
      for (int q = 0; q < D - 1; ++q) {
#pragma unroll
        for (int v = 0; v < nv; ++v) r[v] = st[q][v] * g.ir;
        gradient<D, T>(g, bK, ibK, r, gs[q]);
      }
    }
    euler_rate<D, T, MULTID>(g, ibK, gx, gs, S, div, N);
    const T sg = r4 * (gx.U[0] - ibK * div);  // deviatoric normal strain
    const T nu = r45 * (T(0.5) * g.it * N.th);
    const T h = nu + sg;
    const T ha = T(0.5) * r4 * gx.th, hai = ha * g.it;
    const T q0 = r45 * N.r - h, q1 = g.it * (r45 * N.U[0]) - T(3) * hai, q2 = g.it * h, q3 = hai * g.it;
    const T J0 = q0 * e[0] + q1 * e[1] + q2 * e[2] + q3 * e[3];
    const T J1 = q0 * e[1] + q1 * e[2] + q2 * e[3] + q3 * e[4];
    const T J2 = q0 * e[2] + q1 * e[3] + q2 * e[4] + q3 * e[5];
    const T J3 = q0 * e[3] + q1 * e[4] + q2 * e[5] + q3 * e[6];
    const T e0 = g.th * (k1d * nu - sg), e1 = k1d * ha;
    m[0] = J0;
    m[1] = J1;
    m[D + 1] = T(0.5) * J2 + hk * J0 + e0 * e[0] + e1 * e[1];
    x[0] = g.U[0] * J0 + J1;
    x[1] = g.U[0] * J1 + J2;
    x[D + 1] = g.U[0] * m[D + 1] + (T(0.5) * J3 + hk * J1 + e0 * e[1] + e1 * e[2]);
#pragma unroll
    for (int k = 0; k < D - 1; ++k) {
      T k0 = r45 * N.U[1 + k], k1 = r4 * gx.U[1 + k];
      if (MULTID) {
        const T hb = T(0.5) * r4 * gs[k].th, k2 = hb * g.it;
        k0 -= hb;
        k1 = r4 * (gx.U[1 + k] + gs[k].U[0]);
        m[2 + k] = k0 * e[0] + k1 * e[1] + k2 * e[2];
        x[2 + k] = g.U[0] * m[2 + k] + (k0 * e[1] + k1 * e[2] + k2 * e[3]);
      } else {
        m[2 + k] = k0 * e[0] + k1 * e[1];
        x[2 + k] = g.U[0] * m[2 + k] + (k0 * e[1] + k1 * e[2]);
      }
    }
  }
  // free transport <u psi> of the side
  const T V0 = g.U[0] * e[0] + e[1], VU = g.U[0] * e[1] + e[2];
  const T VE = T(0.5) * (g.U[0] * e[2] + e[3]) + hk * V0;
  x[0] = Dn * x[0] + T3 * V0;
  x[1] = Dn * x[1] + T3 * VU;
  x[D + 1] = Dn * x[D + 1] + T3 * VE;
#pragma unroll
  for (int k = 0; k < D - 1; ++k) x[2 + k] = Dn * x[2 + k];
  // into the frame of g0
  T hd2 = T(0), sm = m[D + 1], sx = x[D + 1];
  rhs[0] = m[0];
  F[0] = x[0];
#pragma unroll
  for (int i = 0; i < D; ++i) {
    const T d = g.U[i] - U0[i];
    hd2 += d * d;
    sm += d * m[1 + i];
    sx += d * x[1 + i];
    rhs[1 + i] = m[1 + i] + d * m[0];
    F[1 + i] = x[1 + i] + d * x[0];
  }
  hd2 = T(0.5) * hd2;
  rhs[D + 1] = sm + hd2 * m[0];
  F[D + 1] = sx + hd2 * x[0];
}

// The equilibrium state (Eq. eqlgform): gradients abar_l, abar_r from W_j -> w0 -> W_{j+1} and the mean
// tangential slopes.  <(u abar + v bbar) psi> over the full line with abar_r is the Euler rate N; what abar_l adds
// on u > 0 is the half-line part of d = abar_l - abar_r: rh = <u d psi>, fl = <u^2 d psi> (frame of g0).
template <int D, class T> struct EqTerms {
  Grad<D, T> N;
  T rh[D + 2], fl[D + 2];
  T sg, ux[Dims<D>::nt], thx;  // U' - div/bK, the shear sums and theta' of the full-line part (abar_r)
};
template <int D, class T, bool MULTID, class In>
GKS_FN void equilibrium_terms(const Maxw<D, T>& g, const T* w0, const In& in, T idxl, T idxr, T bK, T ibK,
                              EqTerms<D, T>& q) {
  constexpr int nv = D + 2;
  const T k1d = bK - T(1);
  Grad<D, T> gr, gd, gs[Dims<D>::nt];
  const T fl = g.ir * idxl, fr = g.ir * idxr;
  T r[nv], d[nv], S, div;
#pragma unroll
  for (int m = 0; m < nv; ++m) {
    r[m] = (in.c(1, m) - w0[m]) * fr;
    d[m] = (w0[m] - in.c(0, m)) * fl - r[m];
  }
  gradient<D, T>(g, bK, ibK, r, gr);
  gradient<D, T>(g, bK, ibK, d, gd);
  if (MULTID) {
    const T hi = T(0.5) * g.ir;
#pragma unroll
    for (int s = 0; s < D - 1; ++s) {
#pragma unroll
      for (int m = 0; m < nv; ++m) r[m] = (in.t(0, s, m) + in.t(1, s, m)) * hi;
      gradient<D, T>(g, bK, ibK, r, gs[s]);
    }
  }
  euler_rate<D, T, MULTID>(g, ibK, gr, gs, S, div, q.N);
  q.sg = gr.U[0] - ibK * div;
  q.thx = gr.th;
#pragma unroll
  for (int k = 0; k < D - 1; ++k) q.ux[k] = MULTID ? gr.U[1 + k] + gs[k].U[0] : gr.U[1 + k];
  // half line u > 0 of u d: <d> = b0 + b1 c + b2 c^2 over the transverse velocities
  T e[7];
  half_moments<D, T>(g, T(1), T(1), e);
  const T hg = T(0.5) * gd.th * g.it;
  const T b0 = gd.r - hg, b1 = gd.U[0] * g.it, b2 = hg * g.it;
  T L[5], M[4];
#pragma unroll
  for (int n = 0; n < 5; ++n) L[n] = b0 * e[n] + b1 * e[n + 1] + b2 * e[n + 2];
#pragma unroll
  for (int n = 0; n < 4; ++n) M[n] = g.U[0] * L[n] + L[n + 1];
  const T V0 = g.U[0] * e[0] + e[1], W2 = g.U[0] * V0 + (g.U[0] * e[1] + e[2]);
  const T hk = T(0.5) * k1d * g.th, dk = T(0.5) * k1d * gd.th;
  q.rh[0] = M[0];
  q.rh[1] = M[1];
  q.rh[D + 1] = T(0.5) * M[2] + hk * M[0] + dk * V0;
  q.fl[0] = g.U[0] * M[0] + M[1];
  q.fl[1] = g.U[0] * M[1] + M[2];
  q.fl[D + 1] = T(0.5) * (g.U[0] * M[2] + M[3]) + hk * q.fl[0] + dk * W2;
#pragma unroll
  for (int k = 0; k < D - 1; ++k) {
    q.rh[2 + k] = gd.U[1 + k] * V0;
    q.fl[2 + k] = gd.U[1 + k] * W2;
  }
}

// |D rho| = |d_t rho + U_n d_n rho| at the face for the rarefaction option (Eqs. tautautilde,
// tautilde): d_t rho = -rho0 (<abar_l . psi u>_{u>0} + <abar_r . psi u>_{u<0} + <bbar . psi v>) from
// the t = 0 compatibility condition of the equilibrium part, d_n rho the mean of the density slopes
// (w0 - W_j)/dxl and (W_{j+1} - w0)/dxr.
template <int D, class T, class In>
GKS_FN T face_drho(const Maxw<D, T>& g0, const EqTerms<D, T>& q, const T* w0, const In& in, T idxl, T idxr) {
  const T dn = T(0.5) * ((w0[0] - in.c(0, 0)) * idxl + (in.c(1, 0) - w0[0]) * idxr);
  return g_abs(g0.U[0] * dn - g0.rho * (q.N.r + q.rh[0]));
}

// Abar and the flux: rhs, F in the frame of g0 hold the two sides' parts (rho-weighted); on return F is
// the time-integrated flux in the frame of the face.
template <int D, class T>
GKS_FN void close_flux(const Maxw<D, T>& g, const EqTerms<D, T>& q, const TimeCoef<T>& c, int abar_t0, T bK, T ibK,
                       const T* rhs, T* F) {
  // Abar from the compatibility condition integrated over [0, dt] (or at t = 0), as gradients of
  // (r, U, theta); the full-line part enters as such
  T r1 = c.r1, ws = g.ir;
  if (abar_t0) {
    r1 = T(-1);
    ws = T(0);
  }
  const T e1 = c.Dn * c.r1;
  const T m0 = r1 * q.rh[0] + ws * rhs[0], mE = r1 * q.rh[D + 1] + ws * rhs[D + 1];
  // Z = T2 Abar + T1 N
  const T n1 = c.T2 * r1 + e1;
  const T Zr = c.T2 * m0 + n1 * q.N.r;
  const T Zt = c.T2 * (T(2) * ibK * mE - g.th * m0) + n1 * q.N.th;
  T Z[D];
#pragma unroll
  for (int i = 0; i < D; ++i) Z[i] = c.T2 * (r1 * q.rh[1 + i] + ws * rhs[1 + i]) + n1 * q.N.U[i];
  // rho0 <u (T0 + T2 Abar + T1 (u abar + v bbar)) psi>: Euler flux of the increments, stress and heat flux
  const T P = g.th * (Zr + c.T0) + Zt, hb = T(0.5) * bK, et = e1 * g.th;
  T f[D + 2];
  f[0] = g.U[0] * (Zr + c.T0) + Z[0] + e1 * q.fl[0];
  f[1] = g.U[0] * Z[0] + P + T(2) * et * q.sg + e1 * q.fl[1];
#pragma unroll
  for (int k = 0; k < D - 1; ++k) f[2 + k] = g.U[0] * Z[1 + k] + et * q.ux[k] + e1 * q.fl[2 + k];
  f[D + 1] = hb * (g.U[0] * P) + (hb + T(1)) * (g.th * Z[0] + et * q.thx) + e1 * q.fl[D + 1];
  // with the sides, and out of the moving frame
#pragma unroll
  for (int m = 0; m < D + 2; ++m) f[m] = g.rho * f[m] + F[m];
  T q2 = T(0), s = f[D + 1];
#pragma unroll
  for (int i = 0; i < D; ++i) {
    q2 += g.U[i] * g.U[i];
    s += g.U[i] * f[1 + i];
    F[1 + i] = f[1 + i] + g.U[i] * f[0];
  }
  F[0] = f[0];
  F[D + 1] = s + T(0.5) * q2 * f[0];
}

// w0 = sum over the sides of <psi> over their half lines (Eq. intermediatestate), the side's part: e the
// rho-weighted half-line moments.
template <int D, class T>
GKS_FN void side_state(const Maxw<D, T>& g, const T* e, T bK, T* w) {
  T c = (bK - T(1)) * g.th;
  w[0] = e[0];
  w[1] = g.U[0] * e[0] + e[1];
#pragma unroll
  for (int i = 0; i < D; ++i) c += g.U[i] * g.U[i];
#pragma unroll
  for (int k = 0; k < D - 1; ++k) w[2 + k] = g.U[1 + k] * e[0];
  w[D + 1] = T(0.5) * (e[2] + c * e[0]) + g.U[0] * e[1];
}

// One face.  Inputs in the face frame:
//   wl, wr   reconstructed states; cl, cr cell averages of the two cells; sl, sr normal slopes;
//   tl, tr   tangential slopes (multi-dimensional expansion only); idxl, idxr inverse centre-to-face
//            distances; tau_t turbulent relaxation time at the face; dt the time step.
// Output: F, the flux integrated over [0, dt] (Eq. fluxesf); tau_out the total relaxation time.
// RAR: the rarefaction option -- the degree of rarefaction eps = tau/tauhat, tauhat = rho0/|D rho|
// (capped at 1e30), replaces tau/dt inside the time coefficients (Eq. epsilonkomega).
// FO: a first-order face (the slopes are taken as zero and not read).
//
// The inputs other than wl, wr come through an accessor `in` (FaceArrays below): in.s(sd, m) the normal slope,
// in.c(sd, m) the cell average and in.t(sd, q, m) the q-th tangential slope of component m on side sd (0 left, 1
// right), each read where it is used.
template <int D, class T, bool MULTID, bool RAR = false, bool FO = false, class In>
GKS_FN void face_flux_in(const T* wl, const T* wr, const In& in, T idxl, T idxr, T tau_t, T dt, const Gas<T>& gas,
                         int abar_t0, T* F, T* tau_out) {
  constexpr int nv = D + 2;
  const T bK = gas.bK, ibK = gas.ibK;
  const Maxw<D, T> gl = maxwellian<D, T>(wl, ibK);
  const Maxw<D, T> gr = maxwellian<D, T>(wr, ibK);
  T w0[nv], w1[nv], el[7], er[7];
  half_moments<D, T>(gl, T(1), gl.rho, el);
  half_moments<D, T>(gr, T(-1), gr.rho, er);
  side_state<D, T>(gl, el, bK, w0);
  side_state<D, T>(gr, er, bK, w1);
#pragma unroll
  for (int m = 0; m < nv; ++m) w0[m] += w1[m];
  w0[0] = g_normal(w0[0]);  // (sides that separate fast leave next to nothing)
  const Maxw<D, T> g0 = maxwellian<D, T>(w0, ibK);
  // Eqs. relaxation time and taua: tau = mu/p0 + tau_t + C_a |p_r - p_l| / (p_r + p_l) dt
  const T pl = gl.rho * gl.th, pr = gr.rho * gr.th;
  const T tau = gas.mu * g0.ir * g0.it + tau_t + gas.C_a * g_abs(pr - pl) * g_rcp(T(pr + pl)) * dt;
  *tau_out = tau;
  TimeCoef<T> c;
  EqTerms<D, T> q;
  if constexpr (RAR) {
    equilibrium_terms<D, T, MULTID>(g0, w0, in, idxl, idxr, bK, ibK, q);
    const T drho = face_drho<D, T>(g0, q, w0, in, idxl, idxr);
    const T eps = drho > T(1e-30) * g0.rho ? g_div(tau * drho, g0.rho) : tau * T(1e-30);
    time_coeffs_hat<T>(dt, tau, eps, c);
  } else {
    time_coeffs<T>(dt, tau, c);
  }
  T rhs[nv];
#pragma unroll
  for (int m = 0; m < nv; ++m) rhs[m] = F[m] = T(0);
  // the two sides in one loop body
#pragma unroll 1
  for (int sd = 0; sd < 2; ++sd) {
    const Maxw<D, T> g = sd ? gr : gl;
    T e[7], sn[nv], st[Dims<D>::nt][nv], rs[nv], Fs[nv];
#pragma unroll
    for (int n = 0; n < 7; ++n) e[n] = sd ? er[n] : el[n];
#pragma unroll
    for (int m = 0; m < nv; ++m) sn[m] = FO ? T(0) : in.s(sd, m);
    if (MULTID) {
#pragma unroll
      for (int s = 0; s < D - 1; ++s)
#pragma unroll
        for (int m = 0; m < nv; ++m) st[s][m] = in.t(sd, s, m);
    }
    side_terms<D, T, MULTID, FO>(g, e, sn, st, g0.U, bK, ibK, c.T3, c.Dn, c.r4, c.r45, rs, Fs);
#pragma unroll
    for (int m = 0; m < nv; ++m) {
      rhs[m] += rs[m];
      F[m] += Fs[m];
    }
  }
  if constexpr (!RAR) equilibrium_terms<D, T, MULTID>(g0, w0, in, idxl, idxr, bK, ibK, q);
  close_flux<D, T>(g0, q, c, abar_t0, bK, ibK, rhs, F);
}

// Face inputs held in the caller's arrays (registers): sl, sr normal slopes, cl, cr cell averages,
// tl, tr tangential slopes (read only with the multi-dimensional expansion).
template <int D, class T> struct FaceArrays {
  const T *sl, *sr, *cl, *cr;
  const T (*tl)[D + 2];
  const T (*tr)[D + 2];
  GKS_FN T s(int sd, int m) const { return sd ? sr[m] : sl[m]; }
  GKS_FN T c(int sd, int m) const { return sd ? cr[m] : cl[m]; }
  GKS_FN T t(int sd, int q, int m) const { return sd ? tr[q][m] : tl[q][m]; }
};

// face_flux_in with the inputs in arrays and the inverse centre-to-face distances given.
template <int D, class T, bool MULTID, bool RAR = false>
GKS_FN void face_flux_inv(const T* wl, const T* wr, const T* cl, const T* cr, const T* sl, const T* sr,
                          const T (*tl)[D + 2], const T (*tr)[D + 2], T idxl, T idxr, T tau_t, T dt,
                          const Gas<T>& gas, int abar_t0, T* F, T* tau_out) {
  const FaceArrays<D, T> in{sl, sr, cl, cr, tl, tr};
  face_flux_in<D, T, MULTID, RAR>(wl, wr, in, idxl, idxr, tau_t, dt, gas, abar_t0, F, tau_out);
}

// face_flux with the inputs in arrays and the centre-to-face distances.
template <int D, class T, bool MULTID, bool RAR = false>
GKS_FN void face_flux(const T* wl, const T* wr, const T* cl, const T* cr, const T* sl, const T* sr,
                      const T (*tl)[D + 2], const T (*tr)[D + 2], T dxl, T dxr, T tau_t, T dt, const Gas<T>& gas,
                      int abar_t0, T* F, T* tau_out) {
  face_flux_inv<D, T, MULTID, RAR>(wl, wr, cl, cr, sl, sr, tl, tr, g_rcp(dxl), g_rcp(dxr), tau_t, dt, gas, abar_t0, F,
                                   tau_out);
}

// face_flux_in in single precision with the two sides of the face evaluated together on the paired
// FP32 instructions: lane x carries the left Maxwellian on u > 0, lane y the right one on u < 0, for
// the intermediate state and the sides' parts of the Abar right-hand side and of the flux.  The paired sums
// are added lane x + lane y at the end of each part.  Same terms as face_flux_in; the artificial part of tau is
// skipped when C_a = 0.
template <int D, bool MULTID, bool RAR = false, bool FO = false, class In>
GKS_FN void face_flux_ps(const float* wl, const float* wr, const In& in, float idxl, float idxr, float tau_t, float dt,
                         const Gas<float>& gas, int abar_t0, float* F, float* tau_out) {
  using T = float;
  constexpr int nv = D + 2;
  const T bK = gas.bK, ibK = gas.ibK;
  F2 w2[nv];
#pragma unroll
  for (int m = 0; m < nv; ++m) w2[m] = F2(wl[m], wr[m]);
  const Maxw<D, F2> gs = maxwellian<D, F2>(w2, F2(ibK));
  F2 e[7];  // rho eta_n over u > 0 (left) and u < 0 (right)
  half_moments<D, F2>(gs, F2(1.0f, -1.0f), gs.rho, e);
  T w0[nv];
  {
    F2 q[nv];
    side_state<D, F2>(gs, e, F2(bK), q);
#pragma unroll
    for (int m = 0; m < nv; ++m) w0[m] = q[m].v.x + q[m].v.y;
  }
  w0[0] = g_normal(w0[0]);  // (sides that separate fast leave next to nothing)
  const Maxw<D, T> g0 = maxwellian<D, T>(w0, ibK);
  // Eqs. relaxation time and taua; the artificial part only with C_a > 0
  T tau = gas.mu * g0.it * g0.ir + tau_t;
  if (gas.C_a != T(0)) {
    // p_r - p_l and p_r + p_l with p_r unrounded
    const T rr = gs.rho.v.y, tr = gs.th.v.y, pl = gs.rho.v.x * gs.th.v.x;
    tau += g_div(gas.C_a * g_abs(g_fma_rn(rr, tr, -pl)), g_fma_rn(rr, tr, pl)) * dt;
  }
  *tau_out = tau;
  TimeCoef<T> c;
  EqTerms<D, T> q;
  if constexpr (RAR) {
    equilibrium_terms<D, T, MULTID>(g0, w0, in, idxl, idxr, bK, ibK, q);
    const T drho = face_drho<D, T>(g0, q, w0, in, idxl, idxr);
    const T eps = drho > T(1e-30) * g0.rho ? g_div(tau * drho, g0.rho) : tau * T(1e-30);
    time_coeffs_hat<T>(dt, tau, eps, c);
  } else {
    time_coeffs<T>(dt, tau, c);
  }
  T rhs[nv];
  {
    F2 sn[nv], st[Dims<D>::nt][nv], U0[D], rs[nv], Fs[nv];
#pragma unroll
    for (int m = 0; m < nv; ++m) sn[m] = FO ? F2(0.0f) : F2(in.s(0, m), in.s(1, m));
    if (MULTID) {
#pragma unroll
      for (int s = 0; s < D - 1; ++s)
#pragma unroll
        for (int m = 0; m < nv; ++m) st[s][m] = F2(in.t(0, s, m), in.t(1, s, m));
    }
#pragma unroll
    for (int i = 0; i < D; ++i) U0[i] = F2(g0.U[i]);
    side_terms<D, F2, MULTID, FO>(gs, e, sn, st, U0, F2(bK), F2(ibK), F2(c.T3), F2(c.Dn), F2(c.r4), F2(c.r45), rs, Fs);
#pragma unroll
    for (int m = 0; m < nv; ++m) {
      rhs[m] = rs[m].v.x + rs[m].v.y;
      F[m] = Fs[m].v.x + Fs[m].v.y;
    }
  }
  if constexpr (!RAR) equilibrium_terms<D, T, MULTID>(g0, w0, in, idxl, idxr, bK, ibK, q);
  close_flux<D, T>(g0, q, c, abar_t0, bK, ibK, rhs, F);
}

// face_flux_ps with the inputs in arrays, the inverse centre-to-face distances given.
template <int D, bool MULTID, bool RAR = false>
GKS_FN void face_flux_ps_inv(const float* wl, const float* wr, const float* cl, const float* cr, const float* sl,
                             const float* sr, const float (*tl)[D + 2], const float (*tr)[D + 2], float idxl,
                             float idxr, float tau_t, float dt, const Gas<float>& gas, int abar_t0, float* F,
                             float* tau_out) {
  const FaceArrays<D, float> in{sl, sr, cl, cr, tl, tr};
  face_flux_ps<D, MULTID, RAR>(wl, wr, in, idxl, idxr, tau_t, dt, gas, abar_t0, F, tau_out);
}

// face_flux_ps with the inputs in arrays and the centre-to-face distances.
template <int D, bool MULTID, bool RAR = false>
GKS_FN void face_flux_ps(const float* wl, const float* wr, const float* cl, const float* cr, const float* sl,
                         const float* sr, const float (*tl)[D + 2], const float (*tr)[D + 2], float dxl, float dxr,
                         float tau_t, float dt, const Gas<float>& gas, int abar_t0, float* F, float* tau_out) {
  face_flux_ps_inv<D, MULTID, RAR>(wl, wr, cl, cr, sl, sr, tl, tr, g_rcp(dxl), g_rcp(dxr), tau_t, dt, gas, abar_t0, F,
                                   tau_out);
}

// A first-order face: the sides are the cells' own states cl, cr (no slopes).
template <int D, class T, bool RAR = false>
GKS_FN void face_flux_first_order(const T* cl, const T* cr, T dxl, T dxr, T tau_t, T dt, const Gas<T>& gas, int abar_t0,
                                  T* F, T* tau_out) {
  const FaceArrays<D, T> in{nullptr, nullptr, cl, cr, nullptr, nullptr};
  if constexpr (std::is_same<T, float>::value)
    face_flux_ps<D, false, RAR, true>(cl, cr, in, g_rcp(dxl), g_rcp(dxr), tau_t, dt, gas, abar_t0, F, tau_out);
  else
    face_flux_in<D, T, false, RAR, true>(cl, cr, in, g_rcp(dxl), g_rcp(dxr), tau_t, dt, gas, abar_t0, F, tau_out);
}

}  // namespace gks
