// The interface flux in moment tables: every <u^k (a . psi) psi_m> as sums of products of the normal half-line
// moments with a table of transverse moments.  Host only: its operation count is the fixed unit of work
// that throughput is quoted in (gks_face_op_count), so that figures of different kernels compare; the kernels
// evaluate the same flux in closed form (gks_flux.cuh) with fewer operations.
#pragma once
#include "gks_flux.cuh"

namespace gks {
namespace tables {

// Macroscopic description of one Maxwellian.
template <int D, class T> struct Maxw {
  T rho, ir, U[D], lam, il;  // ir = 1/rho, il = 1/(2 lambda)
  T c, f4;               // |U|^2 + bK il and 4 lambda^2 / bK (used by every slope solve)
};

// (rho, U, lambda) of the Maxwellian carrying the conservative state w (Section 2: E = (u^2 + xi^2)/2,
// so rho E = rho |U|^2 / 2 + bK rho / (4 lambda)).  Two reciprocals: 1/rho, and 1/(2 lambda) =
// (2 rho E - rho |U|^2) / (bK rho) is a product, lambda its reciprocal; ibK = 1/bK.
template <int D, class T>
GKS_FN Maxw<D, T> maxwellian(const T* w, T bK, T ibK) {
  Maxw<D, T> g;
  g.rho = w[0];
  g.ir = g_rcp(w[0]);
  T q = T(0);
#pragma unroll
  for (int i = 0; i < D; ++i) {
    g.U[i] = w[1 + i] * g.ir;
    q += g.U[i] * g.U[i];
  }
  g.il = (T(2) * w[D + 1] - w[0] * q) * g.ir * ibK;
  g.lam = T(0.5) * g_rcp(g.il);
  g.c = q + bK * g.il;
  g.f4 = T(4) * g.lam * g.lam * ibK;
  return g;
}

// Moments of one Maxwellian, split into the normal velocity u and the transverse part.
//
// Every polynomial the flux needs is linear in the transverse basis {1, v_s, Et}, with
// Et = (sum_s v_s^2 + xi^2)/2 (so psi_E = u^2/2 + Et), and has polynomial coefficients in u.  Under
// the Maxwellian u, the v_s and xi are independent, so a moment factors into a moment of u over the
// chosen half line and a transverse moment over the full space.  The transverse moments of products
// of up to three basis functions are tabulated once per Maxwellian.
template <int D> struct Basis {
  static constexpr int NB = D + 1;  // 0: 1, 1..D-1: v_s, D: Et
};

template <int D, class T> struct Trans {
  T m1[D + 1];                     // <beta>
  T m2[D + 1][D + 1];              // <alpha beta>
  T m3[Dims<D>::nt][D + 1][D + 1];  // <v_s alpha beta>
};

// Gaussian moments <x^n>, n = 0..N-1, of mean U and variance il: x^{n+2} = U x^{n+1} + (n+1) il x^n.
template <int N, class T>
GKS_FN void recur(T U, T il, T* m) {
#pragma unroll
  for (int n = 0; n + 2 < N; ++n) m[n + 2] = U * m[n + 1] + T(n + 1) * il * m[n];
}

template <int D, class T>
GKS_FN void transverse(const Maxw<D, T>& g, T K, Trans<D, T>& t) {
  const T X1 = K * g.il;                        // <xi^2>
  const T X2 = K * (K + T(2)) * g.il * g.il;    // <xi^4>
  T V[Dims<D>::nt][6];
#pragma unroll
  for (int s = 0; s < D - 1; ++s) {
    V[s][0] = T(1);
    V[s][1] = g.U[1 + s];
    recur<6>(g.U[1 + s], g.il, V[s]);
  }
  t.m1[0] = T(1);
#pragma unroll
  for (int b = 0; b <= D; ++b) t.m2[0][b] = T(0);
  if (D == 1) {
    // basis {1, Et}, Et = xi^2 / 2
    t.m1[1] = T(0.5) * X1;
    t.m2[0][0] = T(1);
    t.m2[0][1] = t.m2[1][0] = t.m1[1];
    t.m2[1][1] = T(0.25) * X2;
  } else if (D == 2) {
    // basis {1, v, Et}, Et = (v^2 + xi^2)/2
    const T* v = V[0];
    const T e1 = v[2] + X1;                          // <2 Et>
    const T ve = v[3] + v[1] * X1;                   // <v 2 Et>
    const T vve = v[4] + v[2] * X1;                  // <v^2 2 Et>
    const T ee = v[4] + T(2) * v[2] * X1 + X2;       // <(2 Et)^2>
    const T vee = v[5] + T(2) * v[3] * X1 + v[1] * X2;  // <v (2 Et)^2>
    t.m1[1] = v[1];
    t.m1[2] = T(0.5) * e1;
    t.m2[0][0] = T(1);
    t.m2[0][1] = t.m2[1][0] = v[1];
    t.m2[0][2] = t.m2[2][0] = t.m1[2];
    t.m2[1][1] = v[2];
    t.m2[1][2] = t.m2[2][1] = T(0.5) * ve;
    t.m2[2][2] = T(0.25) * ee;
    // <v alpha beta>
    t.m3[0][0][0] = v[1];
    t.m3[0][0][1] = t.m3[0][1][0] = v[2];
    t.m3[0][0][2] = t.m3[0][2][0] = t.m2[1][2];
    t.m3[0][1][1] = v[3];
    t.m3[0][1][2] = t.m3[0][2][1] = T(0.5) * vve;
    t.m3[0][2][2] = T(0.25) * vee;
  } else {
    // basis {1, v, w, Et}, Et = (v^2 + w^2 + xi^2)/2
    const T* v = V[0];
    const T* w = V[Dims<D>::nt - 1];
    const T rv1 = w[2] + X1, rv2 = w[4] + T(2) * w[2] * X1 + X2;  // moments of 2Et - v^2
    const T rw1 = v[2] + X1, rw2 = v[4] + T(2) * v[2] * X1 + X2;  // moments of 2Et - w^2
    const T e1 = v[2] + rv1;
    const T ee = v[4] + T(2) * v[2] * rv1 + rv2;
    t.m1[1] = v[1];
    t.m1[2] = w[1];
    t.m1[3] = T(0.5) * e1;
    t.m2[0][0] = T(1);
#pragma unroll
    for (int b = 1; b <= 3; ++b) t.m2[0][b] = t.m2[b][0] = t.m1[b];
    t.m2[1][1] = v[2];
    t.m2[1][2] = t.m2[2][1] = v[1] * w[1];
    t.m2[2][2] = w[2];
    t.m2[1][3] = t.m2[3][1] = T(0.5) * (v[3] + v[1] * rv1);
    t.m2[2][3] = t.m2[3][2] = T(0.5) * (w[3] + w[1] * rw1);
    t.m2[3][3] = T(0.25) * ee;
    const T vwe = T(0.5) * (v[3] * w[1] + v[1] * w[3] + v[1] * w[1] * X1);  // <v w Et>
    // gamma = v
    t.m3[0][0][0] = v[1];
    t.m3[0][0][1] = t.m3[0][1][0] = v[2];
    t.m3[0][0][2] = t.m3[0][2][0] = t.m2[1][2];
    t.m3[0][0][3] = t.m3[0][3][0] = t.m2[1][3];
    t.m3[0][1][1] = v[3];
    t.m3[0][1][2] = t.m3[0][2][1] = v[2] * w[1];
    t.m3[0][2][2] = v[1] * w[2];
    t.m3[0][1][3] = t.m3[0][3][1] = T(0.5) * (v[4] + v[2] * rv1);
    t.m3[0][2][3] = t.m3[0][3][2] = vwe;
    t.m3[0][3][3] = T(0.25) * (v[5] + T(2) * v[3] * rv1 + v[1] * rv2);
    // gamma = w
    t.m3[1][0][0] = w[1];
    t.m3[1][0][1] = t.m3[1][1][0] = t.m2[1][2];
    t.m3[1][0][2] = t.m3[1][2][0] = w[2];
    t.m3[1][0][3] = t.m3[1][3][0] = t.m2[2][3];
    t.m3[1][1][1] = v[2] * w[1];
    t.m3[1][1][2] = t.m3[1][2][1] = v[1] * w[2];
    t.m3[1][2][2] = w[3];
    t.m3[1][1][3] = t.m3[1][3][1] = vwe;
    t.m3[1][2][3] = t.m3[1][3][2] = T(0.5) * (w[4] + w[2] * rw1);
    t.m3[1][3][3] = T(0.25) * (w[5] + T(2) * w[3] * rw1 + w[1] * rw2);
  }
}

// <beta> for the transverse basis {1, v_s, Et} (the first row of the transverse table).
template <int D, class T>
GKS_FN void trans_mean(const Maxw<D, T>& g, T K, T* m1) {
  T e = K * g.il;  // <xi^2>
#pragma unroll
  for (int s = 0; s < D - 1; ++s) {
    m1[1 + s] = g.U[1 + s];
    e += g.U[1 + s] * g.U[1 + s] + g.il;  // <v_s^2>
  }
  m1[0] = T(1);
  m1[D] = T(0.5) * e;
}

// <u^n>, n = 0..6, over the full line.
template <int D, class T>
GKS_FN void u_full(const Maxw<D, T>& g, T* u) {
  u[0] = T(1);
  u[1] = g.U[0];
  recur<7>(g.U[0], g.il, u);
}

// <u^n> over u > 0 (sgn = +1) or u < 0 (sgn = -1), from the textbook half-line Gaussian integrals
//   <1>_{u>0} = erfc(-sqrt(lam) U)/2,  <u>_{u>0} = U <1>_{u>0} + exp(-lam U^2)/(2 sqrt(pi lam)).
template <int D, class T>
GKS_FN void u_half(const Maxw<D, T>& g, T sgn, T* u) {
  const T rs = g_rsqrt(g.lam);  // 1/sqrt(lambda); sqrt(lambda) = lambda / sqrt(lambda)
  const T z = g.lam * rs * g.U[0];
  u[0] = T(0.5) * g_erfc(-sgn * z);
  u[1] = g.U[0] * u[0] + sgn * T(0.5) * g_exp(-z * z) * T(kInvSqrtPi) * rs;
  recur<7>(g.U[0], g.il, u);
}

// <psi_m> over the region of table u, m1 the transverse means.
template <int D, class T>
GKS_FN void psi_mean(const T* u, const T* m1, T* out) {
  out[0] = u[0];
  out[1] = u[1];
#pragma unroll
  for (int s = 0; s < D - 1; ++s) out[2 + s] = u[0] * m1[1 + s];
  out[D + 1] = T(0.5) * u[2] + u[0] * m1[D];
}

// acc[m] += s * <u^k gamma (a . psi) psi_m>, gamma = 1 (tg = -1) or v_tg.
// With a . psi = A(u) + sum_beta a_beta beta, A(u) = a0 + a1 u + aE u^2 / 2, and
// psi_m = P_m(u) + (transverse part), the moment is a sum of (u moment) x (transverse moment).
template <int D, class T>
GKS_FN void amom(const T* u, const Trans<D, T>& t, int k, int tg, const T* a, T s, T* acc) {
  constexpr int NB = D + 1;
  const T hE = T(0.5) * a[D + 1];
  const T SA0 = a[0] * u[k] + a[1] * u[k + 1] + hE * u[k + 2];
  const T SA1 = a[0] * u[k + 1] + a[1] * u[k + 2] + hE * u[k + 3];
  const T SA2 = a[0] * u[k + 2] + a[1] * u[k + 3] + hE * u[k + 4];
  // transverse factors: <gamma beta> and <gamma beta tau>
  T g1[NB], c2[NB];
#pragma unroll
  for (int b = 0; b < NB; ++b) g1[b] = tg < 0 ? t.m1[b] : t.m2[1 + tg][b];
  T c1 = T(0);
#pragma unroll
  for (int b = 1; b < NB; ++b) c1 += a[b == D ? D + 1 : 1 + b] * g1[b];
#pragma unroll
  for (int tau = 1; tau < NB; ++tau) {
    T q = T(0);
#pragma unroll
    for (int b = 1; b < NB; ++b) q += a[b == D ? D + 1 : 1 + b] * (tg < 0 ? t.m2[b][tau] : t.m3[tg][b][tau]);
    c2[tau] = q;
  }
  acc[0] += s * (SA0 * g1[0] + u[k] * c1);
  acc[1] += s * (SA1 * g1[0] + u[k + 1] * c1);
#pragma unroll
  for (int v = 0; v < D - 1; ++v) acc[2 + v] += s * (SA0 * g1[1 + v] + u[k] * c2[1 + v]);
  acc[D + 1] += s * (T(0.5) * (SA2 * g1[0] + u[k + 2] * c1) + SA0 * g1[D] + u[k] * c2[D]);
}

// The pair <u^k gamma (a . psi) psi_m> and <u^(k+1) gamma (a . psi) psi_m>, which share the u-moments
// of A(u) and the transverse sums: acc_lo += s_lo * first, acc_hi += s_hi * second (k <= 1).
template <int D, class T>
GKS_FN void amom2(const T* u, const Trans<D, T>& t, int k, int tg, const T* a, T s_lo, T* acc_lo, T s_hi,
                  T* acc_hi) {
  constexpr int NB = D + 1;
  const T hE = T(0.5) * a[D + 1];
  T SA[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) SA[j] = a[0] * u[k + j] + a[1] * u[k + j + 1] + hE * u[k + j + 2];
  T g1[NB], c2[NB];
#pragma unroll
  for (int b = 0; b < NB; ++b) g1[b] = tg < 0 ? t.m1[b] : t.m2[1 + tg][b];
  T c1 = T(0);
#pragma unroll
  for (int b = 1; b < NB; ++b) c1 += a[b == D ? D + 1 : 1 + b] * g1[b];
#pragma unroll
  for (int tau = 1; tau < NB; ++tau) {
    T q = T(0);
#pragma unroll
    for (int b = 1; b < NB; ++b) q += a[b == D ? D + 1 : 1 + b] * (tg < 0 ? t.m2[b][tau] : t.m3[tg][b][tau]);
    c2[tau] = q;
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const T s = h ? s_hi : s_lo;
    T* acc = h ? acc_hi : acc_lo;
    const int kk = k + h;
    acc[0] += s * (SA[h] * g1[0] + u[kk] * c1);
    acc[1] += s * (SA[h + 1] * g1[0] + u[kk + 1] * c1);
#pragma unroll
    for (int v = 0; v < D - 1; ++v) acc[2 + v] += s * (SA[h] * g1[1 + v] + u[kk] * c2[1 + v]);
    acc[D + 1] += s * (T(0.5) * (SA[h + 2] * g1[0] + u[kk + 2] * c1) + SA[h] * g1[D] + u[kk] * c2[D]);
  }
}

// Coefficients a of a . psi with <(a . psi) psi> = rhs (already divided by rho): closed-form inverse
// of the Maxwellian moment matrix.
template <int D, class T>
GKS_FN void slope(const Maxw<D, T>& g, T bK, const T* rhs, T* a) {
  T R[D], UR = T(0);
#pragma unroll
  for (int i = 0; i < D; ++i) {
    R[i] = rhs[1 + i] - g.U[i] * rhs[0];
    UR += g.U[i] * R[i];
  }
  const T RE = T(2) * rhs[D + 1] - g.c * rhs[0];
  const T aE = g.f4 * (RE - T(2) * UR);
  const T l2 = T(2) * g.lam;
  T a0 = rhs[0] - T(0.5) * aE * g.c;
#pragma unroll
  for (int i = 0; i < D; ++i) {
    a[1 + i] = l2 * R[i] - g.U[i] * aE;
    a0 -= g.U[i] * a[1 + i];
  }
  a[0] = a0;
  a[D + 1] = aE;
}

template <class T>
GKS_FN void time_coeffs(T dt, T tau, T* Tc, T& r1, T& r4, T& r5) {
  const T x = g_div(dt, tau);
  if (x < T(1)) {
    // series branch (phi_k summed, no cancellation) in the arithmetic type
    T p1, p2, p3, e;
    const T xd = x, dtd = dt, taud = tau;
    phi_series(xd, p1, p2, p3, e);
    const T Dn = dtd * dtd * p2;
    const T T1 = -dtd * dtd * xd * (p2 - T(2) * p3);
    const T T4 = taud * dtd * (e - T(2) * p1);
    const T T5 = -taud * dtd * p1;
    Tc[0] = dtd * xd * p2;
    Tc[1] = T1;
    Tc[2] = dtd * dtd * xd * p3;
    Tc[3] = dtd * p1;
    Tc[4] = T4;
    Tc[5] = T5;
    const T iDn = g_rcp(Dn);
    r1 = T1 * iDn;
    r4 = T4 * iDn;
    r5 = T5 * iDn;
  } else {
    const T e = g_exp(-x);
    const T q = T(1) - e;
    const T tq = tau * q;
    Tc[0] = dt - tq;
    Tc[1] = -tau * dt * (T(1) + e) + T(2) * tau * tq;
    Tc[2] = T(0.5) * dt * dt - tau * dt + tau * tq;
    Tc[3] = tq;
    Tc[4] = tau * dt * e - T(2) * tau * tq;
    Tc[5] = -tau * tq;
    const T y = g_div(tau, dt);
    const T yq = y * q;
    const T inv = g_rcp(T(1) - yq);
    r1 = (T(2) * yq - (T(1) + e)) * inv;
    r4 = (e - T(2) * yq) * inv;
    r5 = -yq * inv;
  }
}

// One face, inputs as gks::face_flux_in (dxl, dxr the centre-to-face distances).
template <int D, class T, bool MULTID, class In>
GKS_FN void face_flux_in(const T* wl, const T* wr, const In& in, T dxl, T dxr, T tau_t, T dt, const Gas<T>& gas,
                         int abar_t0, T* F, T* tau_out) {
  constexpr int nv = D + 2;
  const T bK = gas.bK, K = gas.K, ibK = gas.ibK;
  const Maxw<D, T> gl = maxwellian<D, T>(wl, bK, ibK);
  const Maxw<D, T> gr = maxwellian<D, T>(wr, bK, ibK);

  // Eq. intermediatestate: w0 = rho_l <psi>_{l,u>0} + rho_r <psi>_{r,u<0}
  T w0[nv];
  T lP[7], rN[7];
  u_half<D, T>(gl, T(1), lP);
  u_half<D, T>(gr, T(-1), rN);
  {
    T a[nv], b[nv], ml[D + 1], mr[D + 1];
    trans_mean<D, T>(gl, K, ml);
    trans_mean<D, T>(gr, K, mr);
    psi_mean<D, T>(lP, ml, a);
    psi_mean<D, T>(rN, mr, b);
#pragma unroll
    for (int m = 0; m < nv; ++m) w0[m] = gl.rho * a[m] + gr.rho * b[m];
  }
  const Maxw<D, T> g0 = maxwellian<D, T>(w0, bK, ibK);

  // Eqs. relaxation time and taua: tau = mu/p0 + tau_t + C_a |p_r - p_l| / (p_r + p_l) dt
  const T p0 = g0.rho * g0.il, pl = gl.rho * gl.il, pr = gr.rho * gr.il;
  const T tau = g_div(gas.mu, p0) + tau_t + g_div(gas.C_a * g_abs(pr - pl), pr + pl) * dt;
  *tau_out = tau;
  T Tc[6], r1, r4, r5;
  time_coeffs<T>(dt, tau, Tc, r1, r4, r5);
  if (abar_t0) {
    r1 = T(-1);
    r4 = r5 = T(0);
  }
  const T i0 = g0.ir;

  // Abar right-hand side (per unit rho0) and flux, accumulated region by region
  T rhs[nv];
#pragma unroll
  for (int m = 0; m < nv; ++m) {
    rhs[m] = T(0);
    F[m] = T(0);
  }

  // The two sides of the initial state, one loop body (sd = 0: left Maxwellian on u > 0, sd = 1:
  // right Maxwellian on u < 0): Eq. initialf0 slopes a (normal), b (tangential), A; their parts of
  // the Abar right-hand side and of the flux.
#pragma unroll 1
  for (int sd = 0; sd < 2; ++sd) {
    const Maxw<D, T> g = sd ? gr : gl;
    Trans<D, T> ts;
    transverse<D, T>(g, K, ts);
    T half[7], a[nv], b[Dims<D>::nt][nv], A[nv], r[nv];
#pragma unroll
    for (int n = 0; n < 7; ++n) half[n] = sd ? rN[n] : lP[n];
    const T ir = g.ir;
#pragma unroll
    for (int m = 0; m < nv; ++m) r[m] = in.s(sd, m) * ir;
    slope<D, T>(g, bK, r, a);
    if (MULTID) {
#pragma unroll
      for (int q = 0; q < D - 1; ++q) {
#pragma unroll
        for (int m = 0; m < nv; ++m) r[m] = in.t(sd, q, m) * ir;
        slope<D, T>(g, bK, r, b[q]);
      }
    }
    // A from the compatibility condition at t = 0: <(a u + b v + A) psi> = 0 (full line)
    {
      T uf[7];
      u_full<D, T>(g, uf);
#pragma unroll
      for (int m = 0; m < nv; ++m) r[m] = T(0);
      amom<D, T>(uf, ts, 1, -1, a, T(-1), r);
      if (MULTID) {
#pragma unroll
        for (int q = 0; q < D - 1; ++q) amom<D, T>(uf, ts, 0, q, b[q], T(-1), r);
      }
      slope<D, T>(g, bK, r, A);
    }
    // Abar rhs: r4 rho/rho0 <(a u + b v) psi> + r5 rho/rho0 <A psi> over the half line, and the
    // flux rho [T3 <u psi> + T5 <u A psi> + T4 (<u^2 a psi> + <u v b psi>)]: each polynomial once,
    // at u^k for the rhs and u^(k+1) for the flux
    const T s4 = r4 * g.rho * i0, s5 = r5 * g.rho * i0, s4f = Tc[4] * g.rho;
    amom2<D, T>(half, ts, 1, -1, a, s4, rhs, s4f, F);
    amom2<D, T>(half, ts, 0, -1, A, s5, rhs, Tc[5] * g.rho, F);
    {
      T m[nv];
      psi_mean<D, T>(half + 1, ts.m1, m);  // <u psi> over the half line
      const T s3 = Tc[3] * g.rho;
#pragma unroll
      for (int q = 0; q < nv; ++q) F[q] += s3 * m[q];
    }
    if (MULTID) {
#pragma unroll
      for (int q = 0; q < D - 1; ++q) amom2<D, T>(half, ts, 0, q, b[q], s4, rhs, s4f, F);
    }
  }

  // equilibrium g0: Eq. eqlgform slopes from W_j -> w0 -> W_{j+1} (and the mean tangential slope)
  Trans<D, T> tr0;
  transverse<D, T>(g0, K, tr0);
  T oF[7], oP[7];
  u_full<D, T>(g0, oF);
  u_half<D, T>(g0, T(1), oP);
  {
    const T fl = g_div(i0, dxl), fr = g_div(i0, dxr);
    const T s1f = Tc[1] * g0.rho;
#pragma unroll 1
    for (int sd = 0; sd < 2; ++sd) {
      // sd = 0: abar_l on u > 0; sd = 1: abar_r on u < 0 (table = full line minus u > 0)
      T r[nv], ab[nv], half[7];
#pragma unroll
      for (int m = 0; m < nv; ++m) r[m] = sd ? (in.c(1, m) - w0[m]) * fr : (w0[m] - in.c(0, m)) * fl;
#pragma unroll
      for (int n = 0; n < 7; ++n) half[n] = sd ? oF[n] - oP[n] : oP[n];
      slope<D, T>(g0, bK, r, ab);
      amom2<D, T>(half, tr0, 1, -1, ab, r1, rhs, s1f, F);
    }
    if (MULTID) {
      T r[nv], ab[nv];
#pragma unroll
      for (int q = 0; q < D - 1; ++q) {
#pragma unroll
        for (int m = 0; m < nv; ++m) r[m] = T(0.5) * (in.t(0, q, m) + in.t(1, q, m)) * i0;
        slope<D, T>(g0, bK, r, ab);
        amom2<D, T>(oF, tr0, 0, q, ab, r1, rhs, s1f, F);
      }
    }
  }
  // Abar from the compatibility condition integrated over [0, dt]; flux rho0 <u (T0 + T2 Abar) psi>
  {
    T Ab[nv];
    slope<D, T>(g0, bK, rhs, Ab);
#pragma unroll
    for (int m = 0; m < nv; ++m) Ab[m] *= Tc[2];
    Ab[0] += Tc[0];
    amom<D, T>(oF, tr0, 1, -1, Ab, g0.rho, F);
  }
}

}  // namespace tables
}  // namespace gks
