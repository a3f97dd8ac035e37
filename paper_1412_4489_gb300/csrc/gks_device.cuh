// Device arithmetic of the compact third-order gas-kinetic scheme
// (Pan & Xu, arXiv:1412.4489), templated on the compute type R (double or float).
//
//   Section 2.1  Maxwellian moments: full space and the half spaces u > 0, u < 0
//   Section 2.2  closed-form solve of <a> = r, the nine coefficient systems,
//                time weights of Eq. dis1 / Eq. dis2 integrated over [0, dt]
//                and at t = dt, assembly of the flux and of Eq. point
//   Section 3.2  compact reconstruction of one cell
//   Section 3.3  equilibrium polynomial across a face
//   Section 4    collision time
#pragma once
#include <cuda_runtime.h>
#include <math.h>

#include "gks_half_normal.cuh"

#ifndef GKS_FN
#define GKS_FN __host__ __device__ __forceinline__
#endif

namespace gks {

template <class R> struct Prec;
// series_below: x = dt/tau below which the time weights are summed from series;
// series_terms: the sums stop before x^series_terms / series_terms!, at which the largest
// relative truncation error over x < series_below is below the type's rounding (FP64: 17
// terms reach it, FP32: 18);
// exp_zero: exp(-x) is exactly 0 from here on, and not evaluated (FP32: always evaluated, a
// branch costs more than its two instructions);
// fp64: arithmetic chosen for the FP64 pipe (quotients from one reciprocal, half_normal's table);
// tie: relative width within which two cross-derivative candidates count as equal.
// FP64: far above its rounding noise, far below any real difference.  FP32: ~16
// ulps, just above the rounding noise of the candidates; a wider band makes FP32
// keep the first stencil where FP64 picks a smaller one of opposite sign, which
// measured worse against the FP64 results on discontinuous data.
template <> struct Prec<double> {
  static constexpr bool fp64 = true;
  static constexpr double series_below = 0.5;
  static constexpr int series_terms = 18;
  static constexpr double exp_zero = 746.0;
  static constexpr double tie = 1e-8;
};
template <> struct Prec<float> {
  static constexpr bool fp64 = false;
  static constexpr float series_below = 2.0f;
  static constexpr int series_terms = 18;
  static constexpr float exp_zero = INFINITY;
  static constexpr float tie = 1e-6f;
};

__device__ __forceinline__ double d_exp(double x) { return exp(x); }
__device__ __forceinline__ float d_exp(float x) { return __expf(x); }
__device__ __forceinline__ double d_erfc(double x) { return erfc(x); }
__device__ __forceinline__ float d_erfc(float x) { return erfcf(x); }
__device__ __forceinline__ double d_rsqrt(double x) { return rsqrt(x); }
__device__ __forceinline__ float d_rsqrt(float x) { return rsqrtf(x); }
// quotient of runtime values: IEEE in FP64; in FP32 the fast division (within
// 2 ulps for divisors below 2^126), far inside the FP32 path's error budget
__device__ __forceinline__ double d_div(double a, double b) { return a / b; }
__device__ __forceinline__ float d_div(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double d_rcp(double a) { return 1.0 / a; }
__device__ __forceinline__ float d_rcp(float a) { return __fdividef(1.0f, a); }

// 2^-511 <= |a| < 2^512, by the exponent bits: squares and reciprocals are normal numbers
__device__ __forceinline__ bool mid_range(double a) {
  return (unsigned)(__double2hiint(a) & 0x7fffffff) - 0x20000000u < 0x3ff00000u;
}

template <class R> GKS_FN R sq(R a) { return a * a; }

// ---------------------------------------------------------------------------
// Section 2.1: moments of g = rho (lam/pi)^((K+2)/2) exp(-lam((u-U)^2+(v-V)^2+xi^2)),
// normalised by rho.  NU u-moments, NV v-moments.
// ---------------------------------------------------------------------------
template <class R, int NU, int NV>
struct Moments {
  R u[NU];
  R v[NV];
  R xi2;
};

// <u^0> and <u^1> over u > 0 (kind +1) or u < 0 (kind -1); l2 = 2 lam
template <class R>
GKS_FN void half_start(R U, R l2, int kind, R& h, R& g) {
  const R lam = R(0.5) * l2;
  const R rs = d_rsqrt(lam);
  const R s = lam * rs;  // sqrt(lam)
  // b: boundary term of the integration by parts at u = 0, 1/(2 sqrt(pi lam)) exp(-lam U^2)
  if constexpr (Prec<R>::fp64) {
    const R a = R(kind) * s * U;
    R t, e;
    half_normal(fabs(a), t, e);
    h = a > R(0) ? R(1) - t : t;
    const R b = e * (R(0.28209479177387814) * rs);
    g = U * h + R(kind) * b;
  } else {
    h = R(0.5) * d_erfc(-R(kind) * s * U);
    const R b = d_exp(-lam * U * U) * R(0.28209479177387814) * rs;
    g = U * h + R(kind) * b;
  }
}

// moments over u > 0 (kind +1) or u < 0 (kind -1); var = 1/(2 lam) = p/rho, formed once per
// Maxwellian by the caller
template <class R, int NU, int NV>
GKS_FN void moments(R U, R V, R lam, R var, R K, int kind, Moments<R, NU, NV>& m) {
  half_start(U, R(2) * lam, kind, m.u[0], m.u[1]);
#pragma unroll
  for (int n = 2; n < NU; ++n) m.u[n] = U * m.u[n - 1] + (n == 2 ? var : R(n - 1) * var) * m.u[n - 2];
  m.v[0] = R(1);
  m.v[1] = V;
  m.v[2] = V * V + var;
#pragma unroll
  for (int n = 3; n < NV; ++n) m.v[n] = V * m.v[n - 1] + R(n - 1) * var * m.v[n - 2];
  m.xi2 = K * var;
}

// <u^A v^B psi>, psi = (1, u, v, (u^2+v^2+xi^2)/2)
template <int A, int B, class R, int NU, int NV>
GKS_FN void psi_mom(const Moments<R, NU, NV>& m, R o[4]) {
  static_assert(A + 2 < NU && B + 2 < NV, "moment table too short");
  const R ab = m.u[A] * m.v[B];
  o[0] = ab;
  o[1] = m.u[A + 1] * m.v[B];
  o[2] = m.u[A] * m.v[B + 1];
  o[3] = R(0.5) * (m.u[A + 2] * m.v[B] + m.u[A] * m.v[B + 2] + ab * m.xi2);
}

// ---------------------------------------------------------------------------
// Time weights.  With x = dt/tau and e = exp(-x): the integrals over [0, dt] of C_1..C_6,
// e^(-t/tau), t e^(-t/tau) and t^2 e^(-t/tau) for the flux, and e and 1 - e for the values
// at t = dt (Eq. point).  Several are differences of nearly equal terms when x is small;
// there they come from three sums of their Taylor series in x.
// ---------------------------------------------------------------------------
template <class R>
struct TimeW {
  R I1, I2, I3, I4, I5, I6;  // integrals of C_1..C_6
  R i7, i9, i10;             // integrals of e^(-t/tau) (C_7), t e^(-t/tau) (-C_8), t^2 e^(-t/tau)
  R e, om, te;               // exp(-x), 1 - exp(-x), tau exp(-x)
};

// Coefficients of x^k, k = n - 3, in the sums over n >= 3 of t_n = (-x)^n / n!, of (n-2) t_n and
// of (n-1)(n-2) t_n, each divided by x^3 (which: 0, 1, 2)
GKS_FN constexpr double series_coef(int which, int k) {
  const int n = k + 3;
  double f = (n & 1) ? -1.0 : 1.0;
  for (int j = 2; j <= n; ++j) f /= j;
  return which == 0 ? f : (which == 1 ? (n - 2) * f : (double)((n - 1) * (n - 2)) * f);
}

template <int W, int K, class R>
GKS_FN R series_sum(R x) {
  if constexpr (K + 4 >= Prec<R>::series_terms) {
    constexpr double c = series_coef(W, K);
    return R(c);
  } else {
    constexpr double c = series_coef(W, K);
    return R(c) + x * series_sum<W, K + 1>(x);
  }
}

template <class R>
GKS_FN void time_weights(R T, R tau, TimeW<R>& w) {
  const R x = tau > R(0) ? T * d_rcp(tau) : R(INFINITY);
  const R t2 = tau * tau, T2h = R(0.5) * T * T;
  if (x < Prec<R>::series_below) {
    // with g = sum t_n, a = sum (n-2) t_n, b = sum (n-1)(n-2) t_n over n >= 3:
    //   x - 1 + e = x^2/2 + g;  1 - (1+x) e = x^2/2 + a + g;  2 - 2e - x - x e = a;
    //   x^2/2 - x + 1 - e = -g;  2 - (x^2 + 2x + 2) e = -b
    const R xx = R(0.5) * x * x, x3 = R(2) * xx * x;
    const R g = x3 * series_sum<0, 0>(x), a = x3 * series_sum<1, 0>(x), b = x3 * series_sum<2, 0>(x);
    const R f1 = xx + g;
    w.om = x - f1;
    w.e = R(1) - w.om;
    w.I1 = tau * f1;
    w.I2 = t2 * a;
    w.I3 = -t2 * g;
    w.i9 = t2 * (f1 + a);
    w.i10 = -(t2 * tau) * b;
    w.i7 = tau * w.om;
  } else {
    // e is exactly 0 for x beyond the type's range: FP64 skips the exponential there (smooth
    // Euler flow, where tau is a tiny fraction of dt)
    w.e = x < Prec<R>::exp_zero ? d_exp(-x) : R(0);
    w.om = R(1) - w.e;
    w.i7 = tau * w.om;
    w.I1 = T - w.i7;
    w.I2 = R(2) * tau * w.i7 - tau * T * (R(1) + w.e);
    w.I3 = T2h - tau * T + tau * w.i7;
    w.i9 = t2 - tau * (tau + T) * w.e;
    w.i10 = tau * (R(2) * t2 - R(2) * (T2h + T * tau + t2) * w.e);
  }
  w.te = tau * w.e;
  w.I4 = -(w.i10 + R(2) * tau * w.i9);
  w.I5 = R(2) * T2h * (R(1.0 / 3.0) * T - tau);
  w.I6 = -tau * (T2h + w.i9);
}

// ---------------------------------------------------------------------------
// Everything below works in a Maxwellian's own frame.  With c = u - U, d = v - V and
// psi' = (1, c, d, (c^2 + d^2 + xi^2) / 2), a 4-vector e of "central" conservative components is
// <psi' X> of a coefficient X expanded in psi' (the density, the momenta and the energy about
// (U, V)): the coefficient itself is never needed over the whole velocity space, since every moment
// of X is a multiple of e's components.  central() takes a derivative of the conservative variables
// there, lab() takes moments back.
// ---------------------------------------------------------------------------
template <class R>
GKS_FN void central(R U, R V, R hq, const R d[4], R e[4]) {  // hq = (U^2 + V^2) / 2
  e[0] = d[0];
  e[1] = d[1] - U * d[0];
  e[2] = d[2] - V * d[0];
  e[3] = d[3] - U * e[1] - V * e[2] - hq * d[0];
}

template <class R>
GKS_FN void lab(R U, R V, R hq, const R e[4], R o[4]) {
  o[0] = e[0];
  o[1] = e[1] + U * e[0];
  o[2] = e[2] + V * e[0];
  o[3] = e[3] + U * e[1] + V * e[2] + hq * e[0];
}

// The time coefficient T of <(X u + Y v + T) psi> = 0 (system after Eq. dis3), all in central
// components: <c psi' X> = (X1, p', 0, kc X1) and <d psi' Y> = (Y2, 0, p', kc Y2) with
// p' = (2/N) X3 (Y3) and kc = (N + 2) / (4 lam).
template <class R>
GKS_FN void time_coef(R U, R V, R i2N, R kc, const R X[4], const R Y[4], R T[4]) {
  T[0] = -(U * X[0] + V * Y[0] + X[1] + Y[2]);
  T[1] = -(U * X[1] + V * Y[1] + i2N * X[3]);
  T[2] = -(U * X[2] + V * Y[2] + i2N * Y[3]);
  T[3] = -(U * X[3] + V * Y[3] + kc * (X[1] + Y[2]));
}

// Coefficient of the Maxwellian (scaled by rho s, s = 1 / (2 lam)) with central components e, in the basis
// (1, u, d, u^2/2 + eta), eta = (d^2 + xi^2)/2 less its mean: what half-space moments in u need.
// c5 = 4 lam / N, hs = (U^2 + s) / 2.
template <class R>
GKS_FN void half_coef(R U, R s, R c5, R hs, const R e[4], R X[4]) {
  X[3] = c5 * e[3] - e[0];
  X[1] = e[1] - U * X[3];
  X[0] = s * e[0] - U * X[1] - hs * X[3];
  X[2] = e[2];
}

// A polynomial P(u, d, xi) of the half-space distribution averaged over d and xi: its mean q(u), and
// its means weighted by d / <d^2> and by eta, r(u) and t(u).  The tangential and internal velocities run over
// their whole range, so d's odd powers vanish and only these three remain of the full set of
// monomials u^a d^b xi^2c.
template <class R>
struct HalfPoly {
  R q[5], r[4], t[3];
};

// P = W + B1 + Bu u + Bd d + wq (xx u^2 + 2 xy u d + yy d^2), each letter a coefficient vector
// of half_coef's basis; s = <d^2> = 1/(2 lam), n1h = (N - 1)/2.  <eta^2> = n1h s^2,
// <d^2 eta> = s^2, <d^2 eta^2> = (n1h + 2) s^3.
template <class R>
GKS_FN void half_poly(R W, const R B1[4], const R Bu[4], const R Bd[4], R wq, const R xx[4], const R xy[4],
                      const R yy[4], R s, R n1h, HalfPoly<R>& P) {
  const R w2 = R(2) * wq, s2 = s * s;
  const R D0 = Bd[2] + wq * yy[0], D1 = w2 * xy[2] + wq * yy[1];
  const R y3 = wq * yy[3], x3 = wq * xx[3], sy3 = s * y3;
  P.q[0] = (W + B1[0]) + s * (D0 + sy3);
  P.q[1] = (B1[1] + Bu[0]) + s * D1;
  P.q[2] = R(0.5) * (B1[3] + sy3) + (Bu[1] + wq * xx[0]);
  P.q[3] = R(0.5) * Bu[3] + wq * xx[1];
  P.q[4] = R(0.5) * x3;
  P.r[0] = (B1[2] + Bd[0]) + s * (Bd[3] + R(3) * wq * yy[2]);
  P.r[1] = (Bu[2] + Bd[1]) + w2 * (xy[0] + s * xy[3]);
  P.r[2] = R(0.5) * Bd[3] + (wq * xx[2] + w2 * xy[1]);
  P.r[3] = wq * xy[3];
  P.t[0] = s2 * (n1h * B1[3] + D0 + (n1h + R(2)) * sy3);
  P.t[1] = s2 * (n1h * Bu[3] + D1);
  P.t[2] = s2 * (n1h * x3 + R(0.5) * y3);
}

// the same without the terms of second order (W = wq = 0)
template <class R>
GKS_FN void half_poly_linear(const R B1[4], const R Bu[4], const R Bd[4], R s, R n1h, HalfPoly<R>& P) {
  const R s2 = s * s;
  P.q[0] = B1[0] + s * Bd[2];
  P.q[1] = B1[1] + Bu[0];
  P.q[2] = R(0.5) * B1[3] + Bu[1];
  P.q[3] = R(0.5) * Bu[3];
  P.r[0] = (B1[2] + Bd[0]) + s * Bd[3];
  P.r[1] = Bu[2] + Bd[1];
  P.r[2] = R(0.5) * Bd[3];
  P.t[0] = s2 * (n1h * B1[3] + Bd[2]);
  P.t[1] = s2 * n1h * Bu[3];
}

// out += <u^SU P psi> over the half space, m[n] = <u^n>; DEG: the degree of q (4, or 3 when linear)
template <int SU, int DEG, class R>
GKS_FN void half_moments(const HalfPoly<R>& P, const R m[8], R V, R s, R n1h, R out[4]) {
  R o0 = P.q[0] * m[SU], o1 = P.q[0] * m[SU + 1], o3 = P.q[0] * m[SU + 2];
#pragma unroll
  for (int n = 1; n <= DEG; ++n) {
    o0 = o0 + P.q[n] * m[SU + n];
    o1 = o1 + P.q[n] * m[SU + n + 1];
    o3 = o3 + P.q[n] * m[SU + n + 2];
  }
  R o2 = P.r[0] * m[SU], t = P.t[0] * m[SU];
#pragma unroll
  for (int n = 1; n < DEG; ++n) {
    o2 = o2 + P.r[n] * m[SU + n];
    if (n < DEG - 1) t = t + P.t[n] * m[SU + n];
  }
  o2 = s * o2;
  out[0] += o0;
  out[1] += o1;
  out[2] += o2 + V * o0;
  out[3] += (R(0.5) * o3 + t) + V * o2 + (n1h * s + R(0.5) * V * V) * o0;
}

// ---------------------------------------------------------------------------
// Face states in the face frame: value and (dn, dt, dnn, dnt, dtt)
// ---------------------------------------------------------------------------
template <class R>
struct FaceState {
  R w[6][4];
};

template <class R>
GKS_FN void prim(const R w[4], R gm1, R& rho, R& ir, R& U, R& V, R& p) {
  rho = w[0];
  ir = d_div(R(1), rho);
  U = w[1] * ir;
  V = w[2] * ir;
  p = gm1 * (w[3] - R(0.5) * (w[1] * U + w[2] * V));
}

// the same with 2 lam = rho / p and 1 / (2 lam).  FP64: both quotients from one reciprocal (a
// reciprocal takes 5.4 FP64 instructions, a quotient 8.6), of rho^2 p; where that or rho is not well inside FP64's
// range, from quotients of their own.  (Inside it every product here is a normal number.)  FP32: a
// reciprocal is one instruction, and rho^2 p would leave the range often.
template <class R>
GKS_FN void prim_lam(const R w[4], R gm1, R& rho, R& U, R& V, R& p, R& l2, R& var) {
  R ir;
  if constexpr (Prec<R>::fp64) {
    rho = w[0];
    const R rp = gm1 * (rho * w[3] - R(0.5) * (w[1] * w[1] + w[2] * w[2]));  // rho p
    const R q = rho * rp;
    if (mid_range(q) && mid_range(rho)) {
      const R t = d_rcp(q);
      ir = t * rp;
      U = w[1] * ir;
      V = w[2] * ir;
      p = rp * ir;
      l2 = rho * rho * (rho * t);
      var = p * ir;
      return;
    }
  }
  prim(w, gm1, rho, ir, U, V, p);
  l2 = d_div(rho, p);
  var = p * ir;
}

struct FaceParams {
  double gamma, mu, Pr, tau_eps, tau_C;
  double dn, dtan;  // cell size normal to and along the face
};

// Per-launch constants of the face routine in the compute type
template <class R>
struct FaceConst {
  R gamma, gm1, K, N, iN, i2N, dn, dtan, y2, mu, pr_fix, tau_eps, tau_C;
  R n1h, n2h, n4h, nh;          // (N - 1)/2, (N + 2)/2, (N + 4)/2, N/2
  R dn2_12, dt2_24;             // dn^2 / 12, dtan^2 / 24 (face values of the cell polynomial)
  R i4n, i4t, i8n2, i2nt, i2t2;  // 1/(4 dn), 1/(4 dt), 1/(8 dn^2), 1/(2 dn dt), 1/(2 dt^2)
  bool ns, prandtl;
};

template <class R>
GKS_FN FaceConst<R> face_const(const FaceParams& P) {
  FaceConst<R> c;
  c.gamma = R(P.gamma);
  c.gm1 = R(P.gamma - 1.0);
  // N = K + 2 degrees of freedom, K = (4 - 2 gamma) / (gamma - 1) internal ones (Section 2.1)
  const double N = 2.0 / (P.gamma - 1.0);
  c.K = R((4.0 - 2.0 * P.gamma) / (P.gamma - 1.0));
  c.N = R(N);
  c.iN = R(0.5 * (P.gamma - 1.0));
  c.i2N = R(P.gamma - 1.0);  // 2 / N
  c.nh = R(0.5 * N);
  c.n1h = R(0.5 * (N - 1.0));
  c.n2h = R(0.5 * (N + 2.0));
  c.n4h = R(0.5 * (N + 4.0));
  c.dn = R(P.dn);
  c.dtan = R(P.dtan);
  c.y2 = R(P.dtan * P.dtan / 12.0);
  c.dn2_12 = R(P.dn * P.dn / 12.0);
  c.dt2_24 = R(P.dtan * P.dtan / 24.0);
  c.i4n = R(1.0 / (4.0 * P.dn));
  c.i4t = R(1.0 / (4.0 * P.dtan));
  c.i8n2 = R(1.0 / (8.0 * P.dn * P.dn));
  c.i2nt = R(1.0 / (2.0 * P.dn * P.dtan));
  c.i2t2 = R(1.0 / (2.0 * P.dtan * P.dtan));
  c.mu = R(P.mu);
  c.pr_fix = R(1.0 / P.Pr - 1.0);
  c.tau_eps = R(P.tau_eps);
  c.tau_C = R(P.tau_C);
  c.ns = P.mu > 0.0;
  c.prandtl = P.Pr != 1.0;
  return c;
}

// A face source over the two sides and the six averages of one face, for
// callers that hold them in arrays (the host operation count).
template <class R>
struct ArrayFaceSource {
  const FaceState<R>* s[2];
  const R (*a)[3][4];
  GKS_FN void side(int k, FaceState<R>& out) const { out = *s[k]; }
  GKS_FN void avg(R out[2][3][4]) const {
    for (int m = 0; m < 2; ++m)
      for (int n = 0; n < 3; ++n)
        for (int v = 0; v < 4; ++v) out[m][n][v] = a[m][n][v];
  }
};

// Wall images G(n, t) = Phi(P(-n, t)) of the inside face state (face frame).
// kind 2: slip wall (normal momentum negated).  kind 3: isothermal no-slip with
// tangential wall velocity uwt and wall temperature Tw: rho' = rho,
// m' = 2 rho u_w - m, rho E' = 2 rho |u_w|^2 - 2 u_w.m + |m|^2/rho + 2 rho Tw/(gamma-1) - rho E.
// kind 4: adiabatic no-slip: rho' = rho, m' = 2 rho u_w - m, T' = T (a linear map).
template <class R>
GKS_FN void wall_image(int kind, R gamma, R uwt, R Tw, const FaceState<R>& in, FaceState<R>& out) {
  if (kind == 2) {
#pragma unroll
    for (int d = 0; d < 6; ++d) {
      const R s = (d == 1 || d == 4) ? R(-1) : R(1);  // odd derivatives in n flip
      out.w[d][0] = s * in.w[d][0];
      out.w[d][1] = -s * in.w[d][1];
      out.w[d][2] = s * in.w[d][2];
      out.w[d][3] = s * in.w[d][3];
    }
    return;
  }
  if (kind == 4) {
    // adiabatic no-slip: the linear map rho' = rho, m_n' = -m_n, m_t' = 2 u_w rho - m_t,
    // rho E' = rho E + 2 u_w^2 rho - 2 u_w m_t applied to the value and every derivative
#pragma unroll
    for (int d = 0; d < 6; ++d) {
      const R s = (d == 1 || d == 4) ? R(-1) : R(1);  // odd derivatives in n flip
      const R r = in.w[d][0], mn = in.w[d][1], mt = in.w[d][2], e = in.w[d][3];
      out.w[d][0] = s * r;
      out.w[d][1] = -s * mn;
      out.w[d][2] = s * (R(2) * uwt * r - mt);
      out.w[d][3] = s * (e + R(2) * uwt * uwt * r - R(2) * uwt * mt);
    }
    return;
  }
  const R rho = in.w[0][0], mn = in.w[0][1], mt = in.w[0][2];
  const R ir = d_div(R(1), rho);
  const R m2 = mn * mn + mt * mt;
  const R cT = d_div(R(2) * Tw, gamma - R(1));
  // value
  out.w[0][0] = rho;
  out.w[0][1] = -mn;
  out.w[0][2] = R(2) * rho * uwt - mt;
  out.w[0][3] = R(2) * rho * uwt * uwt - R(2) * uwt * mt + m2 * ir + rho * cT - in.w[0][3];
  // Jacobian rows applied to a derivative vector a
  auto lin = [&](const R a[4], R o[4]) {
    o[0] = a[0];
    o[1] = -a[1];
    o[2] = R(2) * uwt * a[0] - a[2];
    o[3] = (R(2) * uwt * uwt - m2 * ir * ir + cT) * a[0] + R(2) * mn * ir * a[1] +
           (R(2) * mt * ir - R(2) * uwt) * a[2] - a[3];
  };
  // second derivative of |m|^2/rho along a, b
  auto hess = [&](const R a[4], const R b[4]) {
    const R ma = mn * a[1] + mt * a[2], mb = mn * b[1] + mt * b[2];
    return R(2) * m2 * ir * ir * ir * a[0] * b[0] - R(2) * ir * ir * (ma * b[0] + mb * a[0]) +
           R(2) * ir * (a[1] * b[1] + a[2] * b[2]);
  };
  R o[4];
  lin(in.w[1], o);
#pragma unroll
  for (int k = 0; k < 4; ++k) out.w[1][k] = -o[k];
  lin(in.w[2], o);
#pragma unroll
  for (int k = 0; k < 4; ++k) out.w[2][k] = o[k];
  lin(in.w[3], o);
#pragma unroll
  for (int k = 0; k < 4; ++k) out.w[3][k] = o[k];
  out.w[3][3] += hess(in.w[1], in.w[1]);
  lin(in.w[4], o);
#pragma unroll
  for (int k = 0; k < 4; ++k) out.w[4][k] = -o[k];
  out.w[4][3] -= hess(in.w[1], in.w[2]);
  lin(in.w[5], o);
#pragma unroll
  for (int k = 0; k < 4; ++k) out.w[5][k] = o[k];
  out.w[5][3] += hess(in.w[2], in.w[2]);
}

// One side of the face: its value as a Maxwellian (s = 1 / (2 lam) = p / rho, l2 = 2 lam) and the
// half-space <u^0>, <u^1>
template <class R>
struct SideData {
  R rho, U, V, s, l2, p, h, g;
};

// the side's Maxwellian from its value w (side 0: u > 0, side 1: u < 0) and its share of
// Eq. compatibility2, U0 += rho <psi>
template <class R>
GKS_FN void side_start(const FaceConst<R>& C, const R w[4], int side, SideData<R>& d, R U0[4]) {
  prim_lam(w, C.gm1, d.rho, d.U, d.V, d.p, d.l2, d.s);
  half_start(d.U, d.l2, side == 0 ? +1 : -1, d.h, d.g);
  const R m2 = d.U * d.g + d.s * d.h;
  U0[0] += d.rho * d.h;
  U0[1] += d.rho * d.g;
  U0[2] += d.rho * (d.V * d.h);
  U0[3] += d.rho * (R(0.5) * m2 + (R(0.5) * d.V * d.V + C.n1h * d.s) * d.h);
}

// Section 4: collision time, from the pressures of the two sides and of g0
template <class R>
GKS_FN R collision_time(const FaceConst<R>& C, bool ns, R pl, R pr, R p0, R dt) {
  const R jump = fabs((pl - pr) * d_rcp(pl + pr)) * dt;
  return ns ? C.mu * d_rcp(p0) + jump : C.tau_eps * dt + C.tau_C * jump;
}

// Section 3.3: the equilibrium polynomial's derivatives (n, t, nn, nt, tt) from the six averages; of the
// nn one without U0's share and factor
template <class R>
GKS_FN void equilibrium_derivatives(const FaceConst<R>& C, const R avg[2][3][4], R d[5][4]) {
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const R um = avg[0][0][k], uc = avg[0][1][k], up = avg[0][2][k];
    const R wm = avg[1][0][k], wc = avg[1][1][k], wp = avg[1][2][k];
    const R Sr = wp + wm, Sl = up + um, Dr = wp - wm, Dl = up - um, cc = wc + uc;
    d[0][k] = ((Sr - Sl) + R(2) * (wc - uc)) * C.i4n;  // b2
    d[1][k] = (Dr + Dl) * C.i4t;                       // b3
    d[2][k] = R(26) * cc - (Sr + Sl);
    d[3][k] = (Dr - Dl) * C.i2nt;                      // b6
    d[4][k] = ((Sr + Sl) - R(2) * cc) * C.i2t2;        // b5
  }
}

// Equilibrium part, Eq. dis1, with g0 and the polynomial of Section 3.3.  All moments of g0 run over the
// whole velocity space: in its frame they are closed forms in the central components of the
// derivatives.  The compatibility conditions turn the moments of a1 u + a2 v into those of A,
// and so on, so that the point value is U0 and its time derivatives.  (r0, u0, v0, var0): g0's
// density, velocity and 1 / (2 lam).
template <class R>
GKS_FN void equilibrium_part(const FaceConst<R>& C, R d[5][4], const R U0[4], R r0, R u0, R v0, R var0,
                             const TimeW<R>& w, R dt, R Fl[4], R P0[4], R P1[4], R Mn[4]) {
  const R U = u0, V = v0, s = var0, hq = R(0.5) * (u0 * u0 + v0 * v0), pN = C.i2N, kc = C.n2h * var0;
  R x[4], y[4], xx[4], xy[4], yy[4];
  {
#pragma unroll
    for (int k = 0; k < 4; ++k) d[2][k] = (d[2][k] - R(48) * U0[k]) * C.i8n2;  // b4
    central(U, V, hq, d[0], x);
    central(U, V, hq, d[1], y);
    central(U, V, hq, d[2], xx);
    central(U, V, hq, d[3], xy);
    central(U, V, hq, d[4], yy);
  }
  R A[4], tx[4], ty[4], tt[4], S[4], qx[4], qy[4];
  const R px = pN * xx[3], pxy = pN * xy[3], pyy = pN * yy[3], pt = px + pyy;
  const R dx = xx[1] + xy[2], dy = xy[1] + yy[2];
  time_coef(U, V, pN, kc, x, y, A);  // <A + a1 u + a2 v> = 0
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    qx[k] = U * xx[k] + V * xy[k];
    qy[k] = U * xy[k] + V * yy[k];
  }
  // <Axx u + Axy v + Atx> = 0, <Axy u + Ayy v + Aty> = 0
  tx[0] = -(qx[0] + dx);
  tx[1] = -(qx[1] + px);
  tx[2] = -(qx[2] + pxy);
  tx[3] = -(qx[3] + kc * dx);
  ty[0] = -(qy[0] + dy);
  ty[1] = -(qy[1] + pxy);
  ty[2] = -(qy[2] + pyy);
  ty[3] = -(qy[3] + kc * dy);
  // <Atx u + Aty v + Att> = 0
  const R qt0 = U * tx[0] + V * ty[0], qt1 = U * tx[1] + V * ty[1];
  const R qt2 = U * tx[2] + V * ty[2], qt3 = U * tx[3] + V * ty[3], dt1 = tx[1] + ty[2];
  tt[0] = -(qt0 + dt1);
  tt[1] = -(qt1 + pN * tx[3]);
  tt[2] = -(qt2 + pN * ty[3]);
  tt[3] = -(qt3 + kc * dt1);
  // S = <(Axx u^2 + 2 Axy u v + Ayy v^2) psi'>
  const R gg = U * dx + V * dy, s1 = s * (R(3) * xx[1] + R(2) * xy[2] + yy[1]);
  S[0] = (gg - qt0) + pt;
  S[1] = (U * px + V * pxy - qt1) + s1;
  S[2] = (U * pxy + V * pyy - qt2) + s * (xx[2] + R(2) * xy[1] + R(3) * yy[2]);
  S[3] = kc * (gg + R(2) * pt - s * (xx[0] + yy[0])) - qt3;
  // G0 = <psi' f> and G1 = <c psi' f>, time-integrated: the flux is U G0 + G1.  Both without g0's own part,
  // whose flux I1 (m, U m + p, V m, U (rho E + p)) is added at the end from U0 itself: the total
  // energy formed again from rho and s would round each time in a way that follows the flow, and such errors add up
  // from step to step (FP32 smooth wave 701 x 499, 48 steps, against 64 bits: 4.0e-7 so, 2.3e-7 from U0;
  // 512^2 7.4e-7 and 5.8e-7; step 43.9 -> 44.5 us).
  const R y2h = R(0.5) * C.y2, h4 = R(0.5) * w.I4, h5 = R(0.5) * w.I5;
  const R wA = w.I3 - w.I2, wyy = y2h * w.I1, wtt = h5 - w.I6;
  R G0[4], f[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) G0[k] = wA * A[k] + wyy * yy[k] + wtt * tt[k] + h4 * S[k];
  const R qa1 = U * x[1] + V * y[1], qa3 = U * x[3] + V * y[3];
  const R b1 = w.I3 * A[1] + h5 * tt[1] + wyy * yy[1] + w.I2 * qa1 + w.I6 * qt1 + h4 * (U * qx[1] + V * qy[1]);
  const R b3 = w.I3 * A[3] + h5 * tt[3] + wyy * yy[3] + w.I2 * qa3 + w.I6 * qt3 + h4 * (U * qx[3] + V * qy[3]);
  const R c0 = w.I2 * x[0] + w.I6 * tx[0] + w.I4 * qx[0], c1 = w.I2 * x[1] + w.I6 * tx[1] + w.I4 * qx[1];
  const R c2 = w.I2 * x[2] + w.I6 * tx[2] + w.I4 * qx[2], c3 = w.I2 * x[3] + w.I6 * tx[3] + w.I4 * qx[3];
  const R d1 = w.I2 * y[1] + w.I6 * ty[1] + w.I4 * qy[1], d2 = w.I2 * y[2] + w.I6 * ty[2] + w.I4 * qy[2];
  const R pB = pN * c3, z = h4 * s1, bz = b1 + pB;
  f[0] = U * G0[0] + (bz + z);
  f[1] = U * G0[1] + pN * b3 +
         s * ((R(3) * c1 + d2) + h4 * ((R(6) * px + R(2) * pyy) - s * (R(3) * xx[0] + yy[0])));
  f[2] = U * G0[2] + s * ((c2 + d1) + w.I4 * (R(2) * pxy - s * xy[0]));
  f[3] = U * G0[3] + kc * (bz + pB - s * c0) + C.n4h * s * z;
  lab(U, V, hq, f, Fl);
  const R mI = w.I1 * U0[1], pI = w.I1 * (r0 * s);
  Fl[0] += mI;
  Fl[1] += U * mI + pI;
  Fl[2] += V * mI;
  Fl[3] += U * (w.I1 * U0[3] + pI);
  if (C.prandtl) {
    lab(U, V, hq, G0, Mn);
#pragma unroll
    for (int k = 0; k < 4; ++k) Mn[k] += w.I1 * U0[k];
  }
  // values at t = dt: (1 - e) (U0 + dt U_t + ...), C_3 - C_2 = dt (1 - e),
  // C_5 / 2 - C_6 = dt^2/2 + dt tau e, C_4 = -(dt^2 + 2 dt tau) e
  const R pA = dt * w.om, pyw = y2h * w.om, te = w.te, ptt = dt * (R(0.5) * dt + te);
  const R pS = -dt * (R(0.5) * dt * w.e + te), rE = r0 * w.om;
  R p[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) p[k] = pA * A[k] + pyw * yy[k] + ptt * tt[k] + pS * S[k];
  p[0] += rE;
  p[3] += rE * (C.nh * s);
  lab(U, V, hq, p, P0);
#pragma unroll
  for (int k = 0; k < 4; ++k) p[k] = w.om * y[k] + pA * ty[k];
  lab(U, V, hq, p, P1);
}

// The coefficients of one side's Maxwellian in half_coef's basis, from its face state's derivatives
// (A, tx, ty: Navier-Stokes only)
template <class R>
struct KineticCoefs {
  R a1[4], a2[4], xx[4], xy[4], yy[4], A[4], tx[4], ty[4];
};

template <class R>
GKS_FN void kinetic_coefs(const FaceConst<R>& C, const FaceState<R>& S, const SideData<R>& sd, bool ns, KineticCoefs<R>& k) {
  const R U = sd.U, V = sd.V, s = sd.s;
  // FP32: formed again (two instructions) rather than kept in a register across the equilibrium part
  const R l2 = Prec<R>::fp64 ? sd.l2 : d_rcp(s);
  const R hq = R(0.5) * (U * U + V * V), hs = R(0.5) * (U * U + s), c5 = C.i2N * l2;
  R e1[4], e2[4], exx[4], exy[4], eyy[4];
  central(U, V, hq, S.w[1], e1);
  central(U, V, hq, S.w[2], e2);
  central(U, V, hq, S.w[3], exx);
  central(U, V, hq, S.w[4], exy);
  central(U, V, hq, S.w[5], eyy);
  half_coef(U, s, c5, hs, e1, k.a1);
  half_coef(U, s, c5, hs, e2, k.a2);
  half_coef(U, s, c5, hs, exx, k.xx);
  half_coef(U, s, c5, hs, exy, k.xy);
  half_coef(U, s, c5, hs, eyy, k.yy);
  if (ns) {
    const R kc = C.n2h * s;
    R t[4];
    time_coef(U, V, C.i2N, kc, e1, e2, t);
    half_coef(U, s, c5, hs, t, k.A);
    time_coef(U, V, C.i2N, kc, exx, exy, t);
    half_coef(U, s, c5, hs, t, k.tx);
    time_coef(U, V, C.i2N, kc, exy, eyy, t);
    half_coef(U, s, c5, hs, t, k.ty);
  }
}

// Kinetic part, Eq. dis2, of one side, added to Fl, P0, P1 and Mn: NS: f_G = g_k - tau (a u + A) g_k;
// Euler: f_G = g_k, the terms with tn are absent (not formed).  kin_point: e > 0.
template <class R>
GKS_FN void kinetic_part(const FaceConst<R>& C, const KineticCoefs<R>& kf, const SideData<R>& sd, bool ns, bool kin_point,
                         const TimeW<R>& w, R tn, R dt, R Fl[4], R P0[4], R P1[4], R Mn[4]) {
  const R rho = sd.rho, U = sd.U, V = sd.V, s = sd.s;
  const R l2 = Prec<R>::fp64 ? sd.l2 : d_rcp(s);
  const R *a1 = kf.a1, *a2 = kf.a2, *xx = kf.xx, *xy = kf.xy, *yy = kf.yy, *A = kf.A, *tx = kf.tx, *ty = kf.ty;
  R m[8];
  m[0] = sd.h;
  m[1] = sd.g;
#pragma unroll
  for (int n = 2; n < 8; ++n) m[n] = U * m[n - 1] + (n == 2 ? s : R(n - 1) * s) * m[n - 2];

  // P for the weights w7, w8 = -w9 and w10 of e^(-t/tau), -t e^(-t/tau) and t^2 e^(-t/tau):
  // v = V + d takes the terms in v to V times themselves and d times themselves
  auto poly = [&](R w7, R w9, R w10, HalfPoly<R>& P) {
    R B1[4], Bu[4], Bd[4], wq = R(0.5) * w10, wu = -w9;
    R t7 = tn * w7, t8 = -tn * w9;
    if (ns) {
      wq -= t8;
      wu -= t7;
      t7 *= l2;
      t8 *= l2;
    }
    // the coefficients carry a factor s
    wq *= l2;
    wu *= l2;
    const R wd = R(2) * wq * V, wyy = R(0.5) * C.y2 * (l2 * w7) - wq * V * V;  // B1 takes V Bd, which holds wd yy
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      Bd[k] = wu * a2[k] + wd * yy[k];
      Bu[k] = wu * a1[k] + wd * xy[k];
      if (ns) {
        Bd[k] = Bd[k] - t8 * ty[k];
        Bu[k] = Bu[k] - t8 * tx[k];
        B1[k] = V * Bd[k] + wyy * yy[k] - t7 * A[k];
      } else {
        B1[k] = V * Bd[k] + wyy * yy[k];
      }
    }
    half_poly(w7 * rho, B1, Bu, Bd, wq, xx, xy, yy, s, C.n1h, P);
  };
  HalfPoly<R> P;
  poly(w.i7, w.i9, w.i10, P);
  half_moments<1, 4>(P, m, V, s, C.n1h, Fl);
  if (C.prandtl) half_moments<0, 4>(P, m, V, s, C.n1h, Mn);
  // Every weight of the kinetic part at t = dt carries e = exp(-dt/tau), which underflows to
  // exactly 0 once tau is a small enough fraction of dt (smooth Euler flow): the point
  // values then get exactly nothing from this side
  if (kin_point) {
    const R e9 = dt * w.e;
    poly(w.e, e9, dt * e9, P);
    half_moments<0, 4>(P, m, V, s, C.n1h, P0);
    // the part linear along the face: y (e (a2 - tau Aty) - (t + tau) e (Axy u + Ayy v))
    const R el = l2 * w.e, wy = l2 * (ns ? -tn * w.e - e9 : -e9), te = tn * el;
    R B1[4], Bu[4], Bd[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      Bd[k] = wy * yy[k];
      Bu[k] = wy * xy[k];
      B1[k] = el * a2[k] + V * Bd[k];
      if (ns) B1[k] = B1[k] - te * ty[k];
    }
    half_poly_linear(B1, Bu, Bd, s, C.n1h, P);
    half_moments<0, 3>(P, m, V, s, C.n1h, P1);
  }
}

// the Prandtl-number fix, and the face's results from the accumulated moments
template <class R>
GKS_FN void finish_face(const FaceConst<R>& C, R u0, R v0, R Fl[4], const R P0[4], const R P1[4], const R Mn[4], R F[4],
                        R Wm[4], R Wp[4]) {
  // Prandtl-number fix: energy flux += (1/Pr - 1) q, q the time-integrated
  // face-mean heat flux (1/2) int (u-U0)((u-U0)^2+(v-V0)^2+xi^2) f, written with the
  // flux and the time-integrated conservative moments.
  if (C.prandtl) {
    const R q20 = u0 * u0 + v0 * v0;
    const R q = Fl[3] - u0 * Fl[1] - v0 * Fl[2] + (R(0.5) * q20 + u0 * u0) * Fl[0] - u0 * Mn[3] +
                u0 * v0 * Mn[2] - R(0.5) * u0 * q20 * Mn[0];
    Fl[3] += C.pr_fix * q;
  }
  const R yg = R(0.28867513459481287) * C.dtan;  // sqrt(3)/6
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    F[k] = Fl[k];
    Wm[k] = P0[k] - yg * P1[k];
    Wp[k] = P0[k] + yg * P1[k];
  }
}

// ---------------------------------------------------------------------------
// Section 2.2 at one face centre.  The two sides (value and derivatives in the
// face frame) and the six cell averages of Section 3.3 (avg[m][k], m = 0 left,
// 1 right; k = tangential -1, 0, 1) come from src.side(k, S) and src.avg(a),
// which are called where they are needed so that they need not stay live in
// registers.  Outputs the time-integrated face-mean flux and the point values
// at the two Gauss points (tangential -/+ sqrt(3)/6 dtan) at t = dt.
// NSM: 1 Navier-Stokes, 0 Euler (mu = 0: the terms of the time derivatives of
// g_k vanish and are not formed), -1 decided at run time by C.ns.
//
// Its bound is arithmetic: the FP32 kernels are held by issue slots, the FP64 ones by the FP64 pipe
// (one warp instruction per 19 cycles and SM), so fewer operations is what makes it faster.  Each Maxwellian
// is evaluated in its own frame, where g0's moments are closed forms in the central derivatives and a half-space's
// reduce to one-dimensional sums over u.  Against expanding the distribution into the monomials
// u^a v^b xi^2c (gks_face_monomials.cuh), in FP32: 1,238 instead of 2,041 counted flops at a smooth
// Euler face (exp(-dt/tau) = 0), 1,738 instead of 2,779 at another, 2,205 instead of 3,907
// Navier-Stokes with the Prandtl correction (FP64, erfc and exp as polynomials: 1,325, 1,825, 2,292).
// x-faces at 512^2 FP32 26.2 -> 20.7 us (Euler), at 1024^2 108 -> 81 us (Navier-Stokes), at
// 4096^2 1,177 -> 881 us; FP64 at 512^2 764 -> 534 us.  With the table for erfc and exp, the reciprocals and the
// launch shapes of today 19.8, 75 and 740 us, FP64 465 us.
// ---------------------------------------------------------------------------
template <class R, int NSM = -1, class Src>
GKS_FN void face_evolution(const FaceConst<R>& C, const Src& src, R dt, R F[4], R Wm[4], R Wp[4]) {
  const bool ns = NSM < 0 ? C.ns : NSM == 1;
  SideData<R> sd[2];
  R U0[4] = {R(0), R(0), R(0), R(0)};
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    FaceState<R> S;
    src.side(k, S);
    side_start(C, S.w[0], k, sd[k], U0);
  }
  R r0, ir0, u0, v0, p0;
  prim(U0, C.gm1, r0, ir0, u0, v0, p0);
  const R tau = collision_time(C, ns, sd[0].p, sd[1].p, p0, dt);
  TimeW<R> w;
  time_weights(dt, tau, w);
  // e = exp(-dt/tau) >= 0 underflows to exactly 0 once tau is a small enough fraction of dt
  // (smooth Euler flow); the point-value terms whose weights carry it are then not formed
  const bool kin_point = w.e > R(0);
  R Fl[4], P0[4], P1[4], Mn[4];
  {
    R avg[2][3][4], d[5][4];
    src.avg(avg);
    equilibrium_derivatives(C, avg, d);
    equilibrium_part(C, d, U0, r0, u0, v0, p0 * ir0, w, dt, Fl, P0, P1, Mn);
  }
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    FaceState<R> S;
    KineticCoefs<R> k;
    src.side(side, S);
    kinetic_coefs(C, S, sd[side], ns, k);
    kinetic_part(C, k, sd[side], ns, kin_point, w, ns ? tau : R(0), dt, Fl, P0, P1, Mn);
  }
  finish_face(C, u0, v0, Fl, P0, P1, Mn, F, Wm, Wp);
}

// ---------------------------------------------------------------------------
// Section 3.2: compact reconstruction of one variable of one cell.
// c: cell average; e, w, n, s: neighbour averages; em/ep: east-face Gauss
// values (y-/y+), wm/wp west face, nm/np north face (x-/x+), sm/sp south face.
// Output a[0..4] = (a2, a3, a4, a5, a6) of
//   U(x,y) = c + a2 x + a3 y + a4 (x^2-dx^2/12)/2 + a5 (y^2-dy^2/12)/2 + a6 x y.
// ---------------------------------------------------------------------------
template <class R>
GKS_FN R minmod(R a, R b) {
  return a * b > R(0) ? (fabs(a) < fabs(b) ? a : b) : R(0);
}

// Cell-size constants of the reconstruction, formed once per cell (not per variable)
template <class R>
struct ReconK {
  R dx, dy, idx, idy;
  R dx6, dy6;          // dx / 6, dy / 6
  R r3;                // sqrt(3) / (dx dy)
  R idx2, idy2;        // 1 / dx^2, 1 / dy^2
  R dx2, dy2;          // smoothness indicator: weights of c2^2, c3^2,
  R kc4, kc5, kc6;     //   c4^2 (13/12 dx^4), c5^2 (13/12 dy^4), c6^2 (7/6 dx^2 dy^2)
  R dx2_12, dy2_12;    // dx^2 / 12, dy^2 / 12 (face values of the polynomial)
  R weps, b1sq;        // eps and (eps + I(U1))^2, I(U1) = C dx dy
};

// idx, idy: 1/dx, 1/dy of the grid (formed once on the host)
template <class R>
GKS_FN ReconK<R> recon_k(R dx, R dy, R idx, R idy, R weps, R wC) {
  ReconK<R> k;
  k.dx = dx;
  k.dy = dy;
  k.idx = idx;
  k.idy = idy;
  k.idx2 = idx * idx;
  k.idy2 = idy * idy;
  k.dx6 = dx * R(1.0 / 6.0);
  k.dy6 = dy * R(1.0 / 6.0);
  k.r3 = R(1.7320508075688772) * idx * idy;  // sqrt(3) / (dx dy)
  k.dx2 = dx * dx;
  k.dy2 = dy * dy;
  k.kc4 = R(13.0 / 12.0) * k.dx2 * k.dx2;
  k.kc5 = R(13.0 / 12.0) * k.dy2 * k.dy2;
  k.kc6 = R(7.0 / 6.0) * k.dx2 * k.dy2;
  k.dx2_12 = k.dx2 * R(1.0 / 12.0);
  k.dy2_12 = k.dy2 * R(1.0 / 12.0);
  k.weps = weps;
  const R b1 = weps + wC * dx * dy;
  k.b1sq = b1 * b1;
  return k;
}

template <class R>
GKS_FN void recon_var(R c, R e, R w, R n, R s, R em, R ep, R wm, R wp, R nm, R np, R sm, R sp,
                      const ReconK<R>& K, R a[5]) {
  // one-sided stencils (Eq. over-sys) from each face's Gauss-point sum (twice its mean) and
  // the neighbour average
  const R se = em + ep, sw = wm + wp, sn = nm + np, ss = sm + sp;
  const R a4 = minmod(R(3) * (c + w - sw) * K.idx2, R(3) * (c + e - se) * K.idx2);
  const R a2 = minmod((R(2) * c - sw) * K.idx + a4 * K.dx6, (se - R(2) * c) * K.idx - a4 * K.dx6);
  const R a5 = minmod(R(3) * (c + s - ss) * K.idy2, R(3) * (c + n - sn) * K.idy2);
  const R a3 = minmod((R(2) * c - ss) * K.idy + a5 * K.dy6, (sn - R(2) * c) * K.idy - a5 * K.dy6);
  // cross derivative of the four one-sided stencils with limited a2, a3:
  // sx (sqrt3 Dx/(dx dy) - a3/dx) + sy (sqrt3 Dy/(dx dy) - a2/dy), smallest magnitude
  const R xe = K.r3 * (ep - em) - a3 * K.idx, xw = K.r3 * (wp - wm) - a3 * K.idx;
  const R yn = K.r3 * (np - nm) - a2 * K.idy, ys = K.r3 * (sp - sm) - a2 * K.idy;
  // magnitudes within a relative Prec<R>::tie of the current choice are ties
  // (piecewise constant data give exact ties of opposite sign); the earlier
  // stencil is kept
  const R keep = R(1) - R(Prec<R>::tie);
  R a6 = xe + yn;        // (+, +)
  R cand = -xw + yn;     // (-, +)
  if (fabs(cand) < fabs(a6) * keep) a6 = cand;
  cand = -xw - ys;       // (-, -)
  if (fabs(cand) < fabs(a6) * keep) a6 = cand;
  cand = xe - ys;        // (+, -)
  if (fabs(cand) < fabs(a6) * keep) a6 = cand;
  // central stencil
  const R c2 = R(0.5) * (e - w) * K.idx, c4 = (e - R(2) * c + w) * K.idx2;
  const R c3 = R(0.5) * (n - s) * K.idy, c5 = (n - R(2) * c + s) * K.idy2;
  const R c6 = R(0.5) * K.r3 * ((ep - em) - (wp - wm) + (np - nm) - (sp - sm));
  // Eq. average: alpha = 1/(eps + I)^2, I(U1) = C dx dy; I(U2), the integral of the
  // squared first and second derivatives of the central polynomial over the cell scaled
  // by |Omega|, collected by coefficient
  const R I2 = c2 * (K.dx2 * c2) + c3 * (K.dy2 * c3) + c4 * (K.kc4 * c4) + c5 * (K.kc5 * c5) + c6 * (K.kc6 * c6);
  const R b2 = K.weps + I2, b2sq = b2 * b2;
  // w1 = (1/b1^2) / (1/b1^2 + 1/b2^2) = b2^2 / (b1^2 + b2^2); a = c + w1 (a_one-sided - c)
  const R w1 = d_div(b2sq, K.b1sq + b2sq);
  a[0] = c2 + w1 * (a2 - c2);
  a[1] = c3 + w1 * (a3 - c3);
  a[2] = c4 + w1 * (a4 - c4);
  a[3] = c5 + w1 * (a5 - c5);
  a[4] = c6 + w1 * (a6 - c6);
}

// ---------------------------------------------------------------------------
// The FP64 form of the same reconstruction of one variable, in units of the cell size: the
// coefficients come out as (a2 dx, a3 dy, a4 dx^2, a5 dy^2, a6 dx dy).  It is bound by the FP64 pipe,
// so the cell size enters once at the end, comparisons of magnitudes and signs run on the integer pipe
// (|a| < |b| as the ordering of their bits), and the weight's quotient is a reciprocal: 86 FP64
// instructions instead of about 115.  Infinities and NaN among the stencil values reach the smoothness
// indicator and make every coefficient NaN, as before.
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool abs_less(double a, double b) {
  return (__double_as_longlong(a) & 0x7fffffffffffffffll) < (__double_as_longlong(b) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ double minmod_bits(double a, double b) {
  return (__double2hiint(a) ^ __double2hiint(b)) < 0 ? 0.0 : (abs_less(a, b) ? a : b);
}

__device__ __forceinline__ void recon_var_scaled(double c, double e, double w, double n, double s, double em, double ep,
                                                 double wm, double wp, double nm, double np, double sm, double sp,
                                                 double weps, double b1sq, double a[5]) {
  constexpr double r3 = 1.7320508075688772, sixth = 1.0 / 6.0;
  const double se = em + ep, sw = wm + wp, sn = nm + np, ss = sm + sp, cc = c + c;
  const double ce = c + e, cw = c + w, cn = c + n, cs = c + s;
  const double a4 = 3.0 * minmod_bits(cw - sw, ce - se), a5 = 3.0 * minmod_bits(cs - ss, cn - sn);
  const double a2 = minmod_bits((cc - sw) + sixth * a4, (se - cc) - sixth * a4);
  const double a3 = minmod_bits((cc - ss) + sixth * a5, (sn - cc) - sixth * a5);
  const double de = ep - em, dw = wp - wm, dn = np - nm, ds = sp - sm;
  const double xe = r3 * de - a3, xw = r3 * dw - a3, yn = r3 * dn - a2, ys = r3 * ds - a2;
  constexpr double keep = 1.0 - Prec<double>::tie;
  double a6 = xe + yn, cand = yn - xw;
  if (abs_less(cand, a6 * keep)) a6 = cand;
  cand = -xw - ys;
  if (abs_less(cand, a6 * keep)) a6 = cand;
  cand = xe - ys;
  if (abs_less(cand, a6 * keep)) a6 = cand;
  const double c2 = 0.5 * (e - w), c3 = 0.5 * (n - s), c4 = (ce + cw) - 2.0 * cc, c5 = (cn + cs) - 2.0 * cc;
  const double c6 = (0.5 * r3) * ((de - dw) + (dn - ds));
  const double I2 = c2 * c2 + c3 * c3 + (13.0 / 12.0) * (c4 * c4 + c5 * c5) + (7.0 / 6.0) * (c6 * c6);
  const double b2 = weps + I2, b2sq = b2 * b2, w1 = b2sq * d_rcp(b1sq + b2sq);
  a[0] = c2 + w1 * (a2 - c2);
  a[1] = c3 + w1 * (a3 - c3);
  a[2] = c4 + w1 * (a4 - c4);
  a[3] = c5 + w1 * (a5 - c5);
  a[4] = c6 + w1 * (a6 - c6);
}

}  // namespace gks
