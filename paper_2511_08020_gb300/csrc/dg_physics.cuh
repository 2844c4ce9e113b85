// Pointwise physics of the element and face kernels: fluxes, two-point fluxes,
// viscous terms and their hand-written adjoints.
#pragma once
#include "dg_kernels.cuh"

namespace dgk {
namespace {

__device__ __forceinline__ bool finite_bits(double x) {
  // exponent field all ones <=> inf or nan (integer test, no FP64 pipe work)
  return ((__double_as_longlong(x) >> 52) & 0x7ff) != 0x7ff;
}

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ unsigned smid() {
  unsigned r;
  asm volatile("mov.u32 %0, %%smid;" : "=r"(r));
  return r;
}

// 1/a: the hardware's estimate x (20 bits or more) and one step of
// Householder's method of order two, x + x (e + e^2) with e = 1 - a x; the
// neglected e^3 is below 2^-60, so the result is the rounded quotient but for
// a few parts in 2^7 of the last bit (0.51 units of it at most, the division
// 0.5).  Arguments near the ends of the range take the division.
__device__ __forceinline__ double rcp(double a) {
  const unsigned ex = ((unsigned)__double2hiint(a) >> 20) & 0x7ffu;
  if (ex - 30u > 1980u) return 1.0 / a;
  double x;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x) : "d"(a));
  const double e = fma(-a, x, 1.0);
  return fma(x, fma(e, e, e), x);
}

// sqrt(a): with y the hardware's estimate of 1/sqrt(a), g = a y, and
// delta = 1 - a y^2 (below 2^-19), sqrt(a) = g (1 - delta)^(-1/2) =
// g + g delta (1/2 + 3 delta/8) + O(delta^3); g delta = (a - g^2) y takes the
// rounding of g into account.
__device__ __forceinline__ double sqrt_hw(double a) {
  const unsigned hi = (unsigned)__double2hiint(a), ex = hi >> 20;
  if (ex - 100u > 1900u) return sqrt(a);   // zero, subnormal, negative, infinite, NaN or extreme
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
  const double g = a * y, r = fma(-g, g, a), h = r * y;
  return fma(h, fma(0.375, h * y, 0.5), g);
}

// ------------------------------------------------------------------ physics
// Euler normal flux F(U).n with u.n, p, 1/rho and c^2 as by-products.
struct NState {
  double F[5];
  double un, p, rinv, H;
};

__device__ __forceinline__ void normal_state(const double* U, const double* n, double gamma, NState& s) {
  s.rinv = rcp(U[0]);
  double u = U[1] * s.rinv, v = U[2] * s.rinv, w = U[3] * s.rinv;
  s.p = (gamma - 1.0) * (U[4] - 0.5 * (U[1] * u + U[2] * v + U[3] * w));
  s.un = u * n[0] + v * n[1] + w * n[2];
  s.F[0] = U[0] * s.un;
  s.F[1] = U[1] * s.un + s.p * n[0];
  s.F[2] = U[2] * s.un + s.p * n[1];
  s.F[3] = U[3] * s.un + s.p * n[2];
  s.F[4] = (U[4] + s.p) * s.un;
  s.H = (U[4] + s.p) * s.rinv;
}

// Lax-Friedrichs: F* = (F- + F+)/2 - lambda (U+ - U-)/2,
// lambda = max(|u-.n| + c-, |u+.n| + c+), multiplied by the face weight
// wS = w S of the point and arranged for few FP64 instructions: with the scaled
// normal s = (wS/2) n and us = m.s/rho per side,
//   wS F*_rho = m-.s + m+.s + lam (rho- - rho+),
//   wS F*_m   = m- us- + m+ us+ + (p- + p+) s + lam (m- - m+),
//   wS F*_E   = (E- + p-) us- + (E+ + p+) us+ + lam (E- - E+),
//   lam       = max(|us-| + (wS/2) c-, |us+| + (wS/2) c+),
// one reciprocal and one square root per side.  fmax passes over the NaN of a
// side whose pressure is negative, so the other side's speed is taken there.
// The face kernel is bound by FP64 issue (16^3 mixed N = 4: 151 us with the
// division, the root and separate side fluxes, 140 with the reciprocals alone,
// 130 in this form; the Navier-Stokes flux phase at 12^3 164 -> 128 us).
struct LfSide {
  double r, p, ms, us, lam;
};

// sig: the face's normal mesh speed times wS/2 (moving meshes), else zero
template <bool MOVING>
__device__ __forceinline__ void lf_side(const double* U, const double* s, double h, double sig, double gm1,
                                        double gamma, LfSide& o) {
  o.r = rcp(U[0]);
  o.ms = fma(U[1], s[0], fma(U[2], s[1], U[3] * s[2]));
  o.us = o.ms * o.r;
  const double m2 = fma(U[1], U[1], fma(U[2], U[2], U[3] * U[3]));
  o.p = gm1 * fma(-0.5 * o.r, m2, U[4]);
  o.lam = fma(h, sqrt_hw(gamma * o.p * o.r), fabs(MOVING ? o.us - sig : o.us));
}

__device__ __forceinline__ void lf_combine(const double* UL, const double* UR, const double* s, const LfSide& L,
                                           const LfSide& R, double* Fs) {
  const double lam = fmax(L.lam, R.lam), P = L.p + R.p;
  Fs[0] = fma(lam, UL[0] - UR[0], L.ms + R.ms);
#pragma unroll
  for (int d = 0; d < 3; ++d)
    Fs[1 + d] = fma(lam, UL[1 + d] - UR[1 + d], fma(UL[1 + d], L.us, fma(UR[1 + d], R.us, P * s[d])));
  Fs[4] = fma(lam, UL[4] - UR[4], fma(UL[4] + L.p, L.us, (UR[4] + R.p) * R.us));
}

// The same in a frame moving with normal speed sn = xdot.n at the point: the
// side fluxes lose sig U, sig = (wS/2) sn.
__device__ __forceinline__ void lf_combine_moving(const double* UL, const double* UR, const double* s, double sig,
                                                  const LfSide& L, const LfSide& R, double* Fs) {
  const double lam = fmax(L.lam, R.lam), P = L.p + R.p, wL = L.us - sig, wR = R.us - sig;
  Fs[0] = fma(lam, UL[0] - UR[0], fma(-sig, UL[0], L.ms) + fma(-sig, UR[0], R.ms));
#pragma unroll
  for (int d = 0; d < 3; ++d)
    Fs[1 + d] = fma(lam, UL[1 + d] - UR[1 + d], fma(UL[1 + d], wL, fma(UR[1 + d], wR, P * s[d])));
  Fs[4] = fma(lam, UL[4] - UR[4], fma(UL[4], wL, fma(UR[4], wR, fma(L.p, L.us, R.p * R.us))));
}

__device__ __forceinline__ void flux_lf_scaled(const double* UL, const double* UR, const double* n, double wS,
                                               double gamma, double* Fs) {
  const double h = 0.5 * wS, gm1 = gamma - 1.0;
  const double s[3] = {h * n[0], h * n[1], h * n[2]};
  LfSide L, R;
  lf_side<false>(UL, s, h, 0.0, gm1, gamma, L);
  lf_side<false>(UR, s, h, 0.0, gm1, gamma, R);
  lf_combine(UL, UR, s, L, R, Fs);
}

__device__ __forceinline__ void flux_lf_moving_scaled(const double* UL, const double* UR, const double* n, double wS,
                                                      double sn, double gamma, double* Fs) {
  const double h = 0.5 * wS, gm1 = gamma - 1.0, sig = h * sn;
  const double s[3] = {h * n[0], h * n[1], h * n[2]};
  LfSide L, R;
  lf_side<true>(UL, s, h, sig, gm1, gamma, L);
  lf_side<true>(UR, s, h, sig, gm1, gamma, R);
  lf_combine_moving(UL, UR, s, sig, L, R, Fs);
}

// Roe: F* = (F- + F+)/2 - sum_k |lambda_k| alpha_k r_k / 2 with
// sqrt(rho)-weighted averages of u and H, no entropy fix.
__device__ __forceinline__ void flux_roe(const double* UL, const double* UR, const double* n, double gamma, double* Fs) {
  NState L, R;
  normal_state(UL, n, gamma, L);
  normal_state(UR, n, gamma, R);
  double sL = sqrt_hw(UL[0]), sR = sqrt_hw(UR[0]);
  double den = rcp(sL + sR);
  double uL[3] = {UL[1] * L.rinv, UL[2] * L.rinv, UL[3] * L.rinv};
  double uR[3] = {UR[1] * R.rinv, UR[2] * R.rinv, UR[3] * R.rinv};
  double u[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) u[d] = (sL * uL[d] + sR * uR[d]) * den;
  double H = (sL * L.H + sR * R.H) * den;
  double rho = sL * sR;
  double q2 = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
  double c2 = (gamma - 1.0) * (H - 0.5 * q2);
  double c = sqrt_hw(c2);
  double un = u[0] * n[0] + u[1] * n[1] + u[2] * n[2];
  double drho = UR[0] - UL[0], dp = R.p - L.p;
  double du[3] = {uR[0] - uL[0], uR[1] - uL[1], uR[2] - uL[2]};
  double dun = du[0] * n[0] + du[1] * n[1] + du[2] * n[2];
  double ic2 = rcp(c2);
  double a1 = 0.5 * (dp - rho * c * dun) * ic2;
  double a5 = 0.5 * (dp + rho * c * dun) * ic2;
  double a2 = drho - dp * ic2;
  double l1 = fabs(un - c) * a1, l5 = fabs(un + c) * a5, l2 = fabs(un);
  double dut[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) dut[d] = du[d] - dun * n[d];
  double D[5];
  D[0] = l1 + l5 + l2 * a2;
#pragma unroll
  for (int d = 0; d < 3; ++d) D[1 + d] = l1 * (u[d] - c * n[d]) + l5 * (u[d] + c * n[d]) + l2 * (a2 * u[d] + rho * dut[d]);
  double udut = u[0] * dut[0] + u[1] * dut[1] + u[2] * dut[2];
  D[4] = l1 * (H - c * un) + l5 * (H + c * un) + l2 * (a2 * 0.5 * q2 + rho * udut);
#pragma unroll
  for (int v = 0; v < 5; ++v) Fs[v] = 0.5 * (L.F[v] + R.F[v]) - 0.5 * D[v];
}

// ------------------------------------------------------------------ two-point flux (split form)
//
// Entropy-stable split form (Sec. 2: entropy-stable DGSEM with a
// summation-by-parts property and Chandrashekar's two-point flux) for the
// entropy U = -rho s/(gamma-1), s = ln(p rho^-gamma).  A state enters the
// two-point flux through kTP = 8 quantities: rho, u, v, w, beta = rho/(2p),
// ln rho, ln beta, |u|^2.
constexpr int kTP = 8;
constexpr double kLn2 = 0.69314718055994530942;

__device__ __forceinline__ void two_point_state(const double* U, double gm1, double* P) {
  const double r = U[0], ri = rcp(r);
  const double u = U[1] * ri, v = U[2] * ri, w = U[3] * ri;
  const double q2 = fma(u, u, fma(v, v, w * w));
  const double p = gm1 * fma(-0.5 * r, q2, U[4]);
  const double b = 0.5 * r / p;
  P[0] = r;
  P[1] = u;
  P[2] = v;
  P[3] = w;
  P[4] = b;
  P[5] = log(r);
  P[6] = log(b);
  P[7] = q2;
}

// Logarithmic mean (a - b)/(ln a - ln b) from the values and their logs.
// With f = (a - b)/(a + b) and u = f^2: for u < 1e-2 it is
// ((a + b)/2) f/artanh(f), the ratio from its Taylor series in u through u^7
// (f/artanh(f) = 1/(1 + u/3 + u^2/5 + ...); truncation below 2e-18), else the
// quotient of the differences (whose denominator is then at least 0.2).
__device__ __forceinline__ double ln_mean(double a, double b, double la, double lb) {
  const double d = a - b, sm = a + b;
  if (d * d < 1e-2 * sm * sm) {
    const double f = d * rcp(sm), u = f * f;
    double g = -5472607916.0 / 488462349375.0;
    g = fma(g, u, -25865068.0 / 1915538625.0);
    g = fma(g, u, -10719068.0 / 638512875.0);
    g = fma(g, u, -10196.0 / 467775.0);
    g = fma(g, u, -428.0 / 14175.0);
    g = fma(g, u, -44.0 / 945.0);
    g = fma(g, u, -4.0 / 45.0);
    g = fma(g, u, -1.0 / 3.0);
    g = fma(g, u, 1.0);
    return 0.5 * sm * g;
  }
  return d / (la - lb);
}

// Chandrashekar's two-point flux F#(L, R) contracted with m:
//   F_rho = rho_ln (u_bar . m),  F_mom = p_hat m + u_bar F_rho,
//   F_E = (1/(2 (gamma-1) beta_ln) - |u|^2_bar/2) F_rho + u_bar . F_mom,
// bars arithmetic means, _ln logarithmic means, p_hat = rho_bar/(2 beta_bar).
__device__ __forceinline__ void two_point_flux(const double* L, int sl, const double* R, int sr, const double* m,
                                               double igm1, double* F) {
  const double rho_ln = ln_mean(L[0], R[0], L[5 * sl], R[5 * sr]);
  // beta: one reciprocal of beta_L + beta_R serves p_hat and the series
  // branch of 1/beta_ln
  const double bL = L[4 * sl], bR = R[4 * sr];
  const double db = bL - bR, sb = bL + bR, isb = rcp(sb);
  double ib_ln;
  if (db * db < 1e-2 * sb * sb) {
    const double f = db * isb, u2 = f * f;
    double h = 1.0 / 15.0;
    h = fma(h, u2, 1.0 / 13.0);
    h = fma(h, u2, 1.0 / 11.0);
    h = fma(h, u2, 1.0 / 9.0);
    h = fma(h, u2, 1.0 / 7.0);
    h = fma(h, u2, 1.0 / 5.0);
    h = fma(h, u2, 1.0 / 3.0);
    h = fma(h, u2, 1.0);
    ib_ln = 2.0 * isb * h;
  } else {
    ib_ln = (L[6 * sl] - R[6 * sr]) / db;
  }
  const double u = 0.5 * (L[sl] + R[sr]), v = 0.5 * (L[2 * sl] + R[2 * sr]), w = 0.5 * (L[3 * sl] + R[3 * sr]);
  const double p_hat = 0.5 * (L[0] + R[0]) * isb;
  const double q2 = 0.5 * (L[7 * sl] + R[7 * sr]);
  const double F0 = rho_ln * fma(u, m[0], fma(v, m[1], w * m[2]));
  F[0] = F0;
  F[1] = fma(p_hat, m[0], u * F0);
  F[2] = fma(p_hat, m[1], v * F0);
  F[3] = fma(p_hat, m[2], w * F0);
  F[4] = fma(fma(0.5 * igm1, ib_ln, -0.5 * q2), F0, fma(u, F[1], fma(v, F[2], w * F[3])));
}

// Entropy variables v = ((gamma - s)/(gamma - 1) - beta |u|^2, 2 beta u, -2 beta)
// from the two-point quantities (s = ln p - gamma ln rho, ln p = ln rho - ln(2 beta)).
__device__ __forceinline__ void entropy_variables(const double* P, int sp, double gamma, double* v) {
  const double igm1 = 1.0 / (gamma - 1.0);
  const double lnp = P[5 * sp] - kLn2 - P[6 * sp];
  const double s = lnp - gamma * P[5 * sp];
  const double b2 = 2.0 * P[4 * sp];
  v[0] = fma(gamma - s, igm1, -P[4 * sp] * P[7 * sp]);
  v[1] = b2 * P[sp];
  v[2] = b2 * P[2 * sp];
  v[3] = b2 * P[3 * sp];
  v[4] = -b2;
}

// The inverse: conservative state U and its two-point quantities P from
// entropy variables: beta = -v4/2, u = -v_{1..3}/v4,
// s = gamma - (gamma - 1)(v0 + beta |u|^2), ln rho = -(s + ln(2 beta))/(gamma - 1).
__device__ __forceinline__ void from_entropy_variables(const double* v, double gamma, double* U, double* P) {
  const double igm1 = 1.0 / (gamma - 1.0);
  const double b = -0.5 * v[4];
  const double iv4 = rcp(v[4]);
  const double u = -v[1] * iv4, vv = -v[2] * iv4, w = -v[3] * iv4;
  const double q2 = fma(u, u, fma(vv, vv, w * w));
  const double s = gamma - (gamma - 1.0) * fma(b, q2, v[0]);
  const double lb = log(b);
  const double lr = -(s + kLn2 + lb) * igm1;
  const double r = exp(lr);
  const double p = 0.5 * r / b;
  U[0] = r;
  U[1] = r * u;
  U[2] = r * vv;
  U[3] = r * w;
  U[4] = fma(p, igm1, 0.5 * r * q2);
  P[0] = r;
  P[1] = u;
  P[2] = vv;
  P[3] = w;
  P[4] = b;
  P[5] = lr;
  P[6] = lb;
  P[7] = q2;
}

// ------------------------------------------------------------------ viscous physics
//
// Navier-Stokes-Fourier fluxes with BR1 lifting of the primitive variables
// W = (rho, u, v, w, p): g[d * 5 + v] = dW_v / dx_d (the lifted gradient),
//   tau  = mu (grad u + grad u^T - 2/3 div u I)          (Stokes hypothesis)
//   F_v[d] = (0, tau_{x d}, tau_{y d}, tau_{z d}, u . tau_{. d} + kappa d(p/rho)/dx_d)
// with kappa = mu gamma / ((gamma - 1) Pr) (Fourier heat flux q = -kappa grad(p/rho)).

__device__ __forceinline__ void primitive(const double* U, double gm1, double* W) {
  const double r = rcp(U[0]);
  W[0] = U[0];
  W[1] = U[1] * r;
  W[2] = U[2] * r;
  W[3] = U[3] * r;
  W[4] = gm1 * (U[4] - 0.5 * (U[1] * W[1] + U[2] * W[2] + U[3] * W[3]));
}

__device__ __forceinline__ void viscous_flux(const double* W, const double* g, double mu, double kappa,
                                             double Fv[3][5]) {
  const double div = g[1] + g[5 + 2] + g[10 + 3];
  const double rinv = rcp(W[0]), Tr = W[4] * rinv;
  const double lam = (2.0 / 3.0) * mu * div;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    double tau[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) tau[i] = mu * (g[d * 5 + 1 + i] + g[i * 5 + 1 + d]) - (i == d ? lam : 0.0);
    const double dT = (g[d * 5 + 4] - Tr * g[d * 5]) * rinv;
    Fv[d][0] = 0.0;
    Fv[d][1] = tau[0];
    Fv[d][2] = tau[1];
    Fv[d][3] = tau[2];
    Fv[d][4] = W[1] * tau[0] + W[2] * tau[1] + W[3] * tau[2] + kappa * dT;
  }
}

// Viscous flux through a face, F_v.s for a (scaled) normal s, from 1/rho, the
// velocity, p and the gradient: q[0..2] momentum, q[3] energy.  The traction is
// contracted with s before the stress is formed: about half the operations of
// the three fluxes and their contraction.
__device__ __forceinline__ void viscous_flux_normal(double r, const double* u, double p, const double* g,
                                                    const double* s, double mu, double kappa, double* q) {
  const double lam = (2.0 / 3.0) * mu * (g[1] + g[5 + 2] + g[10 + 3]);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    double a = s[0] * g[1 + i];
    a = fma(s[1], g[5 + 1 + i], a);
    a = fma(s[2], g[10 + 1 + i], a);
#pragma unroll
    for (int d = 0; d < 3; ++d) a = fma(s[d], g[i * 5 + 1 + d], a);
    q[i] = fma(mu, a, -lam * s[i]);
  }
  const double gp = fma(s[0], g[4], fma(s[1], g[9], s[2] * g[14]));
  const double gr = fma(s[0], g[0], fma(s[1], g[5], s[2] * g[10]));
  const double dT = fma(-p * r, gr, gp) * r;
  q[3] = fma(kappa, dT, fma(u[0], q[0], fma(u[1], q[1], u[2] * q[2])));
}

// Reverse mode of viscous_flux: Fb[d][v] cotangent of F_v[d][v]; adds the
// cotangents of W (5) to Wb and of the gradient (15) to gb.
__device__ __forceinline__ void viscous_flux_vjp(const double* W, const double* g, double mu, double kappa,
                                                 const double Fb[3][5], double* Wb, double* gb) {
  const double div = g[1] + g[5 + 2] + g[10 + 3];
  const double rinv = rcp(W[0]), Tr = W[4] * rinv;
  const double lam = (2.0 / 3.0) * mu * div;
  double lamb = 0.0, rinvb = 0.0, Trb = 0.0;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const double e = Fb[d][4];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const double tau = mu * (g[d * 5 + 1 + i] + g[i * 5 + 1 + d]) - (i == d ? lam : 0.0);
      const double taub = Fb[d][1 + i] + W[1 + i] * e;
      Wb[1 + i] += tau * e;
      gb[d * 5 + 1 + i] += mu * taub;
      gb[i * 5 + 1 + d] += mu * taub;
      if (i == d) lamb -= taub;
    }
    const double dTb = kappa * e;
    gb[d * 5 + 4] += dTb * rinv;
    gb[d * 5] -= Tr * rinv * dTb;
    Trb -= g[d * 5] * rinv * dTb;
    rinvb += (g[d * 5 + 4] - Tr * g[d * 5]) * dTb;
  }
  Wb[4] += rinv * Trb;
  rinvb += W[4] * Trb;
  Wb[0] -= rinv * rinv * rinvb;
  const double divb = (2.0 / 3.0) * mu * lamb;
  gb[1] += divb;
  gb[5 + 2] += divb;
  gb[10 + 3] += divb;
}

// Reverse mode of primitive: adds the cotangent of U to Ub.
__device__ __forceinline__ void primitive_vjp(const double* U, double gm1, const double* Wb, double* Ub) {
  const double r = rcp(U[0]);
  const double hp = 0.5 * gm1 * Wb[4];
  double rb = 0.0;
  Ub[4] += gm1 * Wb[4];
#pragma unroll
  for (int i = 1; i <= 3; ++i) {
    const double Wi = U[i] * r;
    const double Wib = Wb[i] - hp * U[i];
    Ub[i] += r * Wib - hp * Wi;
    rb += U[i] * Wib;
  }
  Ub[0] += Wb[0] - r * r * rb;
}

// ------------------------------------------------------------------ adjoint physics
// Hand-written reverse mode of the functions above.  Readings at the kinks:
// d|x|/dx = sign(x) with sign(0) = 0; max(aL, aR) passes its cotangent to the
// left ('-') argument at ties.

__device__ __forceinline__ double sgn0(double x) { return x > 0.0 ? 1.0 : (x < 0.0 ? -1.0 : 0.0); }

// Cotangents of a side's normal-state quantities -> cotangent of U.
// Fb: cotangent of F(U).n; unb, pb, Hb: of u.n, p, H; ub: of u (3).
__device__ __forceinline__ void normal_state_vjp(const double* U, const double* n, double gamma, const NState& s,
                                                 const double* Fb, double unb, double pb, double Hb, double* ub,
                                                 double* Ub) {
  const double gm1 = gamma - 1.0;
  const double u[3] = {U[1] * s.rinv, U[2] * s.rinv, U[3] * s.rinv};
  // F[0] = rho un ; F[1+i] = m_i un + p n_i ; F[4] = (E + p) un
  Ub[0] += Fb[0] * s.un;
  unb += Fb[0] * U[0];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    Ub[1 + i] += Fb[1 + i] * s.un;
    unb += Fb[1 + i] * U[1 + i];
    pb += Fb[1 + i] * n[i];
  }
  Ub[4] += Fb[4] * s.un;
  pb += Fb[4] * s.un;
  unb += Fb[4] * (U[4] + s.p);
  // H = (E + p) / rho
  Ub[4] += Hb * s.rinv;
  pb += Hb * s.rinv;
  Ub[0] -= Hb * s.H * s.rinv;
  // un = u.n
#pragma unroll
  for (int d = 0; d < 3; ++d) ub[d] += unb * n[d];
  // p = (gamma-1)(E - |m|^2 / (2 rho))
  Ub[4] += gm1 * pb;
  const double q2 = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
#pragma unroll
  for (int d = 0; d < 3; ++d) Ub[1 + d] -= gm1 * u[d] * pb;
  Ub[0] += 0.5 * gm1 * q2 * pb;
  // u = m / rho
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    Ub[1 + d] += ub[d] * s.rinv;
    Ub[0] -= ub[d] * u[d] * s.rinv;
  }
}

// Lax-Friedrichs: given Fsb = cotangent of F*, accumulate UbL, UbR.
__device__ __forceinline__ void flux_lf_vjp(const double* UL, const double* UR, const double* n, double gamma,
                                            const double* Fsb, double* UbL, double* UbR) {
  NState L, R;
  normal_state(UL, n, gamma, L);
  normal_state(UR, n, gamma, R);
  const double cL = sqrt_hw(gamma * L.p * L.rinv), cR = sqrt_hw(gamma * R.p * R.rinv);
  const double aL = fabs(L.un) + cL, aR = fabs(R.un) + cR;
  const double lam = aL >= aR ? aL : aR;
  double Fb[5], lamb = 0.0;
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    Fb[v] = 0.5 * Fsb[v];
    lamb -= 0.5 * Fsb[v] * (UR[v] - UL[v]);
    UbR[v] -= 0.5 * lam * Fsb[v];
    UbL[v] += 0.5 * lam * Fsb[v];
  }
  const double aLb = aL >= aR ? lamb : 0.0, aRb = aL >= aR ? 0.0 : lamb;
  // c = sqrt(gamma p / rho): dc = gamma dp / (2 c rho) - c drho / (2 rho)
  double ubL[3] = {0, 0, 0}, ubR[3] = {0, 0, 0};
  const double pbL = 0.5 * aLb * gamma * L.rinv * rcp(cL), pbR = 0.5 * aRb * gamma * R.rinv * rcp(cR);
  UbL[0] -= aLb * 0.5 * cL * L.rinv;
  UbR[0] -= aRb * 0.5 * cR * R.rinv;
  normal_state_vjp(UL, n, gamma, L, Fb, sgn0(L.un) * aLb, pbL, 0.0, ubL, UbL);
  normal_state_vjp(UR, n, gamma, R, Fb, sgn0(R.un) * aRb, pbR, 0.0, ubR, UbR);
}

// Roe: given Fsb = cotangent of F*, accumulate UbL, UbR (reverse of flux_roe).
__device__ __forceinline__ void flux_roe_vjp(const double* UL, const double* UR, const double* n, double gamma,
                                             const double* Fsb, double* UbL, double* UbR) {
  NState L, R;
  normal_state(UL, n, gamma, L);
  normal_state(UR, n, gamma, R);
  // forward recomputation
  const double sL = sqrt_hw(UL[0]), sR = sqrt_hw(UR[0]);
  const double den = rcp(sL + sR);
  const double uL[3] = {UL[1] * L.rinv, UL[2] * L.rinv, UL[3] * L.rinv};
  const double uR[3] = {UR[1] * R.rinv, UR[2] * R.rinv, UR[3] * R.rinv};
  double u[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) u[d] = (sL * uL[d] + sR * uR[d]) * den;
  const double H = (sL * L.H + sR * R.H) * den;
  const double rho = sL * sR;
  const double q2 = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
  const double gm1 = gamma - 1.0;
  const double c2 = gm1 * (H - 0.5 * q2);
  const double c = sqrt_hw(c2);
  const double un = u[0] * n[0] + u[1] * n[1] + u[2] * n[2];
  const double dp = R.p - L.p;
  const double du[3] = {uR[0] - uL[0], uR[1] - uL[1], uR[2] - uL[2]};
  const double dun = du[0] * n[0] + du[1] * n[1] + du[2] * n[2];
  const double ic2 = rcp(c2);
  const double a1 = 0.5 * (dp - rho * c * dun) * ic2;
  const double a5 = 0.5 * (dp + rho * c * dun) * ic2;
  const double a2 = (UR[0] - UL[0]) - dp * ic2;
  const double e1 = fabs(un - c), e5 = fabs(un + c), l2 = fabs(un);
  const double l1 = e1 * a1, l5 = e5 * a5;
  double dut[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) dut[d] = du[d] - dun * n[d];
  const double udut = u[0] * dut[0] + u[1] * dut[1] + u[2] * dut[2];
  // reverse
  double Db[5], FbL[5], FbR[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    Db[v] = -0.5 * Fsb[v];
    FbL[v] = FbR[v] = 0.5 * Fsb[v];
  }
  double l1b = 0, l5b = 0, l2b = 0, Hb = 0, cb = 0, unb = 0, a2b = 0, q2b = 0, rhob = 0, udutb = 0;
  double ub[3] = {0, 0, 0}, dutb[3] = {0, 0, 0};
  // D4
  l1b += Db[4] * (H - c * un);
  l5b += Db[4] * (H + c * un);
  l2b += Db[4] * (a2 * 0.5 * q2 + rho * udut);
  Hb += Db[4] * (l1 + l5);
  cb += Db[4] * (l5 - l1) * un;
  unb += Db[4] * (l5 - l1) * c;
  a2b += Db[4] * l2 * 0.5 * q2;
  q2b += Db[4] * l2 * a2 * 0.5;
  rhob += Db[4] * l2 * udut;
  udutb += Db[4] * l2 * rho;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    ub[d] += udutb * dut[d];
    dutb[d] += udutb * u[d];
  }
  // D1..D3
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const double b = Db[1 + d];
    l1b += b * (u[d] - c * n[d]);
    l5b += b * (u[d] + c * n[d]);
    l2b += b * (a2 * u[d] + rho * dut[d]);
    ub[d] += b * (l1 + l5 + l2 * a2);
    cb += b * (l5 - l1) * n[d];
    a2b += b * l2 * u[d];
    rhob += b * l2 * dut[d];
    dutb[d] += b * l2 * rho;
  }
  // D0
  l1b += Db[0];
  l5b += Db[0];
  l2b += Db[0] * a2;
  a2b += Db[0] * l2;
  // dut = du - dun n
  double dub[3], dunb = 0.0;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    dub[d] = dutb[d];
    dunb -= dutb[d] * n[d];
  }
  // eigenvalue magnitudes
  unb += sgn0(un) * l2b;
  const double s5 = sgn0(un + c), s1 = sgn0(un - c);
  unb += s5 * a5 * l5b + s1 * a1 * l1b;
  cb += s5 * a5 * l5b - s1 * a1 * l1b;
  const double a5b = e5 * l5b, a1b = e1 * l1b;
  // wave strengths
  double dpb = 0, ic2b = 0, drhob = a2b;
  dpb -= a2b * ic2;
  ic2b -= a2b * dp;
  dpb += 0.5 * ic2 * (a5b + a1b);
  rhob += 0.5 * ic2 * c * dun * (a5b - a1b);
  cb += 0.5 * ic2 * rho * dun * (a5b - a1b);
  dunb += 0.5 * ic2 * rho * c * (a5b - a1b);
  ic2b += 0.5 * (dp + rho * c * dun) * a5b + 0.5 * (dp - rho * c * dun) * a1b;
  double c2b = -ic2b * ic2 * ic2;
#pragma unroll
  for (int d = 0; d < 3; ++d) dub[d] += dunb * n[d];
  // un = u.n
#pragma unroll
  for (int d = 0; d < 3; ++d) ub[d] += unb * n[d];
  // c = sqrt(c2), c2 = (gamma-1)(H - q2/2), q2 = |u|^2
  c2b += 0.5 * cb * rcp(c);
  Hb += gm1 * c2b;
  q2b -= 0.5 * gm1 * c2b;
#pragma unroll
  for (int d = 0; d < 3; ++d) ub[d] += 2.0 * u[d] * q2b;
  // Roe averages
  double sLb = rhob * sR, sRb = rhob * sL, denb = 0.0;
  double HLb = Hb * sL * den, HRb = Hb * sR * den;
  sLb += Hb * L.H * den;
  sRb += Hb * R.H * den;
  denb += Hb * (sL * L.H + sR * R.H);
  double ubL[3], ubR[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    sLb += ub[d] * uL[d] * den;
    sRb += ub[d] * uR[d] * den;
    ubL[d] = ub[d] * sL * den - dub[d];
    ubR[d] = ub[d] * sR * den + dub[d];
    denb += ub[d] * (sL * uL[d] + sR * uR[d]);
  }
  sLb -= denb * den * den;
  sRb -= denb * den * den;
  UbL[0] += 0.5 * sLb * rcp(sL) - drhob;
  UbR[0] += 0.5 * sRb * rcp(sR) + drhob;
  normal_state_vjp(UL, n, gamma, L, FbL, 0.0, -dpb, HLb, ubL, UbL);
  normal_state_vjp(UR, n, gamma, R, FbR, 0.0, dpb, HRb, ubR, UbR);
}

// Contravariant flux at a volume point (G_l = V_l U + p (0, M_l., V_l),
// V_l = M_l.u) in reverse: Gb[l][v] -> Ub[v].
__device__ __forceinline__ void contravariant_vjp(const double* U, const double M[3][3], double gamma,
                                                  const double Gb[3][5], double* Ub) {
  const double gm1 = gamma - 1.0;
  const double rinv = rcp(U[0]);
  const double u[3] = {U[1] * rinv, U[2] * rinv, U[3] * rinv};
  const double p = gm1 * (U[4] - 0.5 * (U[1] * u[0] + U[2] * u[1] + U[3] * u[2]));
  const double Ep = U[4] + p;
  double pb = 0.0, ub[3] = {0, 0, 0};
#pragma unroll
  for (int v = 0; v < 5; ++v) Ub[v] = 0.0;
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    const double Vl = M[l][0] * u[0] + M[l][1] * u[1] + M[l][2] * u[2];
    const double Vb = Gb[l][0] * U[0] + Gb[l][1] * U[1] + Gb[l][2] * U[2] + Gb[l][3] * U[3] + Gb[l][4] * Ep;
    Ub[0] += Gb[l][0] * Vl;
    Ub[1] += Gb[l][1] * Vl;
    Ub[2] += Gb[l][2] * Vl;
    Ub[3] += Gb[l][3] * Vl;
    Ub[4] += Gb[l][4] * Vl;
    pb += Gb[l][1] * M[l][0] + Gb[l][2] * M[l][1] + Gb[l][3] * M[l][2] + Gb[l][4] * Vl;
#pragma unroll
    for (int d = 0; d < 3; ++d) ub[d] += Vb * M[l][d];
  }
  Ub[4] += gm1 * pb;
  const double q2 = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
#pragma unroll
  for (int d = 0; d < 3; ++d) Ub[1 + d] += ub[d] * rinv - gm1 * u[d] * pb;
  Ub[0] += 0.5 * gm1 * q2 * pb - (ub[0] * u[0] + ub[1] * u[1] + ub[2] * u[2]) * rinv;
}


}  // namespace
}  // namespace dgk
