// Reverse-mode (vector-Jacobian) derivatives of the pointwise pieces of the
// DGSEM operator (GALAEXI Sec. 3.1, Eqs. 1-3), written by hand from the
// forward formulas in dg_physics.cuh / dg_stage.cuh.  FP64.  Branches follow
// the primal values (the log-mean series/log switch as in the forward); at the
// kinks of the LLF speed max(|u.n| + c) -- a tie, or u.n = 0, to within 1e-12
// of the local scale -- the derivative is the mean of the one-sided ones.
#pragma once

#include "dg_physics.cuh"

namespace dg {

// The FP64 pipe bounds the point-wise adjoints (k_adj_face 81 % busy, one FP64
// instruction per warp in 68 cycles), so they are written for few FP64
// operations: reciprocals by rcp.approx and one cubic step, primitive adjoints
// collected over all terms and directions before one prim_vjp, one viscous
// VJP for a node's three directions.  One VJP of R(U), 16^3 elements: N = 5
// 2124 -> 1584 us, N = 7 5666 -> 4571 us, Gauss nodes N = 3 859 -> 696 us.
// 1/x for the adjoint's positive operands (densities, pressures, beta sums,
// log means): hardware approximation and one cubic Newton-Raphson step
// (below 1 ulp), a fraction of an IEEE division on GB300's narrow FP64 pipe.
__device__ __forceinline__ double adj_rcp(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

// Primitive adjoints (rho, u, v, w, p) -> conserved adjoints.
// rho = q0, u_a = q_{1+a}/rho, p = (gamma-1)(q4 - |q_{1:3}|^2 / (2 rho));
// ir = 1/rho and the velocity come from the caller.
__device__ __forceinline__ void prim_vjp(double ir, double u0, double u1, double u2, double rb, const double ub[3],
                                         double pb, double gm1, double qb[5]) {
  const double k = 0.5 * (u0 * u0 + u1 * u1 + u2 * u2);
  const double gp = gm1 * pb;
  qb[0] += rb - (ub[0] * u0 + ub[1] * u1 + ub[2] * u2) * ir + gp * k;
  qb[1] += ub[0] * ir - gp * u0;
  qb[2] += ub[1] * ir - gp * u1;
  qb[3] += ub[2] * ir - gp * u2;
  qb[4] += gp;
}

// Logarithmic mean and its partial derivatives, consistent with log_mean():
// series branch L = s G(u), G = 1/F2, F2 = 2 (1 + u/3 + u^2/5 + u^3/7),
// u = f^2, f = (a-b)/s; with du/da = 4 f b / s^2 and du/db = -4 f a / s^2,
// dL/da = G + c b and dL/db = G - c a, c = 4 G'(u) f / s = -4 F2'(u) G^2 f / s;
// logarithmic branch L = (a - b) / ln(a/b) with dL/da = (1 - L/a)/ln(a/b),
// dL/db = (L/b - 1)/ln(a/b).
__device__ __forceinline__ double log_mean_d(double a, double b, double& La, double& Lb) {
  const double s = a + b;
  const double is = adj_rcp(s);
  const double f = (a - b) * is;
  const double u = f * f;
  if (u < 1e-4) {
    const double F2 = fma(u, fma(u, fma(u, 2.0 / 7.0, 2.0 / 5.0), 2.0 / 3.0), 2.0);
    const double F2p_m4 = fma(u, fma(u, -24.0 / 7.0, -16.0 / 5.0), -8.0 / 3.0);   // -4 F2'(u)
    const double G = adj_rcp(F2);
    const double c = F2p_m4 * (G * G) * (f * is);
    La = fma(c, b, G);
    Lb = fma(-c, a, G);
    return s * G;
  }
  const double z = a / b;
  const double F = log(z) / (2.0 * ((z - 1.0) / (z + 1.0)));
  const double L = s / (2.0 * F);
  const double ell = log(z);
  La = (1.0 - L / a) / ell;
  Lb = (L / b - 1.0) / ell;
  return L;
}

// Adjoint of the Chandrashekar two-point flux f(a, b; n) (ec_flux): given
// fb = df-bar (5), adds to the primitive adjoints (rho, u, v, w, p) of a and b.
// hipA, hipB are 1/(2p), bipA, bipB are beta/p and kA, kB are |u|^2 of the two
// states (per node, so the volume kernel computes them once per node, not once
// per pair; the p members of A and B are not read).
__device__ __forceinline__ void ec_flux_vjp(const NodePrim<double>& A, const NodePrim<double>& B, double nx,
                                            double ny, double nz, double inv_gm1, const double fb[5], double pa[5],
                                            double pbv[5], double hipA, double hipB, double bipA, double bipB,
                                            double kA, double kB) {
  double Lra, Lrb, Lba, Lbb;
  const double rho_ln = log_mean_d(A.rho, B.rho, Lra, Lrb);
  const double beta_ln = log_mean_d(A.beta, B.beta, Lba, Lbb);
  const double ua = 0.5 * (A.u + B.u), va = 0.5 * (A.v + B.v), wa = 0.5 * (A.w + B.w);
  const double sr = A.rho + B.rho, sb = A.beta + B.beta;
  const double isb = adj_rcp(sb), ibl = adj_rcp(beta_ln);
  const double p_hat = 0.5 * sr * isb;
  const double K = 0.25 * (kA + kB);
  const double un = ua * nx + va * ny + wa * nz;
  const double f0 = rho_ln * un;
  const double fm0 = f0 * ua + p_hat * nx, fm1 = f0 * va + p_hat * ny, fm2 = f0 * wa + p_hat * nz;
  const double H = 0.5 * inv_gm1 * ibl - K;
  // f4 = f0 H + ubar . fm
  const double fmb0 = fb[1] + fb[4] * ua, fmb1 = fb[2] + fb[4] * va, fmb2 = fb[3] + fb[4] * wa;
  double ubb0 = fb[4] * fm0 + f0 * fmb0;
  double ubb1 = fb[4] * fm1 + f0 * fmb1;
  double ubb2 = fb[4] * fm2 + f0 * fmb2;
  const double f0b = fb[0] + fb[4] * H + fmb0 * ua + fmb1 * va + fmb2 * wa;
  const double Hb = fb[4] * f0;
  const double phb = fmb0 * nx + fmb1 * ny + fmb2 * nz;
  const double rlb = f0b * un;
  const double unb = f0b * rho_ln;
  ubb0 += unb * nx; ubb1 += unb * ny; ubb2 += unb * nz;
  const double blb = -Hb * 0.5 * inv_gm1 * (ibl * ibl);
  const double Kb = -Hb;
  // ubar = (u_a + u_b)/2, K = (|u_a|^2 + |u_b|^2)/4
  pa[1] += 0.5 * ubb0 + 0.5 * Kb * A.u;  pbv[1] += 0.5 * ubb0 + 0.5 * Kb * B.u;
  pa[2] += 0.5 * ubb1 + 0.5 * Kb * A.v;  pbv[2] += 0.5 * ubb1 + 0.5 * Kb * B.v;
  pa[3] += 0.5 * ubb2 + 0.5 * Kb * A.w;  pbv[3] += 0.5 * ubb2 + 0.5 * Kb * B.w;
  // p_hat = sr / (2 sb)
  const double srb = phb * 0.5 * isb;
  const double sbb = -phb * p_hat * isb;
  double rab = srb + rlb * Lra, rbb = srb + rlb * Lrb;
  const double bab = sbb + blb * Lba, bbb = sbb + blb * Lbb;
  // beta = rho / (2 p): d beta / d rho = 1/(2p), d beta / d p = -beta/p
  rab = fma(bab, hipA, rab);  pa[4] = fma(-bab, bipA, pa[4]);
  rbb = fma(bbb, hipB, rbb);  pbv[4] = fma(-bbb, bipB, pbv[4]);
  pa[0] += rab;
  pbv[0] += rbb;
}

__device__ __forceinline__ void ec_flux_vjp(const NodePrim<double>& A, const NodePrim<double>& B, double nx,
                                            double ny, double nz, double inv_gm1, const double fb[5], double pa[5],
                                            double pbv[5]) {
  const double ipA = adj_rcp(A.p), ipB = adj_rcp(B.p);
  ec_flux_vjp(A, B, nx, ny, nz, inv_gm1, fb, pa, pbv, 0.5 * ipA, 0.5 * ipB, A.beta * ipA, B.beta * ipB,
              A.u * A.u + A.v * A.v + A.w * A.w, B.u * B.u + B.v * B.v + B.w * B.w);
}

// Adjoint of the Euler flux f(q) . n (q conserved, n any vector): adds the
// direct dependence on the conserved variables to qb and that through the
// velocity and the pressure to ub and pb (one prim_vjp for all directions).
__device__ __forceinline__ void euler_flux_vjp(const double q[5], double u, double v, double w, double p, double nx,
                                               double ny, double nz, const double fb[5], double qb[5], double ub[3],
                                               double& pb) {
  const double un = u * nx + v * ny + w * nz;
  // f0 = m . n, f_m = m un + p n, f_E = (E + p) un
  qb[1] += fb[0] * nx + fb[1] * un;
  qb[2] += fb[0] * ny + fb[2] * un;
  qb[3] += fb[0] * nz + fb[3] * un;
  const double Eb = fb[4] * un;
  qb[4] += Eb;
  const double unb = fb[1] * q[1] + fb[2] * q[2] + fb[3] * q[3] + fb[4] * (q[4] + p);
  pb += fb[1] * nx + fb[2] * ny + fb[3] * nz + Eb;
  ub[0] += unb * nx;
  ub[1] += unb * ny;
  ub[2] += unb * nz;
}

// Adjoint of the local Lax-Friedrichs flux (llf in k_face): adds to the direct
// conserved adjoints qb and the primitive adjoints (rb, ub, pb) of both sides;
// irL, uL, pL (and R) are 1/rho, the velocity and the pressure of the sides.
__device__ __forceinline__ void llf_vjp(const double qL[5], const double qR[5], double irL, const double uL[3], double pL,
                                        double irR, const double uR[3], double pR, double nx, double ny, double nz,
                                        double gamma, const double fb[5], double qbL[5], double qbR[5], double& rbL,
                                        double ubL[3], double& pbL, double& rbR, double ubR[3], double& pbR) {
  const double cL = sqrt(gamma * pL * irL), cR = sqrt(gamma * pR * irR);
  const double unL = uL[0] * nx + uL[1] * ny + uL[2] * nz, unR = uR[0] * nx + uR[1] * ny + uR[2] * nz;
  const double lL = fabs(unL) + cL, lR = fabs(unR) + cR;
  const bool right = lR > lL;
  const double lmax = right ? lR : lL;
  double half[5];
#pragma unroll
  for (int c = 0; c < 5; ++c) half[c] = 0.5 * fb[c];
  euler_flux_vjp(qL, uL[0], uL[1], uL[2], pL, nx, ny, nz, half, qbL, ubL, pbL);
  euler_flux_vjp(qR, uR[0], uR[1], uR[2], pR, nx, ny, nz, half, qbR, ubR, pbR);
  double lb = 0.0;
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    const double lf = lmax * half[c];
    qbR[c] -= lf;
    qbL[c] += lf;
    lb -= half[c] * (qR[c] - qL[c]);
  }
  // lambda = |u . n| + c of the chosen side; c = sqrt(gamma p / rho):
  // dc = c/2 (dp/p - drho/rho).  At the kinks (a tie of the two speeds, or
  // u . n = 0, to within 1e-12 of the local scale, as on symmetry planes) the
  // derivative is the mean of the one-sided derivatives.
  const bool tie = fabs(lR - lL) <= 1e-12 * fmax(lL, lR);
  const double sideL = tie ? 0.5 : (right ? 0.0 : 1.0), sideR = tie ? 0.5 : (right ? 1.0 : 0.0);
  auto speed = [&](double side, double un, double c, double ir, double p, double& rb, double ub[3], double& pb) {
    const double lbw = lb * side;
    const double sg = fabs(un) <= 1e-12 * c ? 0.0 : (un < 0.0 ? -1.0 : 1.0);
    const double ls = lbw * sg, hc = 0.5 * lbw * c;
    ub[0] += ls * nx;
    ub[1] += ls * ny;
    ub[2] += ls * nz;
    rb -= hc * ir;
    pb += hc * adj_rcp(p);
  };
  speed(sideL, unL, cL, irL, pL, rbL, ubL, pbL);
  speed(sideR, unR, cR, irR, pR, rbR, ubR, pbR);
}

// Forward-mode dual number (value, one directional derivative) to
// differentiate the Roe flux mechanically: the templated forward flux runs on
// it.  Kinks follow the value as in the oracle's dual numbers: |x| by the sign
// of the value (derivative +1 at 0), max ties to its first argument.  In a
// namespace of its own, found by argument-dependent lookup, so that sqrt,
// fabs and fmax of doubles keep their meaning everywhere else.
namespace ad {
struct Dual {
  double v, d;
  __device__ Dual() : v(0.0), d(0.0) {}
  __device__ Dual(double x) : v(x), d(0.0) {}
  __device__ Dual(double x, double dx) : v(x), d(dx) {}
};
__device__ __forceinline__ Dual operator+(Dual a, Dual b) { return Dual(a.v + b.v, a.d + b.d); }
__device__ __forceinline__ Dual operator-(Dual a, Dual b) { return Dual(a.v - b.v, a.d - b.d); }
__device__ __forceinline__ Dual operator-(Dual a) { return Dual(-a.v, -a.d); }
__device__ __forceinline__ Dual operator*(Dual a, Dual b) { return Dual(a.v * b.v, fma(a.d, b.v, a.v * b.d)); }
__device__ __forceinline__ Dual operator/(Dual a, Dual b) {
  const double q = a.v / b.v;
  return Dual(q, (a.d - q * b.d) / b.v);
}
__device__ __forceinline__ bool operator<(Dual a, Dual b) { return a.v < b.v; }
__device__ __forceinline__ bool operator>(Dual a, Dual b) { return a.v > b.v; }
__device__ __forceinline__ Dual sqrt(Dual a) {
  const double s = ::sqrt(a.v);
  return Dual(s, a.d / (2.0 * s));
}
__device__ __forceinline__ Dual fabs(Dual a) { return a.v < 0.0 ? -a : a; }
__device__ __forceinline__ Dual fmax(Dual a, Dual b) { return b.v > a.v ? b : a; }
}  // namespace ad

// Adjoint of the Roe flux with the Harten-Hyman entropy fix (roe_flux, FP64,
// no pressure offset) w.r.t. both conserved states: ten forward passes on
// dual numbers, one per input component, each contracted with fb.
static __device__ __noinline__ void roe_vjp(const double qL[5], const double qR[5], double nx, double ny, double nz,
                                     double gamma, double gm1, const double fb[5], double qbL[5], double qbR[5]) {
  using ad::Dual;
#pragma unroll 1
  for (int k = 0; k < 10; ++k) {
    Dual a[5], b[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      a[v] = Dual(qL[v], k == v ? 1.0 : 0.0);
      b[v] = Dual(qR[v], k == 5 + v ? 1.0 : 0.0);
    }
    const Dual irL = Dual(1.0) / a[0], irR = Dual(1.0) / b[0];
    const Dual uL = a[1] * irL, vL = a[2] * irL, wL = a[3] * irL;
    const Dual uR = b[1] * irR, vR = b[2] * irR, wR = b[3] * irR;
    const Dual pL = Dual(gm1) * (a[4] - Dual(0.5) * (a[1] * uL + a[2] * vL + a[3] * wL));
    const Dual pR = Dual(gm1) * (b[4] - Dual(0.5) * (b[1] * uR + b[2] * vR + b[3] * wR));
    Dual F[5];
    roe_flux<Dual>(a, uL, vL, wL, pL, b, uR, vR, wR, pR, Dual(nx), Dual(ny), Dual(nz), Dual(gamma), Dual(gm1), F, pL,
                   pR, b[0] - a[0]);
    double s = 0.0;
#pragma unroll
    for (int v = 0; v < 5; ++v) s = fma(fb[v], F[v].d, s);
    if (k < 5) qbL[k] += s;
    else qbR[k - 5] += s;
  }
}

// Viscosity factor s(T) = mu(T)/mu_ref and ds/dT: Sutherland's law
// s = x^(3/2) (T_ref + S)/(T + S), x = T/T_ref, so ds/dT = s (3/(2T) - 1/(T + S));
// s = 1, ds = 0 for constant viscosity.
__device__ __forceinline__ void visc_factor_d(const Gas& g, double T, double& s, double& ds) {
  if (g.visc_law != DG_VISC_SUTHERLAND) {
    s = 1.0;
    ds = 0.0;
    return;
  }
  const double x = T * g.inv_T_ref, den = 1.0 / (T + g.S_suth);
  s = x * sqrt(x) * g.suth_c * den;
  ds = s * (1.5 / T - den);
}

// Adjoint of the viscous fluxes f_v . n^d of one state over several directions
// n^d, given the adjoints fb^d (4): with A^d = fb^d_m + fb^d_E u, M = sum_d A^d
// (x) n^d and Q = sum_d fb^d_E n^d carry all of it, so the stress is formed once.
struct ViscVjp {
  double M[9], Q[3];
};
__device__ __forceinline__ void visc_vjp_add(ViscVjp& s, double u, double v, double w, double nx, double ny, double nz,
                                             const double fb[4]) {
  const double A[3] = {fma(fb[3], u, fb[0]), fma(fb[3], v, fb[1]), fma(fb[3], w, fb[2])};
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    s.M[a * 3] = fma(A[a], nx, s.M[a * 3]);
    s.M[a * 3 + 1] = fma(A[a], ny, s.M[a * 3 + 1]);
    s.M[a * 3 + 2] = fma(A[a], nz, s.M[a * 3 + 2]);
  }
  s.Q[0] = fma(fb[3], nx, s.Q[0]);
  s.Q[1] = fma(fb[3], ny, s.Q[1]);
  s.Q[2] = fma(fb[3], nz, s.Q[2]);
}
// The adjoints of the gradients (gb, 12, set) and the velocity (added to ub);
// returns sum_d fb^d . f_v1^d, f_v1 the flux with unit viscosity (f_v = mu f_v1
// is linear in mu: the return value is the derivative by mu, and with
// Sutherland's law the caller scales it by s(T) and, for the T-derivative, by
// mu_ref ds/dT).
__device__ __forceinline__ double visc_vjp_end(const ViscVjp& s, const double g[12], double mu, double kappa,
                                               double gb[12], double ub[3]) {
  const double div = (2.0 / 3.0) * (g[0] + g[4] + g[8]);
  const double t00 = 2.0 * g[0] - div, t11 = 2.0 * g[4] - div, t22 = 2.0 * g[8] - div;
  const double t01 = g[1] + g[3], t02 = g[2] + g[6], t12 = g[5] + g[7];
  const double* M = s.M;
  const double* Q = s.Q;
  ub[0] += mu * (t00 * Q[0] + t01 * Q[1] + t02 * Q[2]);
  ub[1] += mu * (t01 * Q[0] + t11 * Q[1] + t12 * Q[2]);
  ub[2] += mu * (t02 * Q[0] + t12 * Q[1] + t22 * Q[2]);
  // tau_aa = mu (2 g_aa - 2/3 div), tau_ab = mu (g_ab + g_ba)
  const double m01 = M[1] + M[3], m02 = M[2] + M[6], m12 = M[5] + M[7], m2 = 2.0 * mu;
  const double divb = -(2.0 / 3.0) * mu * (M[0] + M[4] + M[8]);
  gb[0] = fma(m2, M[0], divb);
  gb[4] = fma(m2, M[4], divb);
  gb[8] = fma(m2, M[8], divb);
  gb[1] = gb[3] = mu * m01;
  gb[2] = gb[6] = mu * m02;
  gb[5] = gb[7] = mu * m12;
  const double km = kappa * mu;
  gb[9] = km * Q[0];
  gb[10] = km * Q[1];
  gb[11] = km * Q[2];
  return t00 * M[0] + t11 * M[4] + t22 * M[8] + t01 * m01 + t02 * m02 + t12 * m12 +
         kappa * (g[9] * Q[0] + g[10] * Q[1] + g[11] * Q[2]);
}

}  // namespace dg
