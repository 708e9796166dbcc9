// Face flux of the FP64 operator with its viscous part in block fixed point
// (dg_fixed.cuh): the terms of face_flux_core<double>, the exponents taken per
// face point from both sides' data.  The Riemann flux stays FP64 (about 90
// operations; the viscous part took as many and is now integer work beside it).
//
// Bound and measured: the FP64 pipe, as before, with half the instructions.  128
// threads, 168 registers; five or six blocks per SM (with fewer registers) took 1
// to 9 % longer.  Manufactured solution, 16^3 elements, LLF, us per launch before
// -> now: N = 1 24 -> 18, 3 73 -> 50, 5 147 -> 93, 7 257 -> 150, 9 397 -> 225.
#pragma once

#include "dg_fx_metrics.cuh"
#include "dg_stage.cuh"

namespace dg {

// Sound speed sqrt(x).  For positive normal x: c = x y from the hardware's
// approximation y of 1/sqrt(x) (2^-20), corrected to third order from the exact
// residual x - c^2, sqrt(x) = c + (x - c^2) y/2 (1 + 3/4 e), e = 1 - c y; within 0.55
// ulp, 6 FP64 operations.  Zero, subnormal, infinite and negative values (a gas
// without pressure has c = 0, while y would be infinite) take sqrt().
__device__ __forceinline__ double sqrt_op(double x) {
  if ((unsigned)__double2hiint(x) - 0x00100000u >= 0x7fe00000u) return sqrt(x);
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double c = x * y, half = __hiloint2double(__double2hiint(y) - 0x00100000, __double2loint(y));
  return fma(fma(-c, c, x) * half, fma(0.75, fma(-c, y, 1.0), 1.0), c);
}

// Sum of the NS sides' viscous fluxes . n over mu, momentum (w[0..2]) and energy
// (w[3]); with NS = 1 of the left side alone.
// False: a non-finite value or an exponent out of range; w is not set.
template <int NS = 2>
__device__ __forceinline__ bool face_visc_fx(const double* __restrict__ gL, const double* __restrict__ gR, size_t stride,
                                             double sfL, double sfR, bool scaled, const double uL[3], const double uR[3],
                                             const double nv[3], double kappa, double w[4]) {
  double g[NS][9], t[NS][3];
#pragma unroll
  for (int r = 0; r < 9; ++r) {
    g[0][r] = gL[r * stride];
    if constexpr (NS == 2) g[1][r] = gR[r * stride];
  }
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    t[0][l] = gL[(9 + l) * stride];
    if constexpr (NS == 2) t[1][l] = gR[(9 + l) * stride];
  }
  if (scaled) {
#pragma unroll
    for (int r = 0; r < 9; ++r) {
      g[0][r] *= sfL;
      if constexpr (NS == 2) g[1][r] *= sfR;
    }
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      t[0][l] *= sfL;
      if constexpr (NS == 2) t[1][l] *= sfR;
    }
  }
  auto mag = [](double x) { return __double2hiint(x) & 0x7fffffff; };
  int mg = 0, mt = 0, mu = 0;
#pragma unroll
  for (int s = 0; s < NS; ++s) {
#pragma unroll
    for (int r = 0; r < 9; ++r) mg = max(mg, mag(g[s][r]));
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      mt = max(mt, mag(t[s][l]));
      mu = max(mu, mag(s ? uR[l] : uL[l]));
    }
  }
  if (!(fx_in_range(mg, 90) & fx_in_range(mt, 90) & fx_in_range(mu, 90))) return false;
  const int eg = fx_expo(mg), et = fx_expo(mt), eu = fx_expo(mu);
  Fx n[3];
#pragma unroll
  for (int l = 0; l < 3; ++l) n[l] = fx_split(fx_from(nv[l], 60));
  const Fx twothird{715827883, -1431655765};   // 2^62 2/3
  i64 v[3] = {0, 0, 0}, en = 0;
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    i64 G[9];
#pragma unroll
    for (int r = 0; r < 9; ++r) G[r] = fx_from(g[s][r], 59 - eg);
    const i64 div = fx_mul<2>(fx_split(G[0] + G[4] + G[8]), twothird);
    const Fx t00 = fx_split(2 * G[0] - div), t11 = fx_split(2 * G[4] - div), t22 = fx_split(2 * G[8] - div);   // < 2^60.4
    const Fx t01 = fx_split(G[1] + G[3]), t02 = fx_split(G[2] + G[6]), t12 = fx_split(G[5] + G[7]);
    FxSum f0 = fx_zero<2>(), f1 = fx_zero<2>(), f2 = fx_zero<2>(), fe = fx_zero<2>();
    fx_add(f0, t00, n[0]); fx_add(f0, t01, n[1]); fx_add(f0, t02, n[2]);
    fx_add(f1, t01, n[0]); fx_add(f1, t11, n[1]); fx_add(f1, t12, n[2]);
    fx_add(f2, t02, n[0]); fx_add(f2, t12, n[1]); fx_add(f2, t22, n[2]);
    const i64 a0 = fx_end<2>(f0), a1 = fx_end<2>(f1), a2 = fx_end<2>(f2);   // 57 - e_g, < 2^59.2
    const double* us = s ? uR : uL;
    fx_add(fe, fx_split(a0), fx_split(fx_from(us[0], 60 - eu)));
    fx_add(fe, fx_split(a1), fx_split(fx_from(us[1], 60 - eu)));
    fx_add(fe, fx_split(a2), fx_split(fx_from(us[2], 60 - eu)));
    v[0] += a0; v[1] += a1; v[2] += a2;
    en += fx_end<2>(fe);                                                     // 55 - e_g - e_u
  }
  FxSum h = fx_zero<2>();
#pragma unroll
  for (int l = 0; l < 3; ++l)
    fx_add(h, fx_split(fx_from(t[0][l], 59 - et) + (NS == 2 ? fx_from(t[NS - 1][l], 59 - et) : 0)), n[l]);
#pragma unroll
  for (int c = 0; c < 3; ++c) w[c] = fx_to(v[c], 57 - eg);
  w[3] = fma(kappa, fx_to(fx_end<2>(h), 57 - et), fx_to(en, 55 - eg - eu));
  return true;
}

// LLF flux of one face point in FP64 with the viscous part above: states qL, qR,
// lifted gradients gL, gR (components `stride` apart), unit normal nv of the
// master side, surface element sJ; F* (5 values, fstride apart) to fo.
__device__ __forceinline__ void face_point_fx(const double qL[5], const double qR[5], const double* __restrict__ gL,
                                              const double* __restrict__ gR, size_t stride, const double nv[3], double sJ,
                                              const Gas& g, double* __restrict__ fo, size_t fstride) {
  const double irL = rcp_op(qL[0]), irR = rcp_op(qR[0]);
  const double uL[3] = {qL[1] * irL, qL[2] * irL, qL[3] * irL}, uR[3] = {qR[1] * irR, qR[2] * irR, qR[3] * irR};
  const double pL = g.gm1 * (qL[4] - 0.5 * (qL[1] * uL[0] + qL[2] * uL[1] + qL[3] * uL[2]));
  const double pR = g.gm1 * (qR[4] - 0.5 * (qR[1] * uR[0] + qR[2] * uR[1] + qR[3] * uR[2]));
  const bool suth = g.visc_law == DG_VISC_SUTHERLAND;
  double sfL = 1, sfR = 1;
  if (suth) {
    sfL = visc_factor<double>(g, pL * irL * g.inv_R);
    sfR = visc_factor<double>(g, pR * irR * g.inv_R);
  }
  double w[4];
  if (!face_visc_fx(gL, gR, stride, sfL, sfR, suth, uL, uR, nv, g.kappa, w)) {
    double a[12], b[12], vL[4], vR[4];
#pragma unroll
    for (int r = 0; r < 12; ++r) {
      a[r] = gL[r * stride];
      b[r] = gR[r * stride];
    }
    visc_flux<double>(a, uL[0], uL[1], uL[2], sfL, g.kappa * sfL, nv[0], nv[1], nv[2], vL);
    visc_flux<double>(b, uR[0], uR[1], uR[2], sfR, g.kappa * sfR, nv[0], nv[1], nv[2], vR);
#pragma unroll
    for (int c = 0; c < 4; ++c) w[c] = vL[c] + vR[c];
  }
  // 2 F = f(q_L) + f(q_R) - lambda (q_R - q_L) - (f_v,L + f_v,R), each . n
  const double nL = uL[0] * nv[0] + uL[1] * nv[1] + uL[2] * nv[2], nR = uR[0] * nv[0] + uR[1] * nv[1] + uR[2] * nv[2];
  const double lL = fabs(nL) + sqrt_op(g.gamma * pL * irL), lR = fabs(nR) + sqrt_op(g.gamma * pR * irR);
  const double lam = lR > lL ? lR : lL, ps = pL + pR, half = 0.5 * sJ;
  fo[0] = half * fma(-lam, qR[0] - qL[0], fma(qL[0], nL, qR[0] * nR));
#pragma unroll
  for (int c = 0; c < 3; ++c)
    fo[(c + 1) * fstride] =
        half * fma(-g.mu, w[c], fma(-lam, qR[c + 1] - qL[c + 1], fma(qL[c + 1], nL, fma(qR[c + 1], nR, ps * nv[c]))));
  fo[4 * fstride] = half * fma(-g.mu, w[3], fma(-lam, qR[4] - qL[4], fma(qL[4] + pL, nL, (qR[4] + pR) * nR)));
}

template <int N>
__device__ __forceinline__ void face_body_fx(const double* __restrict__ U, const double* __restrict__ grad,
                                             const FaceInfo* __restrict__ faces, const double* __restrict__ facegeo,
                                             double* __restrict__ fstar, int F, int E, const Gas& g, long gid) {
  constexpr int n = N + 1, P = n * n * n, NN = n * n;
  if (g.surf_flux != DG_FLUX_LLF) {   // the EC and Roe fluxes: all FP64
    face_body<N, double>(U, grad, faces, facegeo, fstar, F, E, g, gid);
    return;
  }
  if (gid >= (long)F * NN) return;
  const int f = (int)(gid / NN), pq = (int)(gid % NN);
  const int p = pq % n, q = pq / n;
  const FaceInfo fi = faces[f];
  const int eM = dg_idx(fi.master >> 3, E, kSiteFaceElems), fM = fi.master & 7;
  const int eS = dg_idx(fi.slave >> 3, E, kSiteFaceElems), fS = fi.slave & 7;
  int p2, q2;
  apply_flip<n>(fi.flip, p, q, p2, q2);
  const int idM = face_node<n>(fM, p, q), idS = face_node<n>(fS, p2, q2);
  double qL[5], qR[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    qL[v] = U[((size_t)eM * 5 + v) * P + idM];
    qR[v] = U[((size_t)eS * 5 + v) * P + idS];
  }
  const double* fg = facegeo + (size_t)f * 4 * NN + pq;
  const double nv[3] = {fg[0], fg[NN], fg[2 * NN]}, sJ = fg[3 * NN];
  face_point_fx(qL, qR, grad + (size_t)eM * 12 * P + idM, grad + (size_t)eS * 12 * P + idS, P, nv, sJ, g,
                fstar + (size_t)f * 5 * NN + pq, NN);
}

}  // namespace dg
