// Weak lifting and weak volume term on Gauss nodes in block fixed point
// (dg_fixed.cuh), the terms of lift_lg_body and volume_lg_body<double>.
// Primitives, the source and the Runge-Kutta update stay FP64; elements out of
// range (state 2) are left to the FP64 bodies, which run after these.
//
// Bound and measured: the FP64 kernels held the FP64 pipe 87 to 92 % busy (421
// FP64 instructions a node in the lifting at N = 3, 233 in the volume kernel).
// Now the lifting's 156 multiply-adds a node and direction (12 cycles each on
// the quarter-rate integer multiplier; ALU and multiplier 56 and 50 % busy at N
// = 3) and the volume kernel's remaining FP64 work and loads hold them.
// Manufactured solution, 16^3 elements, us per launch before -> now: lifting
// with prolongation N = 3 226 -> 119, 5 792 -> 356, 7 1985 -> 900; volume N = 3
// 134 -> 74, 5 466 -> 199, 7 1225 -> 500.
#pragma once

#include "dg_fx_metrics.cuh"
#include "dg_gauss.cuh"

namespace dg {

// |D^w|, l(+-1)/w < 2^e per degree: at most 1.37, 2.66, 4.39, 6.55, 9.14, 12.2,
// 15.7, 19.6, 23.9.  l(+-1) itself is below 2.
constexpr int fx_eDw(int N) { return N == 1 ? 1 : (N == 2 ? 2 : (N <= 4 ? 3 : (N <= 7 ? 4 : 5))); }

template <int N, int EPB>
constexpr size_t lift_lg_fx_smem() {
  constexpr int n = N + 1, P = n * n * n, NN = n * n;
  return 8 * (((n * n + 4 * n + 1) & ~1) + (size_t)EPB * (12 * P + 72 * NN));
}

// Returns whether the block holds elements left to FP64 (state[le] = 2).
// STRETCH (both kernels): the mesh may hold elements with shifted metric terms
// (FxMetricShifts); without it every shift is 0.
template <int N, int EPB, bool MORTAR, bool STRETCH>
__device__ __forceinline__ bool lift_lg_fx(const double* __restrict__ U, const double* __restrict__ Uf,
                                           const i64* __restrict__ jx, const float4* __restrict__ ejx,
                                           const double* __restrict__ facegeo, const int* __restrict__ elem_face,
                                           const int* __restrict__ elem_nbr, const double* __restrict__ tab,
                                           double* __restrict__ grad, double* __restrict__ gf, int E, int F, const Gas& g,
                                           const double* __restrict__ mvirt, int n_mortar, int* state) {
  using S = Shape<N, EPB>;
  constexpr int n = S::n, P = S::P, NN = n * n, PER = 12 * P + 72 * NN, eD = fx_eDw(N);
  extern __shared__ __align__(16) unsigned char lift_lg_raw[];
  Fx* sDw = reinterpret_cast<Fx*>(lift_lg_raw);   // weak D and l(+-1)/w: 60 - e_D bits
  Fx* sT = sDw + n * n;                            // [2][n] l(+-1)/w, [2][n] l(+-1): 59 bits
  i64* const tile0 = reinterpret_cast<i64*>(lift_lg_raw) + ((n * n + 4 * n + 1) & ~1);
  __shared__ int s_mx[EPB][2];                     // velocity, temperature
  const int le = threadIdx.x / P, id = threadIdx.x - le * P;
  const int e = blockIdx.x * EPB + le;
  const bool active = e < E;
  i64* sprod = tile0 + le * PER;                   // [12][P]
  i64* sS = sprod + 12 * P;                        // [6][12][NN]
  for (int t = threadIdx.x; t < n * n; t += blockDim.x) sDw[t] = fx_split(fx_round(tab[GaussTab::Dw(n) + t], kFxQD - eD));
  for (int t = threadIdx.x; t < 4 * n; t += blockDim.x)
    sT[t] = fx_split(fx_round(tab[GaussTab::lmw(n) + t], t < 2 * n ? kFxQD - eD : 59));
  for (int t = threadIdx.x; t < 2 * EPB; t += blockDim.x) s_mx[t >> 1][t & 1] = 0;
  __syncthreads();
  double ph[4] = {0, 0, 0, 0};
  int m2[2] = {0, 0};
  auto add_max = [&](const double f[4]) {
    m2[0] = max(m2[0], max(max(fx_mag(f[0]), fx_mag(f[1])), fx_mag(f[2])));
    m2[1] = max(m2[1], fx_mag(f[3]));
  };
  if (active) {
    state_phi<double>(U + (size_t)e * 5 * P + id, P, g, ph);
    add_max(ph);
    // face averages and n sJ as FP64, converted below once the range is known
    for (int o = id; o < 6 * NN; o += P) {
      const int f = o / NN, pq = o - f * NN, p = pq % n, q = pq / n;
      const int code = elem_face[e * 6 + f], nb = elem_nbr[e * 6 + f];
      const int fid = dg_idx(code >> 4, F, kSiteGaussLift);
      int p2, q2;
      apply_flip<n>(code & 7, p, q, p2, q2);
      const int pq2 = p2 + n * q2;
      double pm[4], pn[4];
      state_phi<double>(Uf + ((size_t)e * 6 + f) * 5 * NN + pq, NN, g, pm);
      bool done = false;
      if constexpr (MORTAR) {
        if (nb < 0) {
          state_phi<double>(mvirt + (size_t)dg_idx(-1 - nb, 5L * n_mortar, kSiteMortar) * 5 * NN + pq, NN, g, pn);
          done = true;
        }
      }
      if (!done) {
        const int e2 = dg_idx(nb >> 3, E, kSiteGaussLift), f2 = nb & 7;
        state_phi<double>(Uf + ((size_t)e2 * 6 + f2) * 5 * NN + pq2, NN, g, pn);
      }
      const bool master = code & 8;
      const double* fg = facegeo + (size_t)fid * 4 * NN + (master ? pq : pq2);
      const double sJ = master ? fg[3 * NN] : -fg[3 * NN];
      double star[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) star[a] = 0.5 * (pm[a] + pn[a]);
      add_max(star);
      i64* s = sS + f * 12 * NN + pq;
#pragma unroll
      for (int a = 0; a < 4; ++a) s[a * NN] = __double_as_longlong(star[a]);
#pragma unroll
      for (int l = 0; l < 3; ++l) s[(4 + l) * NN] = __double_as_longlong(sJ * fg[l * NN]);
    }
    fx_maxima<2>(le, s_mx[le], m2);
  }
  __syncthreads();
  const int eu = fx_expo(s_mx[le][0]), et = fx_expo(s_mx[le][1]);
  const float4 ej = active ? ejx[e] : make_float4(1000.0f, 0.0f, 0.0f, 0.0f);
  const bool act = active && fx_in_range(s_mx[le][0], 90) && fx_in_range(s_mx[le][1], 90) && ej.x < 90.0f;
  if (id == 0) state[le] = active ? (act ? 1 : 2) : 0;
  i64 Ja[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0}, iJ = 0;
  Fx X[4];
  const FxMetricShifts sh{STRETCH ? __float_as_int(ej.w) : 0};
  if (act) {
    const i64* mt = jx + (size_t)e * 10 * P + id;
#pragma unroll
    for (int r = 0; r < 9; ++r) Ja[r] = fx_up(mt[r * P], sh.c(r % 3));
    iJ = mt[9 * P];
#pragma unroll
    for (int a = 0; a < 4; ++a) X[a] = fx_split(fx_from(ph[a], 62 - (a < 3 ? eu : et)));
    for (int o = id; o < 6 * NN; o += P) {
      const int f = o / NN, pq = o - f * NN;
      i64* s = sS + f * 12 * NN + pq;
      Fx st[4], ns[3];
#pragma unroll
      for (int a = 0; a < 4; ++a) st[a] = fx_split(fx_from(__longlong_as_double(s[a * NN]), 62 - (a < 3 ? eu : et)));
#pragma unroll
      for (int l = 0; l < 3; ++l) ns[l] = fx_split(fx_from(__longlong_as_double(s[(4 + l) * NN]), kFxQ - (int)ej.x + sh.c(l)));
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int l = 0; l < 3; ++l) s[(a * 3 + l) * NN] = fx_mul<2>(st[a], ns[l]);   // 60 - e - e_j + c_l
    }
  }
  const int i = id % n, j = (id / n) % n, k = id / NN;
  i64 acc[12] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0};   // 59 - e - e_j + c_l - e_D, below 2^62
#pragma unroll 1
  for (int d = 0; d < 3; ++d) {
    __syncthreads();
    if (act) {
      const Fx J0 = fx_split(d == 0 ? Ja[0] : (d == 1 ? Ja[3] : Ja[6])), J1 = fx_split(d == 0 ? Ja[1] : (d == 1 ? Ja[4] : Ja[7])),
               J2 = fx_split(d == 0 ? Ja[2] : (d == 1 ? Ja[5] : Ja[8]));
#pragma unroll
      for (int a = 0; a < 4; ++a) {   // negated: the volume term enters with a minus sign
        sprod[(a * 3) * P + id] = -fx_mul<2>(X[a], J0);
        sprod[(a * 3 + 1) * P + id] = -fx_mul<2>(X[a], J1);
        sprod[(a * 3 + 2) * P + id] = -fx_mul<2>(X[a], J2);
      }
    }
    __syncthreads();
    if (act) {
      const int r = d == 0 ? i : (d == 1 ? j : k);
      const int stride = d == 0 ? 1 : (d == 1 ? n : NN);
      const int line0 = id - r * stride, pq = d == 0 ? j + n * k : (d == 1 ? i + n * k : i + n * j);
      const Fx* Dr = sDw + r * n;
      const Fx t0 = sT[r], t1 = sT[n + r];
      const i64* f0 = sS + (2 * d) * 12 * NN + pq;
#pragma unroll
      for (int al = 0; al < 12; ++al) {
        FxSum s = fx_zero<kFxUpWeak>();
        const i64* line = sprod + al * P + line0;
#pragma unroll
        for (int m = 0; m < n; ++m) fx_add(s, Dr[m], fx_split(line[m * stride]));
        fx_add(s, t0, fx_split(f0[al * NN]));
        fx_add(s, t1, fx_split(f0[(12 + al) * NN]));
        acc[al] += fx_end<kFxUpWeak>(s);
      }
    }
  }
  __syncthreads();   // every thread is done with sprod
  const int qg = 59 + 62 - 64 + 1 - (int)ej.x - eD - (int)ej.z;   // less e, + c_l
  if (act) {
    double* go = grad + (size_t)e * 12 * P + id;
    const Fx iJx = fx_split(iJ);
#pragma unroll
    for (int al = 0; al < 12; ++al) {
      const i64 G = fx_mul<1>(fx_split(acc[al]), iJx);   // below 2^61
      go[al * P] = fx_to(G, qg + sh.c(al % 3) - (al < 9 ? eu : et));
      sprod[al * P + id] = G;
    }
  }
  __syncthreads();
  int bad = 0;
#pragma unroll
  for (int l = 0; l < EPB; ++l) bad |= state[l] == 2;
  if (!act) return bad;
  for (int o = id; o < 72 * NN; o += P) {
    const int f = o / (12 * NN), r = o - f * 12 * NN, al = r / NN, pq = r - al * NN;
    const int p = pq % n, q = pq / n, d = f >> 1;
    const Fx* l = sT + (2 + (f & 1)) * n;
    const int stride = d == 0 ? 1 : (d == 1 ? n : NN);
    const i64* line = sprod + al * P + line_node<n>(d, 0, p, q);
    FxSum s = fx_zero<4>();
#pragma unroll
    for (int m = 0; m < n; ++m) {
      if (n > 5 && m == n / 2) fx_fold(s);   // five terms fill c
      fx_add(s, l[m], fx_split(line[m * stride]));
    }
    gf[((size_t)e * 6 + f) * 12 * NN + (size_t)al * NN + pq] = fx_to(fx_end<4>(s), qg + sh.c(al % 3) + 59 - 64 + 4 - (al < 9 ? eu : et));
  }
  return bad;
}

template <int N, int EPB>
constexpr size_t volume_lg_fx_smem() {
  constexpr int n = N + 1, P = n * n * n, NN = n * n;
  return 8 * (((n * n + 2 * n + 1) & ~1) + (size_t)EPB * (15 * P + 30 * NN));
}

// Returns whether the block holds elements left to FP64 (state[le] = 2).
template <int N, int EPB, bool LIST, bool STRETCH>
__device__ __forceinline__ bool volume_lg_fx(const StageArgs& a, const double* __restrict__ metrics,
                                             const i64* __restrict__ jx, const float4* __restrict__ ejx,
                                             const double* __restrict__ grad, const double* __restrict__ fstar,
                                             const int* __restrict__ elem_face, const double* __restrict__ mms,
                                             const double* __restrict__ tab, int E, const Gas& g, int* state) {
  using S = Shape<N, EPB>;
  constexpr int n = S::n, P = S::P, NN = n * n, PER = 15 * P + 30 * NN, eD = fx_eDw(N);
  extern __shared__ __align__(16) unsigned char volume_lg_raw[];
  Fx* sDw = reinterpret_cast<Fx*>(volume_lg_raw);   // weak D, [2][n] l(+-1)/w: 60 - e_D bits
  Fx* sT = sDw + n * n;
  i64* const tile0 = reinterpret_cast<i64*>(volume_lg_raw) + ((n * n + 2 * n + 1) & ~1);
  enum { kR, kU, kP, kH, kG, kT, kF0, kFm, kFe, kCount };
  __shared__ int s_mx[EPB][kCount];
  __shared__ double s_tc[2];
  const int le = threadIdx.x / P, id = threadIdx.x - le * P;
  int e = blockIdx.x * EPB + le;
  if constexpr (LIST) {
    const int nslot = *a.list_len;
    e = e < nslot ? a.list[e] : E;
    if constexpr (EPB == 1) {
      if (e >= E) return false;   // the whole block, before any barrier
    }
  }
  const bool active = e < E;
  i64* sF = tile0 + le * PER;   // [3][5][P] contravariant fluxes, negated
  i64* sFs = sF + 15 * P;       // [6][5][NN] outward surface fluxes
  for (int t = threadIdx.x; t < n * n; t += blockDim.x) sDw[t] = fx_split(fx_round(tab[GaussTab::Dw(n) + t], kFxQD - eD));
  for (int t = threadIdx.x; t < 2 * n; t += blockDim.x) sT[t] = fx_split(fx_round(tab[GaussTab::lmw(n) + t], kFxQD - eD));
  for (int t = threadIdx.x; t < EPB * kCount; t += blockDim.x) s_mx[t / kCount][t % kCount] = 0;
  if (threadIdx.x == 0 && g.source == DG_SOURCE_MMS)
    sincospi(a.clock[0] + a.c_stage * a.clock[1], &s_tc[0], &s_tc[1]);
  const FxMetricShifts sh{STRETCH && active ? __float_as_int(ejx[e].w) : 0};
  __syncthreads();
  double q[5] = {1, 0, 0, 0, 0}, gr[12];
  double u = 0, v = 0, w = 0, p = 0;
  if (active) {
#pragma unroll
    for (int c = 0; c < 5; ++c) q[c] = a.U[((size_t)e * 5 + c) * P + id];
#pragma unroll
    for (int r = 0; r < 12; ++r) gr[r] = grad[((size_t)e * 12 + r) * P + id];
    const double ir = rcp_op(q[0]);
    u = q[1] * ir; v = q[2] * ir; w = q[3] * ir;
    p = g.gm1 * (q[4] - 0.5 * (q[1] * u + q[2] * v + q[3] * w));
    if (g.visc_law == DG_VISC_SUTHERLAND) {
      const double sf = visc_factor<double>(g, p * ir * g.inv_R);
#pragma unroll
      for (int r = 0; r < 12; ++r) gr[r] *= sf;
    }
    int m[kCount];
    m[kR] = fx_mag(q[0]);
    m[kU] = max(max(fx_mag(u), fx_mag(v)), fx_mag(w));
    m[kP] = fx_mag(p);
    m[kH] = fx_mag(q[4] + p);
    m[kG] = 0;
#pragma unroll
    for (int r = 0; r < 9; ++r) m[kG] = max(m[kG], fx_mag(gr[r]));
    m[kT] = max(max(fx_mag(gr[9]), fx_mag(gr[10])), fx_mag(gr[11]));
    m[kF0] = m[kFm] = m[kFe] = 0;
    for (int o = id; o < 30 * NN; o += P) {
      const int f = o / (5 * NN), r = o - f * 5 * NN, v2 = r / NN, pq = r - v2 * NN;
      const int code = elem_face[e * 6 + f], fid = dg_idx(code >> 4, a.nfaces > 0 ? a.nfaces : 3L * E, kSiteGaussVol);
      double val;
      if (code & 8) {
        val = fstar[((size_t)fid * 5 + v2) * NN + pq];
      } else {
        int p2, q2;
        apply_flip<n>(code & 7, pq % n, pq / n, p2, q2);
        val = -fstar[((size_t)fid * 5 + v2) * NN + p2 + n * q2];
      }
      sFs[(f * 5 + v2) * NN + pq] = __double_as_longlong(val);
      const int hv = fx_mag(val), mv = hv ? hv + (sh.t(f >> 1) << 20) : 0;   // of val 2^t, as it is held below
      if (v2 == 0) m[kF0] = max(m[kF0], mv);
      else if (v2 == 4) m[kFe] = max(m[kFe], mv);
      else m[kFm] = max(m[kFm], mv);
    }
    fx_maxima<kCount>(le, s_mx[le], m);
  }
  __syncthreads();
  int x[kCount];
  bool in = true;
#pragma unroll
  for (int c = 0; c < kCount; ++c) {
    x[c] = fx_expo(s_mx[le][c]);
    in = in & fx_in_range(s_mx[le][c], 90);
  }
  const int ej = active ? (int)ejx[e].x : 1000, hm = fx_mag(g.mu), hl = fx_mag(g.mu * g.kappa);
  const int em = fx_expo(hm), el = fx_expo(hl);
  const bool act = active & in & (ej < 90) & fx_in_range(hm, 90) & fx_in_range(hl, 90);
  if (id == 0) state[le] = active ? (act ? 1 : 2) : 0;
  // bits after the point of the mass (q0), momentum (qm) and energy (qe) fluxes,
  // + t_d in direction d: below 2^61.3, so that six of a line's n + 2 terms fit in FxSum's c (the part of
  // the products that fx_add leaves out is the sums' largest error, and a bit
  // more in the factors halves it)
  const int n0 = 61 - x[kR] - x[kU] - ej;                                             // rho {u . Ja}
  const int n1 = 61 - x[kR] - 2 * x[kU] - ej, n2 = 60 - x[kP] - ej, n3 = 59 - x[kG] - em - ej;
  const int qm = min(min(n1 - 1, n2), min(n3 - 2, 60 - x[kFm]));
  const int n4 = 60 - x[kH] - x[kU] - ej, n5 = n3 - 2 - x[kU], n6 = 60 - x[kT] - el - ej;
  const int qe = min(min(n4, n5 - 1), min(n6 - 1, 60 - x[kFe]));
  const int q0 = min(n0, 60 - x[kF0]);
  if (act) {
    const Fx U[3] = {fx_split(fx_from(u, 62 - x[kU])), fx_split(fx_from(v, 62 - x[kU])), fx_split(fx_from(w, 62 - x[kU]))};
    const Fx rho = fx_split(fx_from(q[0], 62 - x[kR])), H = fx_split(fx_from(q[4] + p, 62 - x[kH]));
    const Fx Pp = fx_split(fx_from(p, 62 - x[kP]) >> fx_clamp(n2 - qm));
    i64 G[9];
#pragma unroll
    for (int r = 0; r < 9; ++r) G[r] = fx_from(gr[r], 59 - x[kG]);
    const Fx twothird{715827883, -1431655765};   // 2^62 2/3
    const Fx mu = fx_split(fx_from(g.mu, 62 - em)), lam = fx_split(fx_from(g.mu * g.kappa, 62 - el));
    const i64 div = fx_mul<2>(fx_split(G[0] + G[4] + G[8]), twothird);
    // mu (stress): 59 - e_g - e_mu, below 2^60.4; heat flux: 60 - e_t - e_lambda
    auto visc = [&](i64 t) { return fx_split(fx_mul<2>(fx_split(t), mu)); };
    const Fx t00 = visc(2 * G[0] - div), t11 = visc(2 * G[4] - div), t22 = visc(2 * G[8] - div);
    const Fx t01 = visc(G[1] + G[3]), t02 = visc(G[2] + G[6]), t12 = visc(G[5] + G[7]);
    Fx T[3];
#pragma unroll
    for (int l = 0; l < 3; ++l) T[l] = fx_split(fx_mul<2>(fx_split(fx_from(gr[9 + l], 60 - x[kT])), lam));
    const i64* mt = jx + (size_t)e * 10 * P + id;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int t = sh.t(d);
      const Fx J[3] = {fx_split(fx_up(mt[(d * 3) * P], t)), fx_split(fx_up(mt[(d * 3 + 1) * P], t)),
                       fx_split(fx_up(mt[(d * 3 + 2) * P], t))};
      FxSum s = fx_zero<3>();
      fx_add(s, U[0], J[0]); fx_add(s, U[1], J[1]); fx_add(s, U[2], J[2]);
      const Fx un = fx_split(fx_end<3>(s));                 // 61 - e_u - e_j
      const i64 f0 = fx_mul<2>(rho, un);                    // n0
      const Fx X = fx_split(f0 >> fx_clamp(n1 - qm));
      FxSum w0 = fx_zero<4>(), w1 = fx_zero<4>(), w2 = fx_zero<4>();
      fx_add(w0, t00, J[0]); fx_add(w0, t01, J[1]); fx_add(w0, t02, J[2]);
      fx_add(w1, t01, J[0]); fx_add(w1, t11, J[1]); fx_add(w1, t12, J[2]);
      fx_add(w2, t02, J[0]); fx_add(w2, t12, J[1]); fx_add(w2, t22, J[2]);
      const i64 V[3] = {fx_end<4>(w0), fx_end<4>(w1), fx_end<4>(w2)};   // n3
      sF[(d * 5) * P + id] = -(f0 >> fx_clamp(n0 - q0));
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        FxSum mo = fx_zero<2>();
        fx_add(mo, X, U[c]);
        fx_add(mo, Pp, J[c]);
        sF[(d * 5 + 1 + c) * P + id] = (V[c] >> fx_clamp(n3 - qm)) - fx_end<2>(mo);
      }
      FxSum en = fx_zero<0>(), h = fx_zero<4>();
      fx_add(en, fx_split(V[0]), U[0]); fx_add(en, fx_split(V[1]), U[1]); fx_add(en, fx_split(V[2]), U[2]);
      fx_add(h, T[0], J[0]); fx_add(h, T[1], J[1]); fx_add(h, T[2], J[2]);
      sF[(d * 5 + 4) * P + id] = (fx_end<0>(en) >> fx_clamp(n5 - qe)) + (fx_end<4>(h) >> fx_clamp(n6 - qe)) -
                                 (fx_mul<1>(H, un) >> fx_clamp(n4 - qe));
    }
    for (int o = id; o < 30 * NN; o += P) {
      const int v2 = (o / NN) % 5;
      i64* s = sFs + o;
      *s = fx_from(__longlong_as_double(*s), (v2 == 0 ? q0 : (v2 == 4 ? qe : qm)) + sh.t(o / (10 * NN)));
    }
  }
  __syncthreads();
  int bad = 0;
#pragma unroll
  for (int l = 0; l < EPB; ++l) bad |= state[l] == 2;
  if (!act) return bad;
  const int i = id % n, j = (id / n) % n, k = id / NN;
  i64 acc[5] = {0, 0, 0, 0, 0};
  const int walk = sh.walk();   // the directions by falling t: the sums are only shifted down
#pragma unroll 1
  for (int pass = 0; pass < 3; ++pass) {
    const int d = STRETCH ? walk >> (2 * pass) & 3 : pass;
    const int r = d == 0 ? i : (d == 1 ? j : k);
    const int stride = d == 0 ? 1 : (d == 1 ? n : NN);
    const int line0 = id - r * stride, pq = d == 0 ? j + n * k : (d == 1 ? i + n * k : i + n * j);
    const Fx* Dr = sDw + r * n;
    const Fx t0 = sT[r], t1 = sT[n + r];
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      FxSum s = fx_zero<kFxUpD>();
      const i64* line = sF + (d * 5 + c) * P + line0;
#pragma unroll
      for (int m = 0; m < n; ++m) {
        if (n + 2 > 6 && m == (n + 2) / 2) fx_fold(s);
        fx_add(s, Dr[m], fx_split(line[m * stride]));
      }
      fx_add(s, t0, fx_split(sFs[(2 * d * 5 + c) * NN + pq]));
      fx_add(s, t1, fx_split(sFs[((2 * d + 1) * 5 + c) * NN + pq]));
      acc[c] += fx_end<kFxUpD>(s);
    }
    if (const int down = walk >> (8 + 4 * pass) & 15) {
#pragma unroll
      for (int c = 0; c < 5; ++c) acc[c] = (acc[c] + ((i64)1 << (down - 1))) >> down;
    }
  }
  double src[5] = {0, 0, 0, 0, 0};
  if (g.source == DG_SOURCE_MMS) mms_source<double>(g, mms, e, P, id, s_tc[0], s_tc[1], src);
  const double iJ = metrics[((size_t)e * 10 + 9) * P + id];
  const size_t o0 = (size_t)e * 5 * P + id;
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    const size_t o = o0 + (size_t)c * P;
    const double R = fma(-fx_to(acc[c], (c == 0 ? q0 : (c == 4 ? qe : qm)) - 2 - eD), iJ, src[c]);
    if (a.mode == 0) {
      a.Ut[o] = R;
    } else {
      const double gk = fma(a.A, rk_register(a, o), a.clock[1] * R);
      a.Gk[o] = gk;
      a.Uw[o] = fma(a.B, gk, q[c]);
    }
  }
  return bad;
}

}  // namespace dg
