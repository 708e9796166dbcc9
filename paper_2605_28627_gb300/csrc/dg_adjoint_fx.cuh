// Pairs of the volume adjoint on LGL nodes in block fixed point (dg_fixed.cuh):
// the reverse mode of the two-point flux (ec_flux_vjp) summed over the pairs of
// a node, with the chain from beta to density and pressure, and from |u|^2 to
// the velocities, applied once per node instead of once per pair.
//
// The state and the adjoint -lambda/J are held with exponents per element; the
// quantities of a pair that carry the adjoint are block floating point with an
// exponent per pair (FxF, FxF3: products of several such factors would lose
// their digits under a bound taken over the element), and the sums over the
// pairs are 96 bits wide with one exponent per element.  With f = (a - b)/(a +
// b), u = f^2, the logarithmic mean is L = (a + b)/2 (1 - V(u)), dL/da = (1 -
// V)/2 - V' f (1 - f), dL/db = (1 - V)/2 + V' f (1 + f).
//
// Bound and measured: the FP64 pairs (about 135 FP64 instructions each) held the
// FP64 pipe 87 % busy; a pair here costs some 900 integer instructions, and the
// viscous part's 250 FP64 instructions a node run beside them.  One
// vector-Jacobian product on 16^3 elements, FP64 pairs -> these (us): N = 3 976 ->
// 717, 5 3787 -> 2124, 7 10464 -> 5666 (with the face and viscous parts as they
// are now 505, 1468, 4306); its error against 64 bits is 0.7 to 1.1 of the FP64
// pairs'.
#pragma once

#include "dg_fixed.cuh"
#ifdef __CUDACC__
#include "dg_adjoint_fn.cuh"
#include "dg_fx_metrics.cuh"
#include "dg_stage.cuh"
#endif

namespace dg {

// A value m 2^(e - 60), |m| < 2^60, and three values with one exponent.
struct FxF {
  i64 m;
  int e;
};
struct FxF3 {
  i64 m[3];
  int e;
};
DG_HD int fx_clz(int x) {
#ifdef __CUDA_ARCH__
  return __clz(x);
#else
  return x ? __builtin_clz((unsigned)x) : 32;
#endif
}
DG_HD int fx_sign_fold(i64 x) {   // high word, complemented if negative
  const int h = fx_high(x);
  return h ^ (h >> 31);
}
// moves the leading digits up to bit 59 (by at most 28 bits)
DG_HD FxF fx_norm(FxF x) {
  const int s = fx_clz(fx_sign_fold(x.m)) - 4;
  return FxF{fx_up(x.m, s), x.e - s};
}
DG_HD FxF3 fx_norm(const FxF3& x) {
  const int s = fx_clz(fx_sign_fold(x.m[0]) | fx_sign_fold(x.m[1]) | fx_sign_fold(x.m[2])) - 4;
  return FxF3{{fx_up(x.m[0], s), fx_up(x.m[1], s), fx_up(x.m[2], s)}, x.e - s};
}
DG_HD int fx_max(int a, int b) { return a > b ? a : b; }
DG_HD i64 fx_down(i64 x, int s) { return x >> (s < 63 ? s : 63); }   // s >= 0

// Exponents of one element: of the state and of the adjoint's components, the
// shift of 1/(b_a + b_b), and the bounds of the sums over the pairs.
struct alignas(16) FxAdjAlign {
  int r, u, b, j;
  int l0, lm, l4, eg;
  int ky, eub, erho, ebt;
  int ek, eD, t, pad;   // t: the directions' shifts (FxMetricShifts)
};
// e: exponents of the state (FxExp, with lb), eg of 1/(gamma - 1); l0, lm, l4 of
// the adjoint -lambda/J (mass, momentum, energy).
DG_HD FxAdjAlign fx_adj_align(const FxExp& e, int eg, int l0, int lm, int l4, int eD) {
  FxAdjAlign a;
  a.r = e.r; a.u = e.u; a.b = e.b; a.j = e.j;
  a.l0 = l0; a.lm = lm; a.l4 = l4; a.eg = eg;
  a.eD = eD;
  a.ky = fx_clamp(fx_floor(62.0f - (118.0f - (60.0f + e.lb))));
  // bounds of the terms (not of their digits): sums of 27 or fewer stay below 2^63
  const int ew0 = l0 + eD + 2, ewm = lm + eD + 2, ew4 = l4 + eD + 2;
  const int ef0 = e.r + e.u + e.j, ep = e.r - e.b + 1 - a.ky, ef = fx_max(ef0 + e.u, ep + e.j) + 1;
  const int eth = 1 - e.b - a.ky + eg, eH = fx_max(eth, 2 * e.u + 1) + 1;
  const int efb = fx_max(ewm, ew4 + e.u) + 1, e0 = fx_max(ew0, fx_max(ew4 + eH, efb + e.u + 2)) + 2;
  const int esr = efb + e.j - e.b - a.ky, ebl = ew4 + ef0 + eth - e.b - a.ky + 2;
  a.eub = fx_max(ew4 + ef, fx_max(ef0 + efb, e0 + e.r + e.j)) + 2 + 2;
  a.erho = fx_max(esr, e0 + e.u + e.j + 1) + 1 + 2;
  a.ebt = fx_max(esr + ep + 1, ebl + 1) + 1 + 2;
  a.ek = ew4 + ef0 + 2;
  a.t = a.pad = 0;
  return a;
}

// V'(u) = sum k b_k u^(k-1), u = U 2^-56 < 2^-8, 62 bits after the point.
DG_HD i64 fx_series_slope(i64 U) {
  constexpr FxSeries S = fx_series();
  const int c2 = (int)(3 * (S.b[2] >> 30)), c3 = (int)(4 * (S.b[3] >> 30)), c4 = (int)(5 * (S.b[4] >> 30)),
            c5 = (int)(6 * (S.b[5] >> 30));                           // 32 bits after the point
  const int u32 = (int)(U >> 24), u39 = (int)(U >> 17);
  int t = c4 + fx_mulhi(u32, c5);
  t = c3 + fx_mulhi(u32, t);
  t = c2 + fx_mulhi(u32, t);
  const i64 h = (S.b[1] >> 1) + (fx_wide(u39, t) >> 11);              // 2 b_2 + u t, 60 bits
  return S.b[0] + fx_mul<0>(fx_split(fx_up(U, 10)), fx_split(h));
}

// Means of one pair and their derivatives: 2 rho_ln (60 - e_r), (1 + w) / (b_a +
// b_b) (59 + e_b + k_y), dL/da and dL/db of both (61 bits: below 1.6).
struct FxMeansD {
  i64 rln2, hib, ra, rb, ba, bb;
};
// dL/da, dL/db from V (64 bits), f (60), V' (62)
DG_HD void fx_mean_slopes(i64 V, i64 f, i64 Vp, i64& La, i64& Lb) {
  const Fx f8 = fx_split(fx_up(f, 3));                               // 63 bits, |f| < 2^-4
  const i64 g = fx_mul<0>(fx_split(Vp), f8), gf = fx_up(fx_mul<0>(fx_split(g), f8), 2);
  const i64 m = ((i64)1 << 61) - (V >> 3) + gf;
  La = (m >> 1) - g;
  Lb = (m >> 1) + g;
}
#ifdef __CUDACC__
// by FP64 where a ratio is large (u >= 2^-8)
struct FxLongD {
  static __device__ __noinline__ FxMeansD run(i64 ra, i64 rb, i64 ba, i64 bb, i64 yb) {
  double La, Lb;
  FxMeansD m;
  m.rln2 = fx_from(2.0 * log_mean_d((double)ra, (double)rb, La, Lb), 0);
  m.ra = fx_from(La, 61);
  m.rb = fx_from(Lb, 61);
  const double a = (double)ba, b = (double)bb;
  const double L = log_mean_d(a, b, La, Lb);
  m.hib = fx_from((double)yb * (0.5 * (a + b) / L), 0);
  m.ba = fx_from(La, 61);
  m.bb = fx_from(Lb, 61);
  return m;
}
  __device__ FxMeansD operator()(i64 ra, i64 rb, i64 ba, i64 bb, i64 yb) const { return run(ra, rb, ba, bb, yb); }
};
#endif

// Adjoint of the two-point flux: S = D_rm lam_r + D_mr lam_m (58 - e_D - l
// bits, below 2^59; half the adjoint of the flux).  Shares of the density
// adjoint of both nodes (r[0], r[1], exponent er), of beta (b[0], b[1], eb), of
// {u} (u) and of |u|^2 (k).  j: exponent of the metric terms (at most al.j).
struct FxPairAdj {
  i64 r[2], b[2];
  int er, eb;
  FxF3 u;
  FxF k;
};
template <class LONG>
DG_HD FxPairAdj fx_pair_vjp(i64 ra, i64 rb, i64 ba, i64 bb, const i64 su[3], i64 sk, const i64 sn[3], Fx G,
                            int j, const i64 S[5], const FxAdjAlign& al, LONG slopes_long) {
  const i64 sr = ra + rb;
  const Fx Sr = fx_split(sr), Sb = fx_split(ba + bb);
  const i64 yr = fx_rcp(Sr);
  const i64 yb0 = fx_rcp_full(Sb, fx_rcp(Sb));
  const i64 fr = fx_up(fx_mul<0>(fx_split(ra - rb), fx_split(yr)), 5);
  const i64 fb = fx_up(fx_mul<0>(fx_split(ba - bb), fx_split(yb0)), 5);
  const i64 Ur = fx_mul<0>(fx_split(fr), fx_split(fr)), Ub = fx_mul<0>(fx_split(fb), fx_split(fb));
  const i64 yb = fx_up(yb0, al.ky);
  const Fx Yb = fx_split(yb);
  FxMeansD mn;
  if (fx_high(Ur | Ub) < (1 << 16)) {
    const i64 Vr = fx_series_sum<true>(Ur);
    mn.rln2 = sr - fx_mul<0>(Sr, fx_split(Vr));
    fx_mean_slopes(Vr, fr, fx_series_slope(Ur), mn.ra, mn.rb);
    mn.hib = yb + fx_mul<0>(Yb, fx_split(fx_series_sum<false>(Ub)));
    fx_mean_slopes(fx_series_sum<true>(Ub), fb, fx_series_slope(Ub), mn.ba, mn.bb);
  } else {
    mn = slopes_long(ra, rb, ba, bb, yb);
  }
  // a product of values below 2^60, and its exponent the sum of theirs
  auto mul = [](Fx a, Fx b) { return fx_mul<4>(a, b); };
  const Fx U[3] = {fx_split(su[0]), fx_split(su[1]), fx_split(su[2])};   // 61 bits of {u}
  const Fx N[3] = {fx_split(sn[0]), fx_split(sn[1]), fx_split(sn[2])};   // 61 bits of {n}
  const Fx Rl = fx_split(mn.rln2), Hi = fx_split(mn.hib);
  const int ei = -al.b - al.ky;                        // of 1/(2 beta_ln): Hi has 62 bits, and of 1/(8 (b_a + b_b))
  FxSum s = fx_zero<2>();
  fx_add(s, U[0], N[0]); fx_add(s, U[1], N[1]); fx_add(s, U[2], N[2]);
  const FxF un = fx_norm(FxF{fx_end<2>(s), al.u + j});
  const Fx unx = fx_split(un.m);
  const FxF f0 = fx_norm(FxF{fx_mul<3>(Rl, unx), al.r + un.e});
  const FxF ph = fx_norm(FxF{fx_mul<1>(Sr, Yb), al.r + 1 + ei});
  const FxF th = fx_norm(FxF{fx_mul<0>(Hi, G), 1 + al.eg + ei});         // 1/(2 (gamma - 1) beta_ln)
  const Fx f0x = fx_split(f0.m), phx = fx_split(ph.m), thx = fx_split(th.m);
  // H = th - K, K = (k_a + k_b)/4
  const int eh = fx_max(th.e, 2 * al.u + 1) + 1;
  const FxF H = fx_norm(FxF{fx_down(th.m, eh - th.e) - fx_down(sk, eh - 2 * al.u), eh});
  // the flux adjoint (2 S): exponents l + e_D + 3
  const FxF w0 = fx_norm(FxF{S[0], al.l0 + al.eD + 3}), w4 = fx_norm(FxF{S[4], al.l4 + al.eD + 3});
  const Fx W4 = fx_split(w4.m);
  // adjoint of the momentum flux: w_m + w_4 {u}
  const int em = al.lm + al.eD + 3, efb = fx_max(em, w4.e + al.u) + 1, d1 = efb - em, d2 = efb - w4.e - al.u;
  FxF3 fmb;
#pragma unroll
  for (int l = 0; l < 3; ++l) fmb.m[l] = fx_down(S[1 + l], d1) + fx_down(fx_mul<3>(W4, U[l]), d2);
  fmb.e = efb;
  fmb = fx_norm(fmb);
  const Fx B[3] = {fx_split(fmb.m[0]), fx_split(fmb.m[1]), fx_split(fmb.m[2])};
  // adjoint of the mass flux: w_0 + w_4 H + fmb . {u}
  s = fx_zero<1>();
  fx_add(s, B[0], U[0]); fx_add(s, B[1], U[1]); fx_add(s, B[2], U[2]);
  const int eq = fmb.e + al.u + 2, e0 = fx_max(fx_max(w0.e, w4.e + H.e), eq) + 2;
  const FxF f0b = fx_norm(FxF{fx_down(w0.m, e0 - w0.e) + fx_down(mul(W4, fx_split(H.m)), e0 - w4.e - H.e) +
                                  fx_down(fx_end<1>(s), e0 - eq), e0});
  const Fx f0bx = fx_split(f0b.m);
  FxPairAdj o;
  const FxF Hb{mul(W4, f0x), w4.e + f0.e};
  o.k = FxF{-Hb.m, Hb.e};
  s = fx_zero<3>();
  fx_add(s, B[0], N[0]); fx_add(s, B[1], N[1]); fx_add(s, B[2], N[2]);
  const FxF phb = fx_norm(FxF{fx_end<3>(s), fmb.e + j});
  // f_m = f0 {u} + p_hat n
  const int ef = fx_max(f0.e + al.u, ph.e + j) + 1;
  const Fx A1 = fx_split(fx_down(f0.m, ef - f0.e - al.u)), A2 = fx_split(fx_down(ph.m, ef - ph.e - j));
  FxF3 fm;
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    FxSum m = fx_zero<3>();
    fx_add(m, A1, U[l]);
    fx_add(m, A2, N[l]);
    fm.m[l] = fx_end<3>(m);
  }
  fm.e = ef;
  fm = fx_norm(fm);
  // adjoint of {u}: w_4 f_m + f0 fmb + (f0b rho_ln) n
  const FxF c3 = fx_norm(FxF{fx_mul<3>(f0bx, Rl), f0b.e + al.r});
  const int e1 = w4.e + fm.e, e2 = f0.e + fmb.e, e3 = c3.e + j, eu = fx_max(fx_max(e1, e2), e3) + 2;
  const Fx C1 = fx_split(fx_down(w4.m, eu - e1)), C2 = fx_split(fx_down(f0.m, eu - e2)),
           C3 = fx_split(fx_down(c3.m, eu - e3 + 1));
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    FxSum t = fx_zero<4>();
    fx_add(t, C1, fx_split(fm.m[l]));
    fx_add(t, C2, B[l]);
    fx_add(t, C3, N[l]);
    o.u.m[l] = fx_end<4>(t);
  }
  o.u.e = eu;
  // density: phb / (2 s_beta) + rlb dL, rlb = f0b un; beta: -phb p_hat / s_beta - blb dL, blb = Hb th / beta_ln
  const FxF sb{fx_mul<2>(fx_split(phb.m), Yb), phb.e + ei};
  const FxF rl = fx_norm(FxF{mul(f0bx, unx), f0b.e + un.e});
  const FxF st{mul(fx_split(sb.m), phx), sb.e + ph.e + 1};
  const FxF bl = fx_norm(FxF{fx_mul<2>(fx_split(mul(fx_split(Hb.m), thx)), Hi), Hb.e + th.e + ei + 2});
  o.er = fx_max(sb.e, rl.e + 1) + 1;
  o.eb = fx_max(st.e, bl.e + 1) + 1;
  const Fx R2 = fx_split(fx_down(rl.m, o.er - rl.e)), B2 = fx_split(fx_down(bl.m, o.eb - bl.e));
  const i64 s0 = fx_down(sb.m, o.er - sb.e), b0 = fx_down(st.m, o.eb - st.e);
  o.r[0] = s0 + fx_mul<3>(R2, fx_split(mn.ra));
  o.r[1] = s0 + fx_mul<3>(R2, fx_split(mn.rb));
  o.b[0] = -b0 - fx_mul<3>(B2, fx_split(mn.ba));
  o.b[1] = -b0 - fx_mul<3>(B2, fx_split(mn.bb));
  return o;
}

#ifdef __CUDACC__
// 96-bit sum: 64 bits and a fraction of 32.
struct FxWide {
  u64 l;
  int h;
};
// adds x / 2^s, s >= 0
__device__ __forceinline__ void fx_wide_add(FxWide& a, i64 x, int s) {
  unsigned l0 = (unsigned)a.l, l1 = (unsigned)(a.l >> 32);
  const i64 v = fx_down(x, s);
  const unsigned x0 = (unsigned)fx_down(fx_up(x, 32), s) , x1 = (unsigned)(u64)v, x2 = (unsigned)fx_high(v);
  const unsigned f = s < 32 ? x0 : (unsigned)fx_down(x, s - 32);
  asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
      : "+r"(l0), "+r"(l1), "+r"(a.h)
      : "r"(f), "r"(x1), "r"(x2));
  a.l = (u64)l1 << 32 | l0;
}
// as a double with q bits of the 64 after the point
__device__ __forceinline__ double fx_wide_to(const FxWide& s, int q) {
  return fx_to2<32>((i64)((u64)(unsigned)s.h << 32 | s.l >> 32), (i64)(unsigned)s.l, q);
}

// Words of 8 bytes per node: rho, b, |u|^2, u (3), metric terms (9), adjoint (5),
// exchange (6, and the exponents as four 16-bit fields).
constexpr int kFxAdjWords = 27;

// The primitive adjoints pr (rho, u, v, w, p) of the two-point terms of every
// element in range (state[le] = 1); out-of-range elements are left (state 2),
// and the return value says whether the block holds any.
template <int N>
__device__ __forceinline__ bool adj_pairs_fx(const double* __restrict__ U, const double* __restrict__ lam,
                                             const double* __restrict__ metrics, const i64* __restrict__ jx,
                                             const float4* __restrict__ ejx, const double* __restrict__ Dg, int E,
                                             const Gas& g, unsigned char* smem, int* state, double pr[5]) {
  using S = Shape<N>;
  constexpr int n = S::n, P = S::P, NN = S::NN, EPB = S::EPB, eD = fx_eD(N);
  constexpr int FULL = (n - 1) / 2;
  constexpr bool HALF = (n % 2) == 0;
  Fx* sD = reinterpret_cast<Fx*>(smem);
  i64* const tile0 = reinterpret_cast<i64*>(smem) + n * n;
  enum { kR, kRmin, kB, kBmin, kU, kL0, kLm, kL4, kCount };
  __shared__ int s_mx[EPB][kCount];
  __shared__ FxAdjAlign s_al[EPB];
  __shared__ Fx s_G;
  const int le = threadIdx.x / P, id = threadIdx.x - le * P;
  const int e = blockIdx.x * EPB + le;
  const bool active = e < E;
  i64* base = tile0 + (size_t)le * kFxAdjWords * P;
  const int eg = fx_expo(fx_mag(g.inv_gm1));
  for (int t = threadIdx.x; t < n * n; t += blockDim.x) sD[t] = fx_split(fx_round(Dg[t], kFxQD - eD));
  for (int t = threadIdx.x; t < EPB * kCount; t += blockDim.x) s_mx[t / kCount][t % kCount] = 0;
  if (threadIdx.x == 0) s_G = fx_split(fx_from(g.inv_gm1, 62 - eg));
  __syncthreads();
  double rho = 1, u = 0, v = 0, w = 0, bt = 1, kk = 0, lv[5] = {0, 0, 0, 0, 0};
  if (active) {
    const double* q = U + (size_t)e * 5 * P + id;
    rho = q[0];
    const double ir = adj_rcp(rho);
    u = q[P] * ir; v = q[2 * P] * ir; w = q[3 * P] * ir;
    kk = u * u + v * v + w * w;
    bt = 0.125 * rho * adj_rcp(g.gm1 * fma(-0.5 * rho, kk, q[4 * P]));   // beta / 4
    const double iJ = metrics[((size_t)e * 10 + 9) * P + id];
#pragma unroll
    for (int c = 0; c < 5; ++c) lv[c] = -lam[((size_t)e * 5 + c) * P + id] * iJ;
    const int hr = max(__double2hiint(rho), 0), hb = max(__double2hiint(bt), 0);
    // the last bit set if any of the low word is: a subnormal adjoint is not zero
    auto mag = [](double x) { return fx_mag(x) | (__double2loint(x) != 0); };
    int m[kCount] = {hr, 0x7fffffff - hr, hb, 0x7fffffff - hb, max(max(mag(u), mag(v)), mag(w)), mag(lv[0]),
                     max(max(mag(lv[1]), mag(lv[2])), mag(lv[3])), mag(lv[4])};
    fx_maxima<kCount>(le, s_mx[le], m);
  }
  __syncthreads();
  const int* mx = s_mx[le];
  const float4 ej = active ? ejx[e] : make_float4(1000.0f, 0.0f, 0.0f, 0.0f);
  const FxMetricShifts sh = fx_shifts(ej);
  FxExp x{fx_expo(mx[kR]), fx_expo(mx[kU]), fx_expo(mx[kB]), (int)ej.x, 0.0f, 0.0f, 0.0f, 0.0f};
  const int l0 = fx_expo(mx[kL0]), lm = fx_expo(mx[kLm]), l4 = fx_expo(mx[kL4]);
  const int rmin = 0x7fffffff - mx[kRmin], bmin = 0x7fffffff - mx[kBmin];
  const int dr = x.r - ((rmin >> 20) - 1023), db = x.b - ((bmin >> 20) - 1023);
  auto in = [](int v) { return v > -60 && v < 60; };
  const bool act = active && rmin > 0 && bmin > 0 && dr <= 4 && db <= 4 && in(x.r) && in(x.b) && in(x.j) &&
                   fx_in_range(mx[kU], 60) && fx_in_range(mx[kL0], 60) && fx_in_range(mx[kLm], 60) &&
                   fx_in_range(mx[kL4], 60);
  if (id == 0) {
    state[le] = active ? (act ? 1 : 2) : 0;
    if (act) {
      x.lb = fx_log_mantissa(bmin, 0) + (float)((bmin >> 20) - 1022 - x.b);
      s_al[le] = fx_adj_align(x, eg, l0, lm, l4, eD);
      s_al[le].t = sh.w;
    }
  }
  if (act) {
    base[id] = fx_from(rho, 60 - x.r);
    base[P + id] = fx_from(bt, 60 - x.b);
    base[2 * P + id] = fx_from(kk, 58 - 2 * x.u);
    base[3 * P + id] = fx_from(u, 60 - x.u);
    base[4 * P + id] = fx_from(v, 60 - x.u);
    base[5 * P + id] = fx_from(w, 60 - x.u);
    const i64* mt = jx + (size_t)e * 10 * P + id;
#pragma unroll
    for (int r = 0; r < 9; ++r) base[(6 + r) * P + id] = fx_up(mt[r * P], sh.t(r / 3));
    base[15 * P + id] = fx_from(lv[0], 60 - l0);
#pragma unroll
    for (int c = 1; c < 4; ++c) base[(15 + c) * P + id] = fx_from(lv[c], 60 - lm);
    base[19 * P + id] = fx_from(lv[4], 60 - l4);
  }
  __syncthreads();
  const int i = id % n, j = (id / n) % n, k = id / NN;
  FxWide acc[6];   // density, beta, {u} (3), |u|^2
#pragma unroll
  for (int c = 0; c < 6; ++c) acc[c] = FxWide{0, 0};
  // pair (ia, ib) of the element at b2, rows ra, rb of D
  auto pair = [&](const i64* b2, int el, int d, int ia, int ib, int ra, int rb) {
    const Fx Dab = sD[ra * n + rb], Dba = sD[rb * n + ra];
    i64 W[5], su[3], sn[3];
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      FxSum s = fx_zero<kFxUpD>();
      fx_add(s, Dab, fx_split(b2[(15 + c) * P + ia]));
      fx_add(s, Dba, fx_split(b2[(15 + c) * P + ib]));
      W[c] = fx_end<kFxUpD>(s);
    }
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      su[l] = b2[(3 + l) * P + ia] + b2[(3 + l) * P + ib];
      sn[l] = b2[(6 + 3 * d + l) * P + ia] + b2[(6 + 3 * d + l) * P + ib];
    }
    return fx_pair_vjp(b2[ia], b2[ib], b2[P + ia], b2[P + ib], su, b2[2 * P + ia] + b2[2 * P + ib], sn, s_G,
                       s_al[el].j - (s_al[el].t >> (4 * d) & 15), W, s_al[el], FxLongD());
  };
  // a pair's shares for one node into its exchange slot; the shifts to the
  // exponents of the sums (at most 255) as bytes
  auto shifts = [&](const FxPairAdj& o, const FxAdjAlign& al) {
    auto c = [](int s) { return (unsigned)(s < 0 ? 0 : (s < 255 ? s : 255)); };
    return c(al.erho - o.er) | c(al.ebt - o.eb) << 8 | c(al.eub - o.u.e) << 16 | c(al.ek - o.k.e) << 24;
  };
  auto put = [&](i64* x, int at, const FxPairAdj& o, int side, unsigned sh) {
    x[at] = o.r[side];
    x[P + at] = o.b[side];
#pragma unroll
    for (int l = 0; l < 3; ++l) x[(2 + l) * P + at] = o.u.m[l];
    x[5 * P + at] = o.k.m;
    x[6 * P + at] = (i64)sh;
  };
  auto add = [&](i64 r, i64 b, const i64 m[3], i64 kx, unsigned sh) {
    const int s2 = (int)(sh >> 16 & 255u);
    fx_wide_add(acc[0], r, (int)(sh & 255u));
    fx_wide_add(acc[1], b, (int)(sh >> 8 & 255u));
#pragma unroll
    for (int l = 0; l < 3; ++l) fx_wide_add(acc[2 + l], m[l], s2);
    fx_wide_add(acc[5], kx, (int)(sh >> 24));
  };
  auto take = [&](const i64* x) {
    const i64 m[3] = {x[2 * P + id], x[3 * P + id], x[4 * P + id]};
    add(x[id], x[P + id], m, x[5 * P + id], (unsigned)x[6 * P + id]);
  };
  i64* sX = base + 20 * P;
#pragma unroll 1
  for (int d = 0; d < 3; ++d) {
    const int r = d == 0 ? i : (d == 1 ? j : k);
    const int stride = d == 0 ? 1 : (d == 1 ? n : NN);
    const int line0 = id - r * stride;
#pragma unroll 1
    for (int s = 1; s <= FULL; ++s) {
      const int m = r + s < n ? r + s : r + s - n;
      const int mid = line0 + m * stride;
      if (act) {
        const FxPairAdj o = pair(base, le, d, id, mid, r, m);
        const unsigned sh = shifts(o, s_al[le]);
        put(sX, mid, o, 1, sh);
        add(o.r[0], o.b[0], o.u.m, o.k.m, sh);
      }
      __syncthreads();
      if (act) take(sX);
      __syncthreads();
    }
    if constexpr (HALF) {
      // s = n/2: P/2 pairs per element, packed on the block's first threads
      constexpr int Hn = n / 2;
      const int t = threadIdx.x;
      const int le2 = t / (P / 2), w2 = t - le2 * (P / 2);
      if (t < EPB * (P / 2) && state[le2] == 1) {
        const int hi = w2 / stride;
        const int ra = hi % Hn;
        const int ia = w2 - hi * stride + stride * (ra + n * (hi / Hn)), ib = ia + Hn * stride;
        i64* b2 = tile0 + (size_t)le2 * kFxAdjWords * P;
        const FxPairAdj o = pair(b2, le2, d, ia, ib, ra, ra + Hn);
        const unsigned sh = shifts(o, s_al[le2]);
        put(b2 + 20 * P, ia, o, 0, sh);
        put(b2 + 20 * P, ib, o, 1, sh);
      }
      __syncthreads();
      if (act) take(sX);
      __syncthreads();
    }
  }
  int bad = 0;
#pragma unroll
  for (int l = 0; l < EPB; ++l) bad |= state[l] == 2;
  if (act) {
    const FxAdjAlign& al = s_al[le];
    const double rb = fx_wide_to(acc[0], 60 - al.erho), bb = fx_wide_to(acc[1], 60 - al.ebt);
    const double kb = 0.5 * fx_wide_to(acc[5], 60 - al.ek);
    const double be = 4.0 * bt, hip = be * adj_rcp(rho);   // 1/(2p) = beta / rho
    pr[0] = fma(bb, hip, rb);
    pr[1] = fma(kb, u, 0.5 * fx_wide_to(acc[2], 60 - al.eub));
    pr[2] = fma(kb, v, 0.5 * fx_wide_to(acc[3], 60 - al.eub));
    pr[3] = fma(kb, w, 0.5 * fx_wide_to(acc[4], 60 - al.eub));
    pr[4] = -2.0 * be * hip * bb;                          // beta / p = 2 beta / (2 p)
  }
  return bad;
}
#endif

}  // namespace dg
