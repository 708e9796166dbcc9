// Host build of the fixed-point arithmetic (csrc/dg_fixed.cuh) against long
// double: error statistics for tests/test_fixed_point.py.
#include <algorithm>
#include <cmath>
#include <cstdlib>

#include "../paper_2605_28627_gb300/csrc/dg_adjoint_fx.cuh"

using namespace dg;
using L = long double;

static double uniform(double a, double b) { return a + (b - a) * drand48(); }
static int expo(double x) {
  int e;
  frexp(x, &e);
  return e;
}
template <class T>
static T ratio_log(T a, T b) {   // atanh(f)/f, f = (a - b)/(a + b)
  const T f = (a - b) / (a + b), u = f * f;
  if (u < T(1e-4)) return 1 + u * (T(1) / 3 + u * (T(1) / 5 + u * (T(1) / 7 + u * (T(1) / 9 + u / 11))));
  const T z = a / b;
  return std::log(z) / (2 * ((z - 1) / (z + 1)));
}
template <class T>
static void flux(T ra, T rb, const T* ua, const T* ub, T ba, T bb, const T* sn, T ig, T* F) {
  T su[3], un = 0, sk = 0;
  for (int a = 0; a < 3; ++a) {
    su[a] = ua[a] + ub[a];
    un += su[a] * sn[a];
    sk += ua[a] * ua[a] + ub[a] * ub[a];
  }
  const T X = (ra + rb) / ratio_log(ra, rb) * un, Y = (ra + rb) / (ba + bb);
  F[0] = X;
  F[4] = X * (ratio_log(ba, bb) / (ba + bb) * ig - sk);
  for (int a = 0; a < 3; ++a) {
    F[1 + a] = X * su[a] + Y * sn[a];
    F[4] += su[a] * F[1 + a];
  }
}

// Logarithmic mean (a + b)/(2 F(f)), F = atanh(f)/f, and its derivatives.
template <class T>
static T log_mean(T a, T b, T& La, T& Lb) {
  const T s = a + b, f = (a - b) / s, u = f * f;
  T F = 1, dF = 0;   // dF = F'(f)
  if (u < T(0.05)) {
    T p = 1;
    for (int k = 1; k < 20; ++k) {
      dF += 2 * k * p * f / (2 * k + 1);
      p *= u;
      F += p / (2 * k + 1);
    }
  } else {
    F = std::log(a / b) / (2 * f);
    dF = (1 / (1 - u) - F) / f;
  }
  const T c = -dF / (F * F * s);   // of f_a = 2 b / s^2, f_b = -2 a / s^2
  La = 1 / (2 * F) + c * b;
  Lb = 1 / (2 * F) - c * a;
  return s / (2 * F);
}
// Adjoint of the two-point flux, o = {density a, b, beta a, b, {u} (3), K}, and
// the sum of each one's terms' magnitudes.
template <class T>
static void flux_vjp(T ra, T rb, const T* ua, const T* ub, T ba, T bb, const T* n, T ig, const T* w, T* o, T* mag) {
  T Lra, Lrb, Lba, Lbb, u[3], un = 0, K = 0, fm[3], fmb[3], phb = 0, f0b = w[0];
  const T rl = log_mean(ra, rb, Lra, Lrb), bl = log_mean(ba, bb, Lba, Lbb), isb = 1 / (ba + bb), ph = (ra + rb) * isb / 2;
  for (int l = 0; l < 3; ++l) {
    u[l] = (ua[l] + ub[l]) / 2;
    un += u[l] * n[l];
    K += (ua[l] * ua[l] + ub[l] * ub[l]) / 4;
  }
  const T f0 = rl * un, H = ig / (2 * bl) - K;
  T m0 = std::fabs(w[0]) + std::fabs(w[4] * H);
  f0b += w[4] * H;
  for (int l = 0; l < 3; ++l) {
    fm[l] = f0 * u[l] + ph * n[l];
    fmb[l] = w[1 + l] + w[4] * u[l];
    phb += fmb[l] * n[l];
    f0b += fmb[l] * u[l];
    m0 += std::fabs(fmb[l] * u[l]);
  }
  const T Hb = w[4] * f0, blb = -Hb * ig / (2 * bl * bl), sr = phb * isb / 2, sb = -phb * ph * isb, rlb = f0b * un;
  o[0] = sr + rlb * Lra; o[1] = sr + rlb * Lrb;
  o[2] = sb + blb * Lba; o[3] = sb + blb * Lbb;
  for (int l = 0; l < 3; ++l) {
    o[4 + l] = w[4] * fm[l] + f0 * fmb[l] + f0b * rl * n[l];
    mag[4 + l] = std::fabs(w[4] * fm[l]) + std::fabs(f0 * fmb[l]) + m0 * rl * std::fabs(n[l]);
  }
  o[7] = -Hb;
  mag[0] = mag[1] = std::fabs(sr) + m0 * std::fabs(un);
  mag[2] = mag[3] = std::fabs(sb) + std::fabs(blb);
  mag[7] = std::fabs(Hb);
}

extern "C" {

// Adjoint of the two-point flux, states and metric terms as in check_pairs, the
// cotangents of mass, momentum and energy below l0, lm, l4, rows of D below
// 2^eD.  out[0..3]: rms error of the density, beta, velocity and |u|^2 adjoints
// over the rms magnitude of their terms, out[4..7] of FP64, out[8]: smallest
// shift to the sums' exponents, out[9]: log2 of the largest share after it,
// out[10]: log2 of the largest share before it, out[11]: pairs outside the range.
void check_pair_vjp(int count, double r0, double r1, double p0, double p1, double um, double jm, int axis, double gamma,
                    int t0, double l0, double lm, double l4, int eD, double* out) {
  srand48(15);
  const double ig = 1.0 / (gamma - 1.0), jl = axis ? jm : 3 * jm, bmax = r1 / (8 * p0);
  FxExp e{expo(r1), expo(um), expo(bmax), expo(jl) + t0, 0, 0, 0, 0};
  const double bmin = std::max(r0 / (8 * p1), ldexp(1.0, e.b - 4));
  e.lb = (float)(log2(bmin) - e.b - 1e-3);
  const int eg = expo(ig);
  auto low = [](double x) { return x > 0 ? std::max(expo(x), -200) : -200; };
  const int e0 = low(l0), em = low(lm), e4 = low(l4);
  const FxAdjAlign al = fx_adj_align(e, eg, e0, em, e4, eD);
  const Fx G = fx_split(fx_from(ig, 62 - eg));
  double ef[4] = {0}, ed[4] = {0}, sc[4] = {0}, least = 1e9, after = 0, before = 0;
  long outside = 0;
  for (int t = 0; t < count; ++t) {
    const double ra = uniform(r0, r1), pa = uniform(p0, p1), near = t % 3 == 1 ? 1e-2 : 1e-5;
    double rb = t % 3 == 0 ? uniform(r0, r1) : std::min(r1, std::max(r0, ra * (1 + uniform(-near, near))));
    double pb = t % 3 == 0 ? uniform(p0, p1) : std::min(p1, std::max(p0, pa * (1 + uniform(-near, near))));
    if (t % 7 == 0) { rb = ra; pb = pa; }
    const double ba = 0.125 * ra / pa, bb = 0.125 * rb / pb;
    const i64 xr[2] = {fx_from(ra, 60 - e.r), fx_from(rb, 60 - e.r)}, xb[2] = {fx_from(ba, 60 - e.b), fx_from(bb, 60 - e.b)};
    if (std::min(std::min(xr[0], xr[1]), std::min(xb[0], xb[1])) < (i64)1 << 56 || ba < bmin || bb < bmin) { ++outside; continue; }
    i64 su[3], sn[3], S[5];
    double ua[3], ub[3], n[3], ka = 0, kb = 0, w[5];
    for (int a = 0; a < 3; ++a) {
      const bool on = !axis || a == 0;
      ua[a] = uniform(-um, um); ub[a] = uniform(-um, um);
      const double na = on ? uniform(-jm, jm) : 0, nb = on ? uniform(-jm, jm) : 0;
      n[a] = 0.5 * (na + nb);
      su[a] = fx_from(ua[a], 60 - e.u) + fx_from(ub[a], 60 - e.u);
      sn[a] = fx_up(fx_from(na, 60 - e.j), t0) + fx_up(fx_from(nb, 60 - e.j), t0);
      ka += ua[a] * ua[a]; kb += ub[a] * ub[a];
    }
    const double dab = uniform(-1, 1) * ldexp(1.0, eD), dba = uniform(-1, 1) * ldexp(1.0, eD);
    L wl[5];
    for (int c = 0; c < 5; ++c) {
      const double top = c == 0 ? l0 : (c < 4 ? lm : l4), la = uniform(-top, top), lb = uniform(-top, top);
      const int ec = c == 0 ? e0 : (c < 4 ? em : e4);
      FxSum s = fx_zero<kFxUpD>();
      fx_add(s, fx_split(fx_round(dab, kFxQD - eD)), fx_split(fx_from(la, 60 - ec)));
      fx_add(s, fx_split(fx_round(dba, kFxQD - eD)), fx_split(fx_from(lb, 60 - ec)));
      S[c] = fx_end<kFxUpD>(s);
      w[c] = 2 * (dab * la + dba * lb);
      wl[c] = 2 * ((L)dab * la + (L)dba * lb);
    }
    const FxPairAdj o = fx_pair_vjp(xr[0], xr[1], xb[0], xb[1], su, fx_from(ka, 58 - 2 * e.u) + fx_from(kb, 58 - 2 * e.u), sn, G,
                                    e.j - t0, S, al, [](i64 a, i64 b, i64 c, i64 d, i64 y) {
      double La, Lb;
      FxMeansD m;
      m.rln2 = fx_from(2.0 * log_mean((double)a, (double)b, La, Lb), 0);
      m.ra = fx_from(La, 61); m.rb = fx_from(Lb, 61);
      const double x = log_mean((double)c, (double)d, La, Lb);
      m.hib = fx_from((double)y * (0.5 * ((double)c + (double)d) / x), 0);
      m.ba = fx_from(La, 61); m.bb = fx_from(Lb, 61);
      return m;
    });
    L lua[3], lub[3], ln[3], R[8], mag[8];
    for (int a = 0; a < 3; ++a) { lua[a] = ua[a]; lub[a] = ub[a]; ln[a] = n[a]; }
    flux_vjp<L>(ra, rb, lua, lub, 4 * (L)ba, 4 * (L)bb, ln, ig, wl, R, mag);
    double D[8], dm[8];
    flux_vjp<double>(ra, rb, ua, ub, 4 * ba, 4 * bb, n, ig, w, D, dm);
    const i64 m[8] = {o.r[0], o.r[1], o.b[0], o.b[1], o.u.m[0], o.u.m[1], o.u.m[2], o.k.m};
    const int ex[8] = {o.er, o.er, o.eb, o.eb, o.u.e, o.u.e, o.u.e, o.k.e}, top[4] = {al.erho, al.ebt, al.eub, al.ek};
    for (int v = 0; v < 8; ++v) {
      const int c = v < 2 ? 0 : (v < 4 ? 1 : (v < 7 ? 2 : 3));
      const L unit = std::ldexp((L)1, top[c] - 60);   // the sums' scale, so that squares stay in range
      ef[c] += (double)std::pow((std::ldexp((L)m[v], ex[v] - 60) - R[v]) / unit, 2);
      ed[c] += (double)std::pow((D[v] - R[v]) / unit, 2);
      sc[c] += (double)std::pow(mag[v] / unit, 2);
      least = std::min(least, (double)(top[c] - ex[v]));
      before = std::max(before, std::fabs((double)m[v]));
      after = std::max(after, std::ldexp(std::fabs((double)m[v]), ex[v] - top[c]));
    }
  }
  for (int c = 0; c < 4; ++c) {
    out[c] = std::sqrt(ef[c] / sc[c]);
    out[4 + c] = std::sqrt(ed[c] / sc[c]);
  }
  out[8] = least;
  out[9] = std::log2(after);
  out[10] = std::log2(before);
  out[11] = (double)outside;
}

// Pairs with density in [r0, r1], pressure in [p0, p1], velocities below um,
// metric terms below jm (axis: one component only) in an element whose largest
// are 2^t0 loose times as large, gamma.  out[0..2]: rms
// error of the fixed-point mass, momentum and energy flux over the rms flux,
// out[3..5]: the same of FP64, out[6]: largest |F| as log2, out[7]: pairs
// outside the range.
void check_pairs(int count, double r0, double r1, double p0, double p1, double um, double jm, int axis, double gamma,
                 int t0, double loose, double* out) {
  srand48(11);
  const double ig = 1.0 / (gamma - 1.0), jl = loose * (axis ? jm : 3 * jm), bmax = r1 / (8 * p0);
  FxExp e{expo(r1), expo(um), expo(bmax), expo(jl), 0, 0, 0, 0};
  const double bmin = std::max(r0 / (8 * p1), ldexp(1.0, e.b - 4));
  e.lr = (float)(log2(r1) - e.r + 1e-3);
  e.lu = (float)(log2(um) - e.u + 1e-3);
  e.lj = (float)(log2(jl) - e.j + 1e-3);
  e.lb = (float)(log2(bmin) - e.b - 1e-3);
  const int eD = 5, eg = expo(ig);
  const FxAlign al = fx_align(e, eg, (float)(log2(ig) - eg + 1e-3), eD);
  const Fx G = fx_split(fx_from(ig, 62 - eg));
  double ef[3] = {0}, ed[3] = {0}, sc[3] = {0}, big = 0;
  long outside = 0;
  for (int t = 0; t < count; ++t) {
    // both nodes anywhere in the range, close together, or equal
    const double ra = uniform(r0, r1), pa = uniform(p0, p1), near = t % 3 == 1 ? 1e-2 : 1e-5;
    double rb = t % 3 == 0 ? uniform(r0, r1) : std::min(r1, std::max(r0, ra * (1 + uniform(-near, near))));
    double pb = t % 3 == 0 ? uniform(p0, p1) : std::min(p1, std::max(p0, pa * (1 + uniform(-near, near))));
    if (t % 7 == 0) { rb = ra; pb = pa; }
    double ua[3], ub[3], na[3], nb[3], sn[3];
    for (int a = 0; a < 3; ++a) {
      const bool on = !axis || a == 0;
      ua[a] = uniform(-um, um); ub[a] = uniform(-um, um);
      na[a] = on ? uniform(-jm, jm) : 0; nb[a] = on ? uniform(-jm, jm) : 0;
      sn[a] = na[a] + nb[a];
    }
    const double ba = 0.125 * ra / pa, bb = 0.125 * rb / pb;
    const i64 xr[2] = {fx_from(ra, 60 - e.r), fx_from(rb, 60 - e.r)}, xb[2] = {fx_from(ba, 60 - e.b), fx_from(bb, 60 - e.b)};
    const i64 least = (i64)1 << 56;
    if (std::min(std::min(xr[0], xr[1]), std::min(xb[0], xb[1])) < least || ba < bmin || bb < bmin) { ++outside; continue; }
    i64 su[3], n2[3];
    double ka = 0, kb = 0;
    for (int a = 0; a < 3; ++a) {
      su[a] = fx_from(ua[a], 60 - e.u) + fx_from(ub[a], 60 - e.u);
      n2[a] = fx_up(fx_from(na[a], 60 - e.j - t0), t0) + fx_up(fx_from(nb[a], 60 - e.j - t0), t0);
      ka += ua[a] * ua[a]; kb += ub[a] * ub[a];
    }
    i64 F[5];
    fx_pair(xr[0], xr[1], xb[0], xb[1], su[0], su[1], su[2], fx_from(ka, 58 - 2 * e.u) + fx_from(kb, 58 - 2 * e.u), n2[0],
            n2[1], n2[2], G, al, F, [](i64 a, i64 b, i64 c, i64 d, i64 y, i64 u, i64 v) {
              return fx_means_long(a, b, c, d, y, u, v, [](double p, double q) { return ratio_log<double>(p, q); });
            });
    L la[3], lb[3], ln[3], R[5];
    for (int a = 0; a < 3; ++a) { la[a] = ua[a]; lb[a] = ub[a]; ln[a] = (L)na[a] + nb[a]; }
    flux<L>(ra, rb, la, lb, ba, bb, ln, ig, R);
    double D[5];
    flux<double>(ra, rb, ua, ub, ba, bb, sn, ig, D);
    for (int v = 0; v < 5; ++v) {
      const int q = (v == 0 ? al.q0 - 2 : (v < 4 ? al.qm - 3 : al.qe - 4)) - (kFxQD - eD - 64);
      const double d = (double)(std::ldexp((L)F[v], -q) - R[v]), s = (double)R[v];
      const int c = v == 0 ? 0 : (v < 4 ? 1 : 2);   // the momentum as one vector
      ef[c] += d * d;
      ed[c] += (double)((D[v] - R[v]) * (D[v] - R[v]));
      sc[c] += s * s;
      big = std::max(big, std::fabs((double)F[v]));
    }
  }
  for (int c = 0; c < 3; ++c) {
    out[c] = std::sqrt(ef[c] / sc[c]);
    out[3 + c] = std::sqrt(ed[c] / sc[c]);
  }
  out[6] = std::log2(big);
  out[7] = (double)outside;
}

// Lifted gradients of one field along a line of n nodes, D [n][n], half = 1/(2
// w_0): g = (1/J_el) J (D phi + jump), the element's largest metric term 2^c
// times as large as this one, the other two derivatives 0.  out: rms
// error of the fixed-point and of the FP64 arithmetic over the rms gradient.
void check_lifting(int count, int n, const double* D, int eD, double half, int c, double* out) {
  srand48(14);
  double ef = 0, ed = 0, sc = 0;
  for (int t = 0; t < count; ++t) {
    const double J = ldexp(uniform(0.5, 1.0), -3), iJ = uniform(0.6, 1.9), base = uniform(-1, 1), amp = uniform(0.01, 0.3),
                 ph = uniform(0, 6);
    double phi[16], top = 0;
    for (int m = 0; m < n; ++m) top = std::max(top, std::fabs(phi[m] = base + amp * std::sin(ph + 2.0 * m / n)));
    const double nbr[2] = {phi[0] + uniform(-1e-3, 1e-3), phi[n - 1] + uniform(-1e-3, 1e-3)};
    top = std::max(top, std::max(std::fabs(nbr[0]), std::fabs(nbr[1])));
    const int e = expo(top), ej = expo(J), ei = expo(iJ);
    const Fx Jx[3] = {fx_split(fx_up(fx_from(J, kFxQ - ej - c), c)), fx_split(0), fx_split(0)}, iJx = fx_split(fx_from(iJ, 62 - ei));
    for (int r = 0; r < n; ++r) {
      const bool edge = r == 0 || r == n - 1;
      const double hs = r == 0 ? -half : half, nb = nbr[r != 0];
      const i64 own = fx_from(phi[r], kFxQ - e);
      FxSum s = fx_lift_start(
          edge ? fx_mul<0>(fx_split(fx_from(nb, kFxQ - e) - own), fx_split(fx_round(hs, kFxQD - eD))) : 0);
      double d = edge ? (nb - phi[r]) * hs : 0;
      L x = edge ? ((L)nb - phi[r]) * hs : 0;
      for (int m = 0; m < n; ++m) {
        fx_add(s, fx_split(fx_round(D[r * n + m], kFxQD - eD)), fx_split(fx_from(phi[m], kFxQ - e)));
        d = std::fma(D[r * n + m], phi[m], d);
        x += (L)D[r * n + m] * phi[m];
      }
      const Fx dd[3] = {fx_split(fx_lift_line(s)), fx_split(0), fx_split(0)};
      const double f = fx_to(fx_lift_gradient(Jx, dd, iJx), fx_lift_bits(eD, ej, ei) - e);
      x = x * J * iJ;
      d = J * d * iJ;
      ef += (double)((f - x) * (f - x));
      ed += (double)((d - x) * (d - x));
      sc += (double)(x * x);
    }
  }
  out[0] = std::sqrt(ef / sc);
  out[1] = std::sqrt(ed / sc);
}

// Largest relative error of 2^119 / S over S in [2^57, 2^61).
double check_rcp(int count) {
  srand48(12);
  double worst = 0;
  for (int t = 0; t < count; ++t) {
    const i64 S = t < 16 ? ((i64)1 << (57 + t % 4)) + t / 4 : (i64)ldexp(1 + drand48(), 57 + t % 4);
    const Fx s = fx_split(S);
    const L y = std::ldexp((L)1, 119) / (L)S;
    worst = std::max(worst, (double)std::fabs(((L)fx_rcp_full(s, fx_rcp(s)) - y) / y));
  }
  return worst;
}

// Conversions: worst error of fx_from in units of its last bit, of fx_to and
// fx_to2 relative to the value.
void check_conversions(int count, double* out) {
  srand48(13);
  out[0] = out[1] = out[2] = 0;
  for (int t = 0; t < count; ++t) {
    double x = t < 4 ? (t & 1 ? -0.0 : 0.0) : ldexp(drand48() - 0.5, (int)(drand48() * 70) - 68);
    if (t == 4) x = 5e-324;
    out[0] = std::max(out[0], (double)std::fabs((L)fx_from(x, 60) - std::ldexp((L)x, 60)));
    const i64 X = (i64)ldexp(drand48() - 0.5, (int)(drand48() * 63)) ^ (i64)(lrand48() & 0xff);
    if (X) out[1] = std::max(out[1], (double)std::fabs(((L)fx_to(X, 9) - std::ldexp((L)X, -9)) / std::ldexp((L)X, -9)));
    const i64 c = (i64)ldexp(drand48() - 0.5, 63);
    {
      const L v = std::ldexp((L)X + std::ldexp((L)c, -32), -9);
      // 2^-32 units of the one's complement apart
      const double err = (double)(std::fabs((L)fx_to2<32>(X, c, 9) - v) - std::ldexp((L)1, -41));
      if (v != 0) out[2] = std::max(out[2], err / (double)std::fabs(v));
    }
  }
  if (fx_to(0, 9) != 0.0 || fx_to2<32>(0, 0, 9) != 0.0) out[1] = 1;
}
}
