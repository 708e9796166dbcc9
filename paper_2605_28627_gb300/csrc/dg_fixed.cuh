// Block fixed-point arithmetic for the FP64 operator.
//
// Why: this GPU issues an FP64 instruction of one warp in 67.6 cycles per SM
// sub-partition (measured with a chain of DFMAs), an integer add in 1.1 and a
// 32 x 32 + 64-bit multiply-add (IMAD.WIDE) in 4.0.  A product of two 62-bit
// fixed-point numbers takes three of those and a few adds, 13 cycles in all,
// and a sum two adds, 2.2 cycles.  So the operator's inner sums run on 64-bit
// integers: a quantity q with |q| < 2^e over the element is held as q 2^(Q - e),
// truncated (D: rounded), with the exponents e taken per element from the data
// (fields of one element share an exponent, as the terms that meet in one sum
// do).  The quantisation is 2^-60 of the element's largest value where FP64
// carries 2^-53 of each value; elements whose density or beta varies by more
// than a factor 8 to 16, whose cells are stretched by 4 or more, or that hold a
// non-finite, non-positive or extremely small value, take the FP64 body instead.
//
// Every function is plain integer C++ (host and device), so that the error
// bounds can be checked on the CPU.
#pragma once

#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define DG_HD __host__ __device__ __forceinline__
#else
#include <cmath>
#define DG_HD inline
#endif

namespace dg {

using i64 = long long;
using u64 = unsigned long long;

// A 64-bit number as high and signed low word: value = h 2^32 + l, so that all
// partial products are signed 32 x 32.
struct Fx {
  int h, l;
};
// The products and the word extraction are written in PTX on the device: from
// plain C++ the compiler makes a 64 x 64-bit product (8 instructions, 11.5
// cycles) of what mad.wide does in one instruction of 4 cycles.
DG_HD Fx fx_split(i64 x) {
  Fx r;
#ifdef __CUDA_ARCH__
  asm("mov.b64 {%0, %1}, %2;" : "=r"(r.l), "=r"(r.h) : "l"(x));
  r.h += (int)((unsigned)r.l >> 31);
#else
  r.l = (int)(uint32_t)(u64)x;
  r.h = (int)((u64)x >> 32) + (int)((uint32_t)(u64)x >> 31);
#endif
  return r;
}
DG_HD i64 fx_wide(int a, int b) {
#ifdef __CUDA_ARCH__
  i64 r;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
  return r;
#else
  return (i64)a * b;
#endif
}
DG_HD i64 fx_wide(int a, int b, i64 c) {   // a b + c
#ifdef __CUDA_ARCH__
  i64 r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return (i64)a * b + c;
#endif
}
DG_HD int fx_mulhi(int a, int b) {   // a b / 2^32, rounded down
#ifdef __CUDA_ARCH__
  return __mulhi(a, b);
#else
  return (int)(((i64)a * b) >> 32);
#endif
}
DG_HD int fx_high(i64 x) {   // x / 2^32, rounded down
#ifdef __CUDA_ARCH__
  int l, h;
  asm("mov.b64 {%0, %1}, %2;" : "=r"(l), "=r"(h) : "l"(x));
  return h;
#else
  return (int)(x >> 32);
#endif
}

// Product sums: p collects high * high (weight 2^64), c the cross terms
// (weight 2^32); low * low (at most 2^-2 of the last bit after the division by
// 2^64) is left out.
struct FxSum {
  i64 p, c;
};
template <int K>
DG_HD FxSum fx_zero() {   // with the rounding constant of fx_end<K>
  return FxSum{0, (i64)1 << (31 - K)};
}
DG_HD void fx_add(FxSum& s, Fx a, Fx b) {
  s.p = fx_wide(a.h, b.h, s.p);
  s.c = fx_wide(a.h, b.l, s.c);
  s.c = fx_wide(a.l, b.h, s.c);
}
// sum / 2^(64 - K), rounded
template <int K>
DG_HD i64 fx_end(const FxSum& s) {
  if constexpr (K == 0) return s.p + fx_high(s.c);
  else return (i64)((u64)s.p << K) + (s.c >> (32 - K));
}
template <int K>
DG_HD i64 fx_mul(Fx a, Fx b) {
  FxSum s{fx_wide(a.h, b.h), fx_wide(a.l, b.h, fx_wide(a.h, b.l, (i64)1 << (31 - K)))};
  return fx_end<K>(s);
}

// Moves the whole units of c to p, so that further terms fit in c.
DG_HD void fx_fold(FxSum& s) {
  s.p += fx_high(s.c);
  s.c &= 0xffffffffll;
}
// x 2^k in the bits of a 64-bit word
DG_HD i64 fx_up(i64 x, int k) { return (i64)((u64)x << k); }

DG_HD i64 fx_bits(double x) {
#ifdef __CUDA_ARCH__
  return __double_as_longlong(x);
#else
  i64 b;
  memcpy(&b, &x, 8);
  return b;
#endif
}
DG_HD double fx_from_bits(i64 b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double(b);
#else
  double x;
  memcpy(&x, &b, 8);
  return x;
#endif
}

// x 2^q truncated to an integer, |x 2^q| < 2^62, integer instructions only.
DG_HD i64 fx_from(double x, int q) {
  const i64 b = fx_bits(x);
  const int hi = fx_high(b);
  const u64 m = (((u64)b & 0xfffffffffffffull) | 0x10000000000000ull) << 9;   // 62 bits
  const unsigned r = (unsigned)(1084 - q - ((hi >> 20) & 0x7ff));              // right shift, >= 0
#ifdef __CUDA_ARCH__
  i64 v;
  asm("shr.u64 %0, %1, %2;" : "=l"(v) : "l"(m), "r"(r));                       // 0 for r > 63
#else
  const i64 v = r < 64 ? (i64)(m >> r) : 0;
#endif
  const i64 s = (i64)(hi >> 31);
  return (v ^ s) - s;
}

// x 2^q to the nearest integer, |x 2^q| < 2^61: tables.
DG_HD i64 fx_round(double x, int q) { return (fx_from(x, q + 1) + 1) >> 1; }

// X 2^(-q) as a double, rounded to nearest (ties away; a negative X by at most
// one unit of X more); the result must be normal or zero.
DG_HD double fx_to(i64 x, int q) {
  uint32_t h = (uint32_t)fx_high(x), l = (uint32_t)(u64)x;
  const uint32_t sg = (uint32_t)((int)h >> 31);
  const u64 t = (((u64)(h ^ sg) << 32) | (l ^ sg)) + (sg & 1u);
  h = (uint32_t)(t >> 32);
  l = (uint32_t)t;
  int e = 1085 - q;
  if (h == 0) {
    h = l;
    l = 0;
    e -= 32;
  }
#ifdef __CUDA_ARCH__
  const int z = __clz((int)h);
  const uint32_t nh = __funnelshift_l(l, h, z), nl = z < 32 ? l << z : 0u;
  const uint32_t lo = __funnelshift_r(nl, nh, 11);
#else
  const int z = h ? __builtin_clz(h) : 32;
  const uint32_t nh = z & 31 ? (h << (z & 31)) | (l >> (32 - (z & 31))) : h, nl = z < 32 ? l << z : 0u;
  const uint32_t lo = (nl >> 11) | (nh << 21);
#endif
  const u64 r = ((u64)((nh >> 11) + ((uint32_t)(e - z) << 20)) << 32 | lo) + ((nl >> 10) & 1u);
  return fx_from_bits((i64)(nh ? r | ((u64)(sg & 0x80000000u) << 32) : 0));
}

// (p + c 2^(-CB)) 2^(-q) as a double, rounded (to 2^-96 of the leading bit's
// binade before that); normal or zero.
template <int CB>
DG_HD double fx_to2(i64 p, i64 c, int q) {
  static_assert(CB <= 32, "fraction bits");
  const i64 v = p + (c >> CB);
  uint32_t h = (uint32_t)((u64)v >> 32), l = (uint32_t)(u64)v, f = (uint32_t)(u64)c << (32 - CB);
  const uint32_t sg = (uint32_t)((int)h >> 31);
  h ^= sg;   // one's complement: off by 2^-32 of the unit
  l ^= sg;
  f ^= sg;
  int z0 = 0;
#pragma unroll
  for (int k = 0; k < 2; ++k)
    if (h == 0) {
      h = l;
      l = f;
      f = 0;
      z0 += 32;
    }
#ifdef __CUDA_ARCH__
  const int z = __clz((int)h);
  const uint32_t nh = __funnelshift_l(l, h, z), nl = __funnelshift_l(f, l, z);
#else
  const int z = h ? __builtin_clz(h) : 32;
  const uint32_t nh = z & 31 ? (h << (z & 31)) | (l >> (32 - (z & 31))) : h;
  const uint32_t nl = z & 31 ? (l << (z & 31)) | (f >> (32 - (z & 31))) : l;
#endif
  if (h == 0) return 0.0;
  const u64 n = ((u64)nh << 32) | nl;
  const u64 m = (n >> 11) + ((n >> 10) & 1);
  const u64 bits = ((u64)(uint32_t)(1085 - z - z0 - q) << 52) + m;
  return fx_from_bits((i64)(bits | ((u64)(sg & 0x80000000u) << 32)));
}

DG_HD int fx_clamp(int s) { return s < 0 ? 0 : (s < 63 ? s : 63); }   // a shift count

// Coefficients of f / atanh(f) = 1 - sum b_k u^k and atanh(f) / f = 1 + sum
// u^k / (2k + 1), u = f^2, k = 1.., as fixed point with 62 bits after the
// point (each below 1/2).
constexpr int kFxTerms = 14;
struct FxSeries {
  i64 b[kFxTerms], a[kFxTerms];
};
constexpr FxSeries fx_series() {
  FxSeries s{};
  double b[kFxTerms + 1] = {};
  for (int k = 1; k <= kFxTerms; ++k) {
    // (sum u^j / (2j + 1)) (1 - sum b_j u^j) = 1
    double v = 1.0 / (2 * k + 1);
    for (int j = 1; j < k; ++j) v -= b[j] / (2 * (k - j) + 1);
    b[k] = v;
    s.b[k - 1] = (i64)(v * 4611686018427387904.0);
    s.a[k - 1] = (i64)(4611686018427387904.0 / (2 * k + 1));
  }
  s.b[0] = s.a[0] = (i64)(4611686018427387904ull / 3);
  return s;
}
#ifdef __CUDACC__
__constant__ const FxSeries kFxSeries = fx_series();
#else
static const FxSeries kFxSeries = fx_series();
#endif

// Exponents of one element: |quantity| < 2^e at all of its nodes, and the
// largest value's logarithm less e (in -1..0, rounded up).
struct FxExp {
  int r, u, b;      // density, velocity components, beta / 4
  int j;            // sum over l of |J a^d_l|, every direction d
  float lr, lu, lj;
  float lb;         // smallest b over 2^e_b, logarithm rounded down
};
// Bits after the binary point of the node data: density, velocity, b and metric
// terms at 60 - e, |u|^2 at 58 - 2 e_u.  Smallest admitted density and b as
// integers: 2^56.
constexpr int kFxQ = 60;

// Shifts of the two-point flux (per element): up by k*, so that the factors of
// the next product fill 62 bits whatever the element's values (sums of few
// products then lose little to rounding), down by s* to align two terms (one
// of each two is zero); bits after the point of the five components, as summed
// with D at 60 - e_D and with the factors 1/4, 1/8, 1/16 of D taken in (see
// fx_pair).
struct alignas(16) FxAlign {
  int ky, ku, kx, k4;       // 1/(b_a + b_b), {u}.n, xf and y4 in the momentum flux
  int ke, kz, sm1, sm2;     // xf and the bracket in the energy flux
  int sz1, sz2, se1, se2;
  int q0, qm, qe, pad;
};
// Bits of D, less e_D (with 58, truncated, the representation of D was the
// largest error of R; 61 would let the sums of nine terms overflow), and what
// line sums shift up by to keep 62 - e_D as their scale.
constexpr int kFxQD = 60;
constexpr int kFxUpD = 62 - kFxQD;
DG_HD int fx_floor(float x) { return (int)x - (x < (float)(int)x ? 1 : 0); }
DG_HD float fx_log2_sum(float a, float b) {   // log2(2^a + 2^b), rounded up
  const float m = a > b ? a : b, d = a > b ? b - a : a - b;
  return m + (d < -20.0f ? 0.01f : log2f(1.0f + exp2f(d)) + 0.001f);
}
DG_HD FxAlign fx_align(const FxExp& e, int eg, float lg, int eD) {
  FxAlign a;
  a.pad = 0;
  const float lr = 60.0f + e.lr, lu = 60.0f + e.lu, lj = 60.0f + e.lj;   // logarithms of the largest integers
  float ly = 118.0f - (60.0f + e.lb);                                     // 1/(b_a + b_b)
  a.ky = fx_clamp(fx_floor(62.0f - ly));
  ly += a.ky;
  float lun = lu + lj + 2.0f - 64.0f;
  a.ku = fx_floor(62.0f - lun);
  lun += a.ku;
  const float lx = lr + 1.0f + lun - 64.0f, l4 = lr + 1.0f + ly - 64.0f;
  a.kx = fx_floor(61.5f - lx);
  a.k4 = fx_floor(61.5f - l4);
  const int qx = 52 + a.ku;                                                // xf, + (-e_r - e_u - e_j)
  const int m1 = qx + a.kx - 4 - 2 * e.u, m2 = 51 + a.ky + a.k4 + e.b;    // Xf su, Y4 sn, + (-e_r - e_j)
  const int qm = (m1 < m2 ? m1 : m2) + 1;            // fx_end<1>
  a.sm1 = fx_clamp(m1 - m2);
  a.sm2 = fx_clamp(m2 - m1);
  const int z1 = 57 + a.ky + e.b - eg, z2 = 58 - 2 * e.u;
  const int qz = z1 < z2 ? z1 : z2;
  a.sz1 = fx_clamp(z1 - z2);
  a.sz2 = fx_clamp(z2 - z1);
  const float lz = fx_log2_sum(ly + 62.0f + lg - 64.0f + 0.1f - a.sz1, 58.0f + 2.0f * e.lu + 2.6f - a.sz2);
  a.ke = fx_floor(62.0f - lx);
  a.kz = fx_clamp(fx_floor(62.0f - lz));
  const int e1 = qx + a.ke + qz + a.kz - 64, e2 = qm - 1;   // Xf Z and su . M (fx_end<3>), + (-e_r - e_u - e_j)
  a.se1 = fx_clamp(e1 - e2);
  a.se2 = fx_clamp(e2 - e1);
  // bound of the energy flux: Xf Z, and su . M = Xf |su|^2 + Y4 su . sn; kept below 2^60.4
  const float b1 = lx + a.ke + lz + a.kz - 64.0f - a.se1;
  const float b2 = fx_log2_sum(lx + a.kx - a.sm1 + 2.0f * lu + 3.6f, l4 + a.k4 - a.sm2 + lu + lj + 2.0f) - 124.0f - a.se2;
  const float over = fx_log2_sum(b1, b2) - 60.4f;
  const int down = over > 0.0f ? fx_floor(over) + 1 : 0;
  a.se1 = fx_clamp(a.se1 + down);
  a.se2 = fx_clamp(a.se2 + down);
  const int qe = (e1 < e2 ? e1 : e2) - down;
  a.q0 = qx - e.r - e.u - e.j + kFxQD - eD - 64 + 2;
  a.qm = qm - e.r - e.j + kFxQD - eD - 64 + 3;
  a.qe = qe - e.r - e.u - e.j + kFxQD - eD - 64 + 4;
  return a;
}

// y = 2^119 / S to a relative error below 2^-50 (S in [2^57, 2^61)): hardware
// reciprocal of the high word, one cubic step on integers.
DG_HD i64 fx_rcp(Fx S) {
#ifdef __CUDA_ARCH__
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__int2float_rn(S.h)));
  const int Y = __float2int_rn(y * 36028797018963968.0f);   // 2^55 / S.h, 24 bits
#else
  const int Y = (int)lrintf((1.0f / (float)S.h) * 36028797018963968.0f);
#endif
  const i64 t = fx_wide(S.h, Y, (i64)fx_mulhi(S.l, Y));
  const int e = -(int)(t >> 4);                            // (1 - S Y / 2^87) 2^51, |.| < 2^30 (2^51 drops out)
  const i64 w = fx_wide(Y, e + (fx_mulhi(e, e) >> 19)) >> 19;               // Y (e + e^2)
  return w + (i64)((u64)(uint32_t)Y << 32);
}
// one more step from the low words of S y: relative error below 2^-55
DG_HD i64 fx_rcp_full(Fx S, i64 y) {
  const Fx Y = fx_split(y);
  const u64 c = (u64)fx_wide(S.l, Y.h, fx_wide(S.h, Y.l));
  const u64 E = c + ((u64)((uint32_t)S.h * (uint32_t)Y.h) << 32);   // (S y / 2^119 - 1) 2^87
  const int e = -(int)((i64)E >> 6);
  return y + (fx_mulhi(Y.h, e) >> 17);
}

// Series of 1 - f/atanh(f) (INV) or atanh(f)/f - 1 in u = f^2 < 2^-8, 64 bits
// after the point; U = u 2^56.  v = u (a1 + u (a2 + u t)), t = a3 + .. + a6 u^3
// on 32 bits (33 after the point; its error enters as u^3 2^-33), truncation
// below 2^-59.
template <bool INV>
DG_HD i64 fx_series_sum(i64 U) {
  constexpr FxSeries S = fx_series();
  const i64* A = INV ? S.b : S.a;
  const int a3 = (int)(A[2] >> 29), a4 = (int)(A[3] >> 29), a5 = (int)(A[4] >> 29), a6 = (int)(A[5] >> 29);
  const int u32 = (int)(U >> 24), u39 = (int)(U >> 17);
  int t = a5 + fx_mulhi(u32, a6);
  t = a4 + fx_mulhi(u32, t);
  t = a3 + fx_mulhi(u32, t);
  const i64 h = (A[1] >> 2) + (fx_wide(u39, t) >> 12);      // 60 bits
  const Fx u = fx_split(fx_up(U, 10));               // 66 bits
  const i64 g = A[0] + fx_mul<0>(u, fx_split(h));           // 62 bits
  return fx_mul<0>(u, fx_split(g));
}
// The same for 2^-8 <= u < 2^-4: Horner's rule with 14 terms on 62 bits.
template <bool INV>
DG_HD i64 fx_series_long(i64 U) {
  const Fx u = fx_split(fx_up(U, 8));                // 64 bits
  const i64* c = INV ? kFxSeries.b : kFxSeries.a;
  i64 g = c[kFxTerms - 1];
#ifdef __CUDA_ARCH__
#pragma unroll 1
#endif
  for (int k = kFxTerms - 2; k >= 0; --k) g = c[k] + fx_mul<0>(u, fx_split(g));
  return fx_up(fx_mul<0>(u, fx_split(g)), 2);
}

// Means of a pair whose density or beta ratio is large (u >= 2^-8): series to
// u = 2^-4, beyond that atanh(f)/f by log(a, b).
struct FxMeans {
  i64 rln2, hib;
};
template <class LOG>
DG_HD FxMeans fx_means_long(i64 ra, i64 rb, i64 ba, i64 bb, i64 yb, i64 Ur, i64 Ub, LOG log) {
  const i64 sr = ra + rb, top = (i64)1 << 52;
  FxMeans m;
  m.rln2 = Ur < top ? sr - fx_mul<0>(fx_split(sr), fx_split(fx_series_long<true>(Ur)))
                    : fx_from((double)sr / log((double)ra, (double)rb), 0);
  m.hib = Ub < top ? yb + fx_mul<0>(fx_split(yb), fx_split(fx_series_long<false>(Ub)))
                   : fx_from((double)yb * log((double)ba, (double)bb), 0);
  return m;
}

// Two-point flux in fixed point (Chandrashekar 2013), the FP64 flux of ec_pair
// with F = (8 f_rho, 16 f_m, 32 f_E): rho, b = beta/4, velocities, |u|^2 and
// metric terms of both nodes as integers (see FxExp), G = 1/(gamma - 1) with
// 62 - e_g bits; LONG evaluates fx_means_long.
// Bounds: sums of two velocities and of two metric terms are below 2^61 (the
// latter also summed over l), so a product sum stays below 2^63 in p and c; xf
// stays below 2^59, M below 2^60 and E below 2^60.4, so that nine terms of a row of D,
// with 60 - e_D bits, fit in c between two fx_fold.  Factors are shifted up
// before a product rather than the product after it, where the low * low part
// that fx_add leaves out would count.
template <class LONG>
DG_HD void fx_pair(i64 ra, i64 rb, i64 ba, i64 bb, i64 su0, i64 su1, i64 su2, i64 sk, i64 sn0, i64 sn1, i64 sn2,
                   Fx G, const FxAlign& al, i64 F[5], LONG means_long) {
  const i64 sr = ra + rb;
  const Fx Sr = fx_split(sr), Sb = fx_split(ba + bb);
  const i64 yr = fx_rcp(Sr);
  const i64 yb0 = fx_rcp_full(Sb, fx_rcp(Sb));
  // f = difference / sum, 60 bits after the point, and u = f^2, 56
  const Fx fr = fx_split(fx_up(fx_mul<0>(fx_split(ra - rb), fx_split(yr)), 5));
  const Fx fb = fx_split(fx_up(fx_mul<0>(fx_split(ba - bb), fx_split(yb0)), 5));
  const i64 Ur = fx_mul<0>(fr, fr), Ub = fx_mul<0>(fb, fb);
  const i64 yb = fx_up(yb0, al.ky);                                  // 59 + k_y + e_b
  const Fx Yb = fx_split(yb);
  FxMeans mn;                    // 2 rho_ln (60 - e_r) and 2 / beta_ln (59 + k_y + e_b)
  if (fx_high(Ur | Ub) < (1 << 16)) {
    mn.rln2 = sr - fx_mul<0>(Sr, fx_split(fx_series_sum<true>(Ur)));
    mn.hib = yb + fx_mul<0>(Yb, fx_split(fx_series_sum<false>(Ub)));
  } else {
    mn = means_long(ra, rb, ba, bb, yb, Ur, Ub);
  }
  const Fx U0 = fx_split(su0), U1 = fx_split(su1), U2 = fx_split(su2);
  const Fx N0 = fx_split(sn0), N1 = fx_split(sn1), N2 = fx_split(sn2);
  FxSum w = fx_zero<0>();
  fx_add(w, U0, N0);
  fx_add(w, U1, N1);
  fx_add(w, U2, N2);
  const i64 xf = fx_mul<0>(fx_split(mn.rln2), fx_split(fx_up(fx_end<0>(w), al.ku)));   // 52 + k_u - e_r - e_u - e_j
  const i64 y4 = fx_mul<0>(Sr, Yb);                                  // 55 + k_y - e_r + e_b
  const Fx X = fx_split(fx_up(xf, al.kx) >> al.sm1), Y = fx_split(fx_up(y4, al.k4) >> al.sm2);
  F[0] = xf;
  FxSum m0 = fx_zero<1>(), m1 = fx_zero<1>(), m2 = fx_zero<1>();
  fx_add(m0, X, U0);
  fx_add(m0, Y, N0);
  fx_add(m1, X, U1);
  fx_add(m1, Y, N1);
  fx_add(m2, X, U2);
  fx_add(m2, Y, N2);
  F[1] = fx_end<1>(m0);
  F[2] = fx_end<1>(m1);
  F[3] = fx_end<1>(m2);
  const i64 z = (fx_mul<0>(fx_split(mn.hib), G) >> al.sz1) - (sk >> al.sz2);   // 57 + k_y + e_b - e_g
  const i64 ea = fx_mul<0>(fx_split(fx_up(xf, al.ke)), fx_split(fx_up(z, al.kz)));
  FxSum b = fx_zero<3>();
  fx_add(b, U0, fx_split(F[1]));
  fx_add(b, U1, fx_split(F[2]));
  fx_add(b, U2, fx_split(F[3]));
  F[4] = (ea >> al.se1) + (fx_end<3>(b) >> al.se2);
}

// Lifting on LGL nodes.  Line sum D phi + jump of a field with exponent e (D and
// the jump factor with 60 - e_D bits, fields with 60 - e): 60 - e - e_D bits,
// below 2^62.1 for N <= 9.  Gradient component (1/J) sum_d Ja^d dd_d: the sum,
// with metric terms of 60 - e_j bits, has 58 - e - e_D - e_j bits and stays
// below 2^61.6, its product with 1/J (62 - e_i) 58 - e - e_D - e_j - e_i.  The
// shifts fill the words: with 3 bits less (as the bound of the single factors
// leaves) the products' rounding was up to 3 times the FP64 kernel's at N = 7.
constexpr int kFxUpLift = kFxUpD + 2;
DG_HD FxSum fx_lift_start(i64 jump) { return FxSum{jump, (i64)1 << (31 - kFxUpLift)}; }
DG_HD i64 fx_lift_line(const FxSum& s) { return fx_end<kFxUpLift>(s); }
DG_HD int fx_lift_bits(int eD, int ej, int ei) { return 58 - eD - ej - ei; }   // less e
DG_HD i64 fx_lift_gradient(const Fx J[3], const Fx dd[3], Fx iJ) {
  FxSum s = fx_zero<2>();
  fx_add(s, J[0], dd[0]);
  fx_add(s, J[1], dd[1]);
  fx_add(s, J[2], dd[2]);
  return fx_mul<2>(fx_split(fx_end<2>(s)), iJ);
}

// Weak lifting: line sums of n + 2 products of 60 bits, shifted up so that the
// three directions' sum (59 - e - e_D - e_j bits) stays below 2^61.8 for N <= 9.
constexpr int kFxUpWeak = kFxUpD + 1;

}  // namespace dg
