// Volume body of the FP64 operator in block fixed point (dg_fixed.cuh): the
// same terms as volume_body<N, double>, with the viscous fluxes, the two-point
// fluxes and all line sums on 64-bit integers.  The primitives of a node (18
// FP64 operations), the surface term, the source and the Runge-Kutta update
// stay FP64: they run on the FP64 pipe beside the integer work of other warps.
//
// Integer sums do not depend on their order, so every tile shape gives the
// same bits.  Elements outside the fixed-point range (FxExp, s_state = 2) are
// left to volume_body<N, double>, which the caller runs after this one.
//
// Bound and measured: the FP64 body held the FP64 pipe 90 % busy (834 FP64
// instructions a node at N = 7, 67.6 cycles each); here a pair costs about 330
// instructions and 445 cycles of the integer multiplier (quarter rate), and a
// node about 70 FP64 instructions.  Neither pipe is full (issue slots and
// multiplier 49 and 50 % busy at N = 7): barriers and the latency of the FP64 prologue
// and epilogue hold it.  Manufactured solution, 16^3 elements, us per launch
// before -> now: N = 1 41 -> 25, 2 146 -> 55, 3 295 -> 92, 4 655 -> 182, 5 1293
// -> 356, 6 2239 -> 607, 7 3533 -> 1010, 8 5822 -> 1843, 9 8806 -> 3130.
#pragma once

#include "dg_fx_metrics.cuh"
#include "dg_stage.cuh"

namespace dg {

// Blocks per SM that the registers and shared memory must allow: about 24
// warps per SM at 80 registers for N <= 5 (N = 3: 88 us against 93 with 16 warps
// and 128 registers and 103 with 32 warps and 64), two blocks for N = 6 and 7,
// where 800 bytes of spilled registers cost less than half the warps (N = 7: 991
// us against 1222 with one block and no spills).
template <int N>
constexpr int fx_min_blocks() {
  constexpr int threads = Shape<N>::THREADS;
  return threads <= 512 ? (768 / threads > 1 ? 768 / threads : 2) : 1;
}

// Shared memory: the Fx table of D (60 - e_D bits), then per element, in words
// of 8 bytes: (rho, b), (|u|^2, u), (v, w) as pairs (6 P), the viscous sums (4
// P), and the metric terms of the three directions as a pair and a single with
// the exchange buffers (pairs F0 F1, F2 F3 and F4), which the viscous fluxes
// (12 P) use first.  Pairs are moved by 16-byte accesses; an odd P is padded.
template <int N>
struct FxBuf {
  static constexpr int P = (N + 1) * (N + 1) * (N + 1), PW = P + (P & 1), ROUNDS = (N + 1) / 2, EPB = Shape<N>::EPB,
                       MINB = fx_min_blocks<N>();
  static constexpr size_t budget = (226 * 1024) / MINB - 2048;
  static constexpr size_t tables = ((N + 1) * (N + 1) + 1) & ~1;
  static constexpr int JW = 2 * P + PW, XW = 4 * P + PW;   // words of one direction's metric terms, of one buffer
  static constexpr int words(int xb) { return 10 * P + 3 * JW + xb * XW; }
  static constexpr int value = 8 * (tables + (size_t)EPB * words(ROUNDS)) <= budget ? ROUNDS : 1;
  static constexpr int PER_ELEM = words(value);
};
template <int N, int EPB>
constexpr size_t volume_fx_smem_bytes() {
  return 8 * (FxBuf<N>::tables + (size_t)EPB * FxBuf<N>::PER_ELEM);
}

// atanh(f)/f for large ratios, on the FP64 pipe.
struct FxLog {
  __device__ double operator()(double a, double b) const { return atanh_ratio_log<double>(a, b); }
};

// Means of pairs with large ratios, out of line.
struct FxLong {
  static __device__ __noinline__ FxMeans run(i64 ra, i64 rb, i64 ba, i64 bb, i64 yb, i64 Ur, i64 Ub) {
    return fx_means_long(ra, rb, ba, bb, yb, Ur, Ub, FxLog());
  }
  __device__ FxMeans operator()(i64 ra, i64 rb, i64 ba, i64 bb, i64 yb, i64 Ur, i64 Ub) const {
    return run(ra, rb, ba, bb, yb, Ur, Ub);
  }
};

// Exponents of one element from the maxima gathered in s_mx: high words of the
// largest density, b, velocity component and gradients, complements of the
// smallest density and b; metric terms from the set-up (ej: 2^(e_j) and the
// logarithm less e_j).
enum { kMxR, kMxRmin, kMxB, kMxBmin, kMxU, kMxG, kMxT, kMxCount };
struct FxElem {
  FxExp e;
  int g, t;   // velocity and temperature gradients
  bool ok;
};
__device__ __forceinline__ FxElem fx_element(const int* mx, float4 ej) {
  FxElem x;
  const int r = mx[kMxR], rmin = 0x7fffffff - mx[kMxRmin], b = mx[kMxB], bmin = 0x7fffffff - mx[kMxBmin];
  x.e.r = (r >> 20) - 1022;
  x.e.b = (b >> 20) - 1022;
  const int dr = x.e.r - ((rmin >> 20) - 1023), db = x.e.b - ((bmin >> 20) - 1023);
  x.e.u = fx_expo(mx[kMxU]);
  x.e.j = (int)ej.x;
  x.g = fx_expo(mx[kMxG]);
  x.t = fx_expo(mx[kMxT]);
  auto in = [](int v) { return v > -90 && v < 90; };
  x.ok = rmin > 0 && bmin > 0 && dr <= 4 && db <= 4 && in(x.e.r) && in(x.e.b) && in(x.e.j) &&
         fx_in_range(mx[kMxU], 90) && fx_in_range(mx[kMxG], 90) && fx_in_range(mx[kMxT], 90);
  x.e.lr = x.e.lu = x.e.lj = x.e.lb = 0.0f;
  return x;
}
// the logarithms too (one thread per element)
__device__ __forceinline__ void fx_element_logs(FxElem& x, const int* mx, float4 ej) {
  const int bmin = 0x7fffffff - mx[kMxBmin];
  x.e.lr = fx_log_mantissa(mx[kMxR], 1);
  x.e.lu = mx[kMxU] != 0 ? fx_log_mantissa(mx[kMxU], 1) : 0.0f;
  x.e.lj = ej.y;
  x.e.lb = fx_log_mantissa(bmin, 0) + (float)((bmin >> 20) - 1022 - x.e.b);
}

// s / 2^t of a viscous line sum, 0 <= t <= 15.
__device__ __forceinline__ void fx_visc_down(FxSum& s, int t) {
  s.c = (s.c >> t) + ((s.p & ((1 << t) - 1)) << (32 - t));
  s.p >>= t;
}

// Returns whether the block holds elements that this body left to FP64
// (s_state[le] = 2); all threads return the same value.
// STRETCH: the mesh may hold elements whose directions' metric terms are shifted
// by different amounts (FxMetricShifts::t); without it every t is 0.
template <int N, int EPB_, bool LIST, bool STRETCH>
__device__ __forceinline__ bool volume_body_fx(const StageArgs& a, const double* __restrict__ metrics,
                                               const i64* __restrict__ jx, const float4* __restrict__ ejx,
                                               const double* __restrict__ grad, const double* __restrict__ fstar,
                                               const int* __restrict__ elem_face, const double* __restrict__ mms,
                                               const double* __restrict__ Dg, int E, const Gas& g, double inv_w0,
                                               int blk, int* s_state) {
  using S = VShape<N, EPB_>;
  constexpr int n = S::n, P = S::P, NN = S::NN, EPB = S::EPB, eD = fx_eD(N);
  using B = FxBuf<N>;
  constexpr int XB = B::value, PER_ELEM = B::PER_ELEM, JW = B::JW, XW = B::XW;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Fx* sD = reinterpret_cast<Fx*>(smem_raw);
  i64* const tile0 = reinterpret_cast<i64*>(smem_raw) + B::tables;
  __shared__ int s_mx[EPB][kMxCount];
  __shared__ FxAlign s_al[EPB];
  __shared__ int s_walk[EPB], s_shift[EPB];      // FxMetricShifts
  __shared__ Fx s_G;
  __shared__ double s_tc[2];                     // sin, cos of pi t (manufactured source)
  __shared__ uint64_t s_bar[EPB];
  const int le = threadIdx.x / P, id = threadIdx.x - le * P;
  i64* base = tile0 + le * PER_ELEM;
  longlong2* sN = reinterpret_cast<longlong2*>(base);   // [3][P] (rho, b), (|u|^2, u), (v, w)
  double* sA = reinterpret_cast<double*>(base + 6 * P); // [4][P] viscous sums
  i64* sJ = base + 10 * P;                       // [3]: (J0, J1) [P], J2 [P]
  i64* sX = sJ + 3 * JW;                         // [XB]: (F0, F1) [P], (F2, F3) [P], F4 [P]
  i64* sFv = sJ;                                 // [3][4][P]
  int nslot = E, e = blk * EPB + le;
  if constexpr (LIST) {
    nslot = *a.list_len;
    e = e < nslot ? a.list[e] : E;
    if constexpr (EPB == 1) {
      if (e >= E) return false;   // the whole block, before any barrier
    }
  }
  const bool active = e < E;
  const int eg = ((__double2hiint(g.inv_gm1) >> 20) & 0x7ff) - 1022;
  if (threadIdx.x == 0) {
    if (g.source == DG_SOURCE_MMS) sincospi(a.clock[0] + a.c_stage * a.clock[1], &s_tc[0], &s_tc[1]);
    s_G = fx_split(fx_from(g.inv_gm1, 62 - eg));
  }
  // operands read after the sweeps, asked for in L2 now (as in volume_body)
  if (active && id < 9) {
    if (id == 0 && a.mode == 1 && a.A != 0.0) l2_prefetch(a.Gk + (size_t)e * 5 * P, 5 * P * sizeof(double));
    else if (id == 1) l2_prefetch(metrics + (size_t)e * 10 * P + 9 * P, P * sizeof(double));
    else if (id == 2 && g.source == DG_SOURCE_MMS) l2_prefetch(mms + (size_t)e * 2 * P, 2 * P * sizeof(double));
    else if (id >= 3)
      l2_prefetch(fstar + (size_t)dg_idx(elem_face[e * 6 + id - 3] >> 4, a.nfaces > 0 ? a.nfaces : 3L * E,
                                         kSiteVolFace) * 5 * NN,
                  5 * NN * sizeof(double));
  }
  for (int t = threadIdx.x; t < n * n; t += blockDim.x) {
    const double d = Dg[t];
    // the corners carry the viscous part of the surface term, as in volume_body
    sD[t] = fx_split(fx_round(t == 0 ? d + inv_w0 : (t == n * n - 1 ? d - inv_w0 : d), kFxQD - eD));
  }
  for (int t = threadIdx.x; t < EPB * kMxCount; t += blockDim.x) s_mx[t / kMxCount][t % kMxCount] = 0;
  // state by bulk copy into the region of the metric terms and fluxes
  if (active && id == 0) {
    const double* src = a.U + (size_t)e * 5 * P;
    bulk_bar_init(&s_bar[le]);
    bulk_expect(&s_bar[le], bulk_middle_bytes(src, 5 * P));
    bulk_stage_range(bulk_stage_ptr(reinterpret_cast<double*>(sJ), src), src, 5 * P, &s_bar[le]);
  }
  i64 Ja[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
  double gr[12] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
  if (active) {
    if (jx != nullptr) {
      const i64* mt = jx + (size_t)e * 10 * P + id;
#pragma unroll
      for (int r = 0; r < 9; ++r) Ja[r] = mt[r * P];
    }
    const double* gg = grad + (size_t)e * 12 * P + id;
#pragma unroll
    for (int r = 0; r < 12; ++r) gr[r] = gg[r * P];
  }
  __syncthreads();
  double q[5] = {0, 0, 0, 0, 0};
  double rho = 1, u = 0, v = 0, w = 0, bt = 1, kk = 0;
  if (active) {
    bulk_wait(&s_bar[le], 0);
    const double* st = bulk_stage_ptr(reinterpret_cast<double*>(sJ), a.U + (size_t)e * 5 * P);
#pragma unroll
    for (int r = 0; r < 5; ++r) q[r] = st[r * P + id];
    rho = q[0];
    const double ir = rcp_op(rho);
    u = q[1] * ir; v = q[2] * ir; w = q[3] * ir;
    kk = u * u + v * v + w * w;
    const double p = g.gm1 * fma(-0.5 * rho, kk, q[4]);
    bt = 0.125 * rho * rcp_op(p);   // beta / 4
    if (g.visc_law == DG_VISC_SUTHERLAND) {
      const double sf = visc_factor<double>(g, p * ir * g.inv_R);
#pragma unroll
      for (int r = 0; r < 12; ++r) gr[r] *= sf;
    }
    // maxima over the element, on the high words (monotonic in the magnitude;
    // non-finite values end above every finite one)
    auto mag = [](double x) { return __double2hiint(x) & 0x7fffffff; };
    auto mag2 = [&](double x, double y) { return max(mag(x), mag(y)); };
    int mx[kMxCount];
    const int hr = __double2hiint(rho), hb = __double2hiint(bt);
    mx[kMxR] = max(hr, 0);
    mx[kMxRmin] = 0x7fffffff - max(hr, 0);
    mx[kMxB] = max(hb, 0);
    mx[kMxBmin] = 0x7fffffff - max(hb, 0);
    mx[kMxU] = max(mag2(u, v), mag(w));
    mx[kMxG] = max(max(mag2(gr[0], gr[1]), mag2(gr[2], gr[3])),
                   max(max(mag2(gr[4], gr[5]), mag2(gr[6], gr[7])), mag(gr[8])));
    mx[kMxT] = max(mag2(gr[9], gr[10]), mag(gr[11]));
    const unsigned lanes = __match_any_sync(__activemask(), le);
    const bool first = (int)(threadIdx.x & 31) == __ffs(lanes) - 1;
#pragma unroll
    for (int m = 0; m < kMxCount; ++m) {
      const unsigned r = __reduce_max_sync(lanes, (unsigned)mx[m]);
      if (first) atomicMax(&s_mx[le][m], (int)r);
    }
  }
  __syncthreads();   // maxima complete; every node has its state: the staging region is free
  if (active && id == 0) bulk_bar_inval(&s_bar[le]);
  const float4 ej = active ? ejx[e] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  const FxMetricShifts sh = fx_shifts(ej);
  FxElem ex = fx_element(s_mx[le], ej);
  const bool act = active && ex.ok;
  if (id == 0) {
    s_state[le] = active ? (ex.ok ? 1 : 2) : 0;
    if (act) {
      fx_element_logs(ex, s_mx[le], ej);
      s_al[le] = fx_align(ex.e, eg, fx_log_mantissa(__double2hiint(g.inv_gm1), 1), eD);
    }
    if constexpr (STRETCH) {
      s_walk[le] = sh.walk();
      s_shift[le] = sh.w;
    }
  }
  if (act) {
    const i64 xu = fx_from(u, kFxQ - ex.e.u), xv = fx_from(v, kFxQ - ex.e.u), xw = fx_from(w, kFxQ - ex.e.u);
    sN[id] = make_longlong2(fx_from(rho, kFxQ - ex.e.r), fx_from(bt, kFxQ - ex.e.b));
    sN[P + id] = make_longlong2(fx_from(kk, kFxQ - 2 - 2 * ex.e.u), xu);
    sN[2 * P + id] = make_longlong2(xv, xw);
    const Fx U[3] = {fx_split(xu), fx_split(xv), fx_split(xw)};
    // stress over mu: 59 - e_g bits, below 2^60.4; heat flux over mu: 60 - e_t - e_k bits
    i64 G[9];
#pragma unroll
    for (int r = 0; r < 9; ++r) G[r] = fx_from(gr[r], 59 - ex.g);
    const Fx twothird{715827883, -1431655765};   // 2^62 2/3 / 2^32 and the low word of 2^62 2/3
    const i64 div = fx_mul<2>(fx_split(G[0] + G[4] + G[8]), twothird);
    const Fx t00 = fx_split(2 * G[0] - div), t11 = fx_split(2 * G[4] - div), t22 = fx_split(2 * G[8] - div);
    const Fx t01 = fx_split(G[1] + G[3]), t02 = fx_split(G[2] + G[6]), t12 = fx_split(G[5] + G[7]);
    const int ek = ((__double2hiint(g.kappa) >> 20) & 0x7ff) - 1022;
    const Fx kap = fx_split(fx_from(g.kappa, kFxQ - ek));
    Fx T[3];
#pragma unroll
    for (int l = 0; l < 3; ++l) T[l] = fx_split(fx_mul<4>(fx_split(fx_from(gr[9 + l], kFxQ - ex.t)), kap));
    const int q1 = 56 - ex.g - ex.e.u, q2 = 59 - ex.t - ek;   // of the energy flux's two terms, + (-e_j + t_d)
    if constexpr (STRETCH) {
#pragma unroll
      for (int r = 0; r < 9; ++r) Ja[r] = fx_up(Ja[r], sh.t(r / 3));
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      Fx J[3];
#pragma unroll
      for (int l = 0; l < 3; ++l) J[l] = fx_split(Ja[d * 3 + l]);
      FxSum f0 = fx_zero<3>(), f1 = fx_zero<3>(), f2 = fx_zero<3>(), h = fx_zero<3>(), en = fx_zero<2>();
      fx_add(f0, t00, J[0]); fx_add(f0, t01, J[1]); fx_add(f0, t02, J[2]);
      fx_add(f1, t01, J[0]); fx_add(f1, t11, J[1]); fx_add(f1, t12, J[2]);
      fx_add(f2, t02, J[0]); fx_add(f2, t12, J[1]); fx_add(f2, t22, J[2]);
      fx_add(h, T[0], J[0]); fx_add(h, T[1], J[1]); fx_add(h, T[2], J[2]);
      const i64 v0 = fx_end<3>(f0), v1 = fx_end<3>(f1), v2 = fx_end<3>(f2);   // 58 - e_g - e_j + t_d
      fx_add(en, fx_split(v0), U[0]); fx_add(en, fx_split(v1), U[1]); fx_add(en, fx_split(v2), U[2]);
      i64 ve = fx_end<2>(en), vh = fx_end<3>(h);
      ve >>= fx_clamp(q1 - q2);
      vh >>= fx_clamp(q2 - q1);
      sFv[(d * 4 + 0) * P + id] = v0;
      sFv[(d * 4 + 1) * P + id] = v1;
      sFv[(d * 4 + 2) * P + id] = v2;
      sFv[(d * 4 + 3) * P + id] = ve + vh;
    }
  }
  __syncthreads();
  const int i = id % n, j = (id / n) % n, k = id / NN;
  const int ijk[3] = {i, j, k};
  if (act) {
    // viscous line sums (with the viscous part of the surface term)
    const int ek = ((__double2hiint(g.kappa) >> 20) & 0x7ff) - 1022;
    const int q1 = 56 - ex.g - ex.e.u, q2 = 59 - ex.t - ek;
    const int qv = kFxQD - 6 - ex.g - ex.e.j - eD, qe = (q1 < q2 ? q1 : q2) - (64 - kFxQD) - ex.e.j - eD;
#pragma unroll 1
    for (int c = 0; c < 4; ++c) {
      i64 p = 0, f = 0;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const int r = ijk[d];
        const int stride = d == 0 ? 1 : (d == 1 ? n : NN);
        const i64* line = sFv + (d * 4 + c) * P + id - r * stride;
        FxSum s{STRETCH ? 0 : p, 0};
#pragma unroll
        for (int m = 0; m < n; ++m) fx_add(s, sD[r * n + m], fx_split(line[m * stride]));
        if constexpr (STRETCH) {
          if (const int t = FxMetricShifts{s_shift[le]}.t(d)) fx_visc_down(s, t);
          p += s.p;
        } else {
          p = s.p;
        }
        f += s.c >> 2;
      }
      sA[c * P + id] = fx_to2<30>(p, f, c < 3 ? qv : qe);
    }
  }
  __syncthreads();   // every line sum has read the viscous fluxes
  if (act) {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      reinterpret_cast<longlong2*>(sJ + d * JW)[id] = make_longlong2(Ja[d * 3], Ja[d * 3 + 1]);
      sJ[d * JW + 2 * P + id] = Ja[d * 3 + 2];
    }
  }
  __syncthreads();

  // two-point fluxes: the pair rounds and exchange groups of volume_body
  FxSum acc[5] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}, {0, 0}};
  constexpr int FULL = (n - 1) / 2;
  constexpr bool HALF = (n % 2) == 0;
  constexpr int SCOPE = (n == 8 && EPB == 1) ? 2 : ((P % 32 == 0 && EPB > 1 && EPB <= 15) ? 1 : 0);
  auto dsync = [&](int dd) {
    if constexpr (SCOPE == 2) {
      if (dd < 2) bar_sync_reg(1 + (threadIdx.x >> 6), 64);
      else __syncthreads();
    } else if constexpr (SCOPE == 1) {
      bar_sync<EPB>(1 + le, P);
    } else {
      __syncthreads();
    }
  };
  // flux of the pair (ia, ib) of the element at b2
  auto pair = [&](const i64* b2, int el, int d, int ia, int ib, i64 F[5]) {
    const longlong2* nd = reinterpret_cast<const longlong2*>(b2);
    const i64* jd = b2 + 10 * P + d * JW;
    const longlong2* jp = reinterpret_cast<const longlong2*>(jd);
    const longlong2 r0 = nd[ia], r1 = nd[ib], k0 = nd[P + ia], k1 = nd[P + ib], v0 = nd[2 * P + ia], v1 = nd[2 * P + ib];
    const longlong2 j0 = jp[ia], j1 = jp[ib];
    fx_pair(r0.x, r1.x, r0.y, r1.y, k0.y + k1.y, v0.x + v1.x, v0.y + v1.y, k0.x + k1.x, j0.x + j1.x, j0.y + j1.y,
            jd[2 * P + ia] + jd[2 * P + ib], s_G, s_al[el], F, FxLong());
  };
  auto put = [&](i64* xs, int at, const i64 F[5]) {
    reinterpret_cast<longlong2*>(xs)[at] = make_longlong2(F[0], F[1]);
    reinterpret_cast<longlong2*>(xs)[P + at] = make_longlong2(F[2], F[3]);
    xs[4 * P + at] = F[4];
  };
  // the directions by falling t, so that the sums are only shifted down on the way
#pragma unroll 1
  for (int x = 0; x < 3; ++x) {
    const int d = STRETCH ? s_walk[le] >> (2 * x) & 3 : x;
    const int r = d == 0 ? i : (d == 1 ? j : k);
    const int stride = d == 0 ? 1 : (d == 1 ? n : NN);
    const int line0 = id - r * stride;
    auto take_share = [&](const i64* xs, int src) {
      const Fx D = sD[r * n + src];
      const longlong2 a0 = reinterpret_cast<const longlong2*>(xs)[id], a1 = reinterpret_cast<const longlong2*>(xs)[P + id];
      fx_add(acc[0], D, fx_split(a0.x));
      fx_add(acc[1], D, fx_split(a0.y));
      fx_add(acc[2], D, fx_split(a1.x));
      fx_add(acc[3], D, fx_split(a1.y));
      fx_add(acc[4], D, fx_split(xs[4 * P + id]));
    };
    // exchange buffers: a direction's first writes wait for the previous
    // direction's last reads (different lines)
    if (x > 0) dsync(d);
#pragma unroll 1
    for (int s = 1; s <= FULL; ++s) {
      const int m = r + s < n ? r + s : r + s - n;
      const int mid = line0 + m * stride;
      i64* sXs = sX + (XB > 1 ? (s - 1) * XW : 0);
      if (act) {
        i64 F[5];
        pair(base, le, d, id, mid, F);
        put(sXs, mid, F);
        const Fx D = sD[r * n + m];
#pragma unroll
        for (int c = 0; c < 5; ++c) fx_add(acc[c], D, fx_split(F[c]));
      }
      if constexpr (XB == 1) {
        dsync(d);
        if (act) take_share(sX, r - s >= 0 ? r - s : r - s + n);
        dsync(d);
      }
    }
    if constexpr (HALF) {
      constexpr int H = n / 2;
      const int t = threadIdx.x;
      int le2, w2;
      bool take;
      if constexpr (SCOPE == 2) {
        if (d < 2) { le2 = 0; w2 = 32 * (t >> 6) + (t & 63); take = (t & 63) < 32; }
        else { le2 = 0; w2 = t; take = t < P / 2; }
      } else if constexpr (SCOPE == 1) {
        le2 = le; w2 = id; take = id < P / 2;
      } else {
        le2 = t / (P / 2); w2 = t - le2 * (P / 2); take = t < EPB * (P / 2);
      }
      if (take && s_state[le2] == 1) {
        const int d2 = STRETCH && SCOPE == 0 && EPB > 1 ? s_walk[le2] >> (2 * x) & 3 : d;   // the pair's own element's
        const int st2 = d2 == 0 ? 1 : (d2 == 1 ? n : NN);
        const int hi = w2 / st2;
        const int ia = w2 - hi * st2 + st2 * (hi % H + n * (hi / H));
        const int ib = ia + H * st2;
        i64* b2 = tile0 + le2 * PER_ELEM;
        i64 F[5];
        pair(b2, le2, d2, ia, ib, F);
        i64* xh = b2 + 10 * P + 3 * JW + (XB > 1 ? FULL * XW : 0);
        put(xh, ia, F);
        put(xh, ib, F);
      }
    }
    if constexpr (XB == 1) {
      if constexpr (HALF) {
        dsync(d);
        if (act) take_share(sX, r >= n / 2 ? r - n / 2 : r + n / 2);
      }
    } else {
      dsync(d);
      if (act) {
#pragma unroll 1
        for (int s = 1; s <= FULL; ++s) take_share(sX + (s - 1) * XW, r - s >= 0 ? r - s : r - s + n);
        if constexpr (HALF) take_share(sX + FULL * XW, r >= n / 2 ? r - n / 2 : r + n / 2);
      }
    }
#pragma unroll
    for (int c = 0; c < 5; ++c) fx_fold(acc[c]);
    if constexpr (STRETCH) {
      if (const int down = s_walk[le] >> (8 + 4 * x) & 15) {
#pragma unroll
        for (int c = 0; c < 5; ++c) fx_shift_down(acc[c], down);
      }
    }
  }
  int bad = 0;
#pragma unroll
  for (int l = 0; l < EPB; ++l) bad |= s_state[l] == 2;
  if (!act) return bad;
  const FxAlign al = s_al[le];
  double R[5];
#pragma unroll
  for (int c = 0; c < 5; ++c) R[c] = fx_to2<32>(acc[c].p, acc[c].c, c == 0 ? al.q0 : (c < 4 ? al.qm : al.qe));
#pragma unroll
  for (int c = 0; c < 4; ++c) R[c + 1] = fma(-g.mu, sA[c * P + id], R[c + 1]);
  // surface integral
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int id_d = ijk[d];
    if (id_d != 0 && id_d != N) continue;
    const int sgn = id_d == N ? 1 : 0;
    const int code = elem_face[e * 6 + 2 * d + sgn];
    const int fid = dg_idx(code >> 4, a.nfaces > 0 ? a.nfaces : 3L * E, kSiteVolFace);
    const int pp = d == 0 ? j : i;
    const int qq = d == 2 ? j : k;
    int p2 = pp, q2 = qq;
    if (!(code & 8)) apply_flip<n>(code & 7, pp, qq, p2, q2);
    const double* fsr = fstar + (size_t)fid * 5 * NN + p2 + n * q2;
    const double fs_sign = (code & 8) ? inv_w0 : -inv_w0;
#pragma unroll
    for (int c = 0; c < 5; ++c) R[c] = fma(fs_sign, fsr[c * NN], R[c]);
  }
  double src[5] = {0, 0, 0, 0, 0};
  if (g.source == DG_SOURCE_MMS) mms_source<double>(g, mms, e, P, id, s_tc[0], s_tc[1], src);
  const size_t o0 = (size_t)e * 5 * P + id;
  const double iJ = metrics[(size_t)e * 10 * P + 9 * P + id];
  if (a.mode == 0) {
#pragma unroll
    for (int c = 0; c < 5; ++c) a.Ut[o0 + (size_t)c * P] = fma(-R[c], iJ, src[c]);
  } else {
    const double dt = a.clock[1];
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      const size_t o = o0 + (size_t)c * P;
      const double gk = fma(a.A, rk_register(a, o), dt * fma(-R[c], iJ, src[c]));
      a.Gk[o] = gk;
      a.Uw[o] = fma(a.B, gk, q[c]);
    }
  }
  return bad;
}

// The FP64 volume body: fixed point, then FP64 for the elements outside its
// range (density or beta varying by more than a factor 8 to 16 inside the
// element, non-finite or non-positive values), which the same block redoes.
template <int N, int EPB, bool LIST = false, bool STRETCH = true>
__device__ __forceinline__ void volume_body_f64(const StageArgs& a, const double* __restrict__ metrics,
                                                const i64* __restrict__ jx, const float4* __restrict__ ejx,
                                                const double* __restrict__ grad, const double* __restrict__ fstar,
                                                const int* __restrict__ elem_face, const double* __restrict__ mms,
                                                const double* __restrict__ Dg, int E, const Gas& g, double inv_w0,
                                                int blk) {
  __shared__ int s_state[EPB];   // 0: no element, 1: done in fixed point, 2: left to FP64
  if (volume_body_fx<N, EPB, LIST, STRETCH>(a, metrics, jx, ejx, grad, fstar, elem_face, mms, Dg, E, g, inv_w0, blk,
                                            s_state)) {
    __syncthreads();
    volume_body<N, double, EPB, LIST>(a, metrics, metrics, grad, fstar, elem_face, mms, Dg, E, g, inv_w0, blk,
                                      s_state);
  }
}
template <int N, int EPB>
constexpr size_t volume_f64_smem_bytes() {
  return volume_fx_smem_bytes<N, EPB>() > volume_smem_bytes<N, double, EPB>() ? volume_fx_smem_bytes<N, EPB>()
                                                                                : volume_smem_bytes<N, double, EPB>();
}

// Shared memory of the volume body in either operator type.
template <int N, typename R, int EPB>
constexpr size_t volume_op_smem_bytes() {
  if constexpr (sizeof(R) == 8) return volume_f64_smem_bytes<N, EPB>();
  else return volume_smem_bytes<N, R, EPB>();
}

}  // namespace dg
