// Latency variants of the FP64 lifting, face-flux and volume kernels for
// meshes too small to fill the GPU (GALAEXI Sec. 3.1, Eqs. 2-3; the method's steps are
// those of dg_stage.cuh).
//
// With few elements (the 4^3 Taylor-Green case has 128 warps for the GPU's
// 608 SM sub-partitions) every warp runs alone on its sub-partition, and the
// FP64 pipe, which takes a warp instruction in about 68 cycles, makes a
// kernel last as long as its longest warp's FP64 instruction stream.  These
// kernels spread a node's work over three threads, one per reference
// direction d: the d-thread evaluates the split-form pairs, the viscous flux,
// the viscous line sum and the surface terms of its direction (volume), or
// the line derivatives of its direction and one component of every lifted
// gradient (lifting); the three directions' partial sums are added in a
// fixed order.  The face flux (LLF) takes two threads per face node, one per
// side.  One element per block of 3 (N+1)^3 threads, N <= 3.  The sums of
// the FP64 parts are grouped differently from the one-thread-per-node kernels,
// so results agree with them to rounding, not bit for bit.
#include "dg_face_fx.cuh"
#include "dg_volume_fx.cuh"

namespace dg {

// The three kernels of a stage are launched so that the next one may start while
// the last ends (programmatic dependent launch): each lets it before its last
// few operations, loads what no kernel writes (metric terms, face lists, D) and
// then waits for the previous kernel's completion.  Let start by a kernel's
// first instruction the next one took its place on the SMs (6^3, N = 3: 32.4 us
// per stage against 23.2, and 23.6 without).  Pointers to data of previous kernels go through after_previous():
// an opaque copy made after the wait, so that no load of theirs is moved before
// it or takes the read-only path.
__device__ __forceinline__ void start_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <typename T>
__device__ __forceinline__ T* after_previous(T* p) {
  asm volatile("" : "+l"(p)::"memory");
  return p;
}

template <int N>
struct LatShape {
  static constexpr int n = N + 1, P = n * n * n, NN = n * n, THREADS = 3 * P;
};

// ---------------------------------------------------------------------------
// Lifting: thread (d, node) forms D_d phi + jump_d for the four lifted
// variables, then the d-th component of their gradients
// g_{a,d} = (1/J) sum_d' Ja^{d'}_d (D_d' phi_a + jump_d').
// The threads of direction 0 evaluate the node's phi while the others evaluate
// the neighbours' at the face points; the jump (phi_nbr - phi) h, h = +-1/(2
// w_0), starts the line sum (its shares summed one by one, the own one through
// D's corners, gave up to 1.9 times the error in the heat flux).  Bound by the
// memory latency of its two dependent loads and by some 55 FP64 instructions a
// warp.
template <int N>
constexpr size_t lift_lat_smem_bytes() {
  constexpr int P = LatShape<N>::P, NN = LatShape<N>::NN;
  return sizeof(double) * ((size_t)4 * P + 24 * NN + 12 * P);
}

// 32 registers for N = 2 and 3, as its blocks start beside the volume kernel's:
// with 36 (40 allocated) a stage on 5^3 elements, N = 3 takes 22.0 us instead of 19.1.
template <int N>
__global__ void __launch_bounds__(LatShape<N>::THREADS, N == 1 ? 1 : 64 / ((LatShape<N>::THREADS + 31) / 32))
k_lift_lat(const double* __restrict__ U_, const double* __restrict__ metrics, const int* __restrict__ elem_nbr,
           const int* __restrict__ elem_face, const double* __restrict__ Dg, double* __restrict__ grad, int E,
           Gas g, double inv_w0) {
  using S = LatShape<N>;
  constexpr int n = S::n, P = S::P, NN = S::NN, NF = 6 * NN;
  __shared__ double sD[n * n];
  extern __shared__ __align__(16) unsigned char lat_raw[];
  double* sphi = reinterpret_cast<double*>(lat_raw);   // [4][P]
  double* snb = sphi + 4 * P;                          // [6][4][NN] phi_nbr
  double* sdd = snb + 24 * NN;                         // [4][3][P]: D_d phi_a + jump_d
  const int d = threadIdx.x / P, id = threadIdx.x - d * P;
  const int e = blockIdx.x;
  const double hw = 0.5 * inv_w0;
  const double* mt = metrics + (size_t)e * 10 * P + id;
  const double J0 = mt[(0 * 3 + d) * P], J1 = mt[(1 * 3 + d) * P], J2 = mt[(2 * 3 + d) * P];
  const double iJ = mt[9 * P];
  auto lifted = [&](const double* q, double* out, int pitch) {
    const double rho = q[0], m0 = q[P], m1 = q[2 * P], m2 = q[3 * P], en = q[4 * P], ir = rcp_op(rho);
    const double u = m0 * ir, v = m1 * ir, w = m2 * ir;
    const double T = g.gm1 * (en - 0.5 * (m0 * u + m1 * v + m2 * w)) * ir * g.inv_R;
    out[0] = u;
    out[pitch] = v;
    out[2 * pitch] = w;
    out[3 * pitch] = T;
  };
  constexpr int NI = (NF + 2 * P - 1) / (2 * P);   // face points of a thread of directions 1 and 2
  int nbr[NI] = {};
  if (d != 0) {
#pragma unroll
    for (int x = 0; x < NI; ++x) {
      const int t = threadIdx.x - P + x * 2 * P;
      if (t >= NF) break;
      const int f = t / NN, pq = t - f * NN;
      const int code = elem_face[e * 6 + f], nb = elem_nbr[e * 6 + f];
      int p2, q2;
      apply_flip<n>(code & 7, pq % n, pq / n, p2, q2);
      nbr[x] = dg_idx(nb >> 3, E, kSiteLiftNbr) * 5 * P + face_node<n>(nb & 7, p2, q2);
    }
    for (int t = threadIdx.x - P; t < n * n; t += 2 * P) sD[t] = Dg[t];
  }
  wait_previous();
  const double* U = after_previous(U_);
  if (d == 0) {
    lifted(U + (size_t)e * 5 * P + id, sphi + id, P);
  } else {
#pragma unroll
    for (int x = 0; x < NI; ++x) {
      const int t = threadIdx.x - P + x * 2 * P;
      if (t >= NF) break;
      const int f = t / NN, pq = t - f * NN;
      lifted(U + nbr[x], snb + f * 4 * NN + pq, NN);
    }
  }
  __syncthreads();
  const int i = id % n, j = (id / n) % n, k = id / NN;
  const int r = d == 0 ? i : (d == 1 ? j : k);
  const int stride = d == 0 ? 1 : (d == 1 ? n : NN);
  const int line0 = id - r * stride;
  const double* jm = nullptr;
  const double h = r == N ? hw : -hw;
  if (r == 0 || r == N)
    jm = snb + (2 * d + (r == N ? 1 : 0)) * 4 * NN + (d == 0 ? j : i) + n * (d == 2 ? j : k);
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    double s = jm ? (jm[a * NN] - sphi[a * P + id]) * h : 0.0;
#pragma unroll
    for (int m = 0; m < n; ++m) s = fma(sD[r * n + m], sphi[a * P + line0 + m * stride], s);
    sdd[(a * 3 + d) * P + id] = s;
  }
  __syncthreads();
  start_next();
  const double K0 = J0 * iJ, K1 = J1 * iJ, K2 = J2 * iJ;
  double* go = grad + (size_t)e * 12 * P + id;
#pragma unroll
  for (int a = 0; a < 4; ++a)
    go[(a * 3 + d) * P] = K0 * sdd[(a * 3) * P + id] + K1 * sdd[(a * 3 + 1) * P + id] + K2 * sdd[(a * 3 + 2) * P + id];
}

// ---------------------------------------------------------------------------
// Volume: thread (d, node) takes direction d's pairs, viscous line sum and
// surface terms; the three directions' sums meet in shared memory, and thread
// (d, node) finishes the variables c = d and c = d + 3.
//
// Component c of the manufactured source (density wave, see volume_body).
__device__ __forceinline__ double mms_source_lat(const Gas& g, double sa, double ca, const double* tc, int c) {
  const double st = tc[0], ct = tc[1];
  const double sphi = fma(sa, ct, -ca * st);
  const double cphi = fma(ca, ct, sa * st);
  const double A = g.mms_amp;
  const double rp = M_PI * A * cphi;
  if (c < 4) return 2.0 * rp;
  const double rw = 2.0 + A * sphi;
  const double irw = rcp_op(rw);
  const double lapT = 3.0 * g.inv_R * fma(M_PI * M_PI * A, sphi, 2.0 * rp * rp * irw) * (irw * irw);
  return fma(-(g.mu * g.kappa), lapT, 3.0 * rp);
}

// Fixed-point body (the terms and scales of volume_body_fx): the FP64 chain of
// a warp is the node's primitives, the surface sums and the update, 30
// instructions instead of 250; what is left is mostly the latency of the launch
// and of the loads, so every operand is asked for at the start.  Taylor-Green,
// CUDA events per launch with the FP64 body -> now: N = 2, 4^3 12.3 -> 10.3 us,
// N = 3, 4^3 16.4 -> 12.3, N = 3, 6^3 24.6 -> 14.3.
// Words of 8 bytes: the Fx table of D, node data (6 P), metric terms, viscous
// fluxes (12 P), exchange buffers, primitives (6 P), the directions' sums (54 P).
template <int N>
struct LatFx {
  static constexpr int n = N + 1, P = n * n * n, PW = P + (P & 1), ROUNDS = n / 2, JW = 2 * P + PW, XW = 4 * P + PW;
  static constexpr int tables = (n * n + 1) & ~1, words = tables + 6 * P + 3 * JW + 12 * P + 3 * ROUNDS * XW + 6 * P + 54 * P;
};

// False (the whole block): the element is out of the fixed-point range.
// STRETCH as in volume_body_fx.
template <int N, bool STRETCH>
__device__ __forceinline__ bool volume_lat_fx(const StageArgs& a, const double* __restrict__ metrics,
                                              const i64* __restrict__ jx, const float4* __restrict__ ejx,
                                              const double* grad_, const double* fstar_,
                                              const int* __restrict__ elem_face, const double* __restrict__ mms,
                                              const double* __restrict__ Dg, int E, const Gas& g, double inv_w0,
                                              unsigned char* raw, double* s_tc) {
  using S = LatShape<N>;
  using B = LatFx<N>;
  constexpr int n = S::n, P = S::P, NN = S::NN, JW = B::JW, XW = B::XW, eD = fx_eD(N);
  Fx* sD = reinterpret_cast<Fx*>(raw);
  i64* base = reinterpret_cast<i64*>(raw) + B::tables;
  longlong2* sN = reinterpret_cast<longlong2*>(base);   // [3][P] (rho, b), (|u|^2, u), (v, w)
  i64* sJ = base + 6 * P;                                // [3]: (J0, J1) [P], J2 [P]
  i64* sFv = sJ + 3 * JW;                                // [3][4][P]
  i64* sX = sFv + 12 * P;                                // [ROUNDS][3]: (F0, F1) [P], (F2, F3) [P], F4 [P]
  double* sQ = reinterpret_cast<double*>(sX + 3 * B::ROUNDS * XW);   // [6][P] u, v, w, rho, b, |u|^2
  longlong2* sS = reinterpret_cast<longlong2*>(sQ + 6 * P);          // [9][3][P] sums: flux (5), viscous (4)
  __shared__ int s_mx[kMxCount];
  __shared__ FxAlign s_al;
  __shared__ Fx s_G;
  const int d = threadIdx.x / P, id = threadIdx.x - d * P;
  const int e = blockIdx.x;
  const int ijk[3] = {id % n, (id / n) % n, id / NN};
  // every operand is asked for here, what no kernel writes before the wait
  if (threadIdx.x < kMxCount) s_mx[threadIdx.x] = 0;
  const i64* mt = jx + (size_t)e * 10 * P + id;
  const i64 Jr[3] = {mt[(d * 3) * P], mt[(d * 3 + 1) * P], mt[(d * 3 + 2) * P]};
  const float4 ej = ejx[e];
  const int td = STRETCH ? fx_shifts(ej).t(d) : 0;
  const i64 Ja[3] = {fx_up(Jr[0], td), fx_up(Jr[1], td), fx_up(Jr[2], td)};
  int fso[3] = {-1, -1, -1};   // surface flux of the node, per direction
  double fsg[3] = {0, 0, 0};
#pragma unroll
  for (int x = 0; x < 3; ++x) {
    if (ijk[x] != 0 && ijk[x] != N) continue;
    const int code = elem_face[e * 6 + 2 * x + (ijk[x] == N ? 1 : 0)];
    const int fid = dg_idx(code >> 4, 3L * E, kSiteVolFace);   // F = 3 E
    int p2 = x == 0 ? ijk[1] : ijk[0], q2 = x == 2 ? ijk[1] : ijk[2];
    if (!(code & 8)) apply_flip<n>(code & 7, p2, q2, p2, q2);
    fso[x] = fid * 5 * NN + p2 + n * q2;
    fsg[x] = (code & 8) ? inv_w0 : -inv_w0;
  }
  for (int t = threadIdx.x; t < n * n; t += blockDim.x) {
    const double dr = Dg[t];
    sD[t] = fx_split(fx_round(t == 0 ? dr + inv_w0 : (t == n * n - 1 ? dr - inv_w0 : dr), kFxQD - eD));
  }
  const double iJ = metrics[((size_t)e * 10 + 9) * P + id];
  double sa = 0.0, ca = 0.0;
  if (g.source == DG_SOURCE_MMS) {
    sa = mms[((size_t)e * 2) * P + id];
    ca = mms[((size_t)e * 2 + 1) * P + id];
  }
  wait_previous();
  const double* grad = after_previous(grad_);
  const double* fstar = after_previous(fstar_);
  if (threadIdx.x == 2 * P && g.source == DG_SOURCE_MMS)
    sincospi(a.clock[0] + a.c_stage * a.clock[1], &s_tc[0], &s_tc[1]);
  double q[5] = {1, 0, 0, 0, 1};
  if (d == 0) {
#pragma unroll
    for (int v = 0; v < 5; ++v) q[v] = a.U[((size_t)e * 5 + v) * P + id];
  }
  double gr[12];
#pragma unroll
  for (int r = 0; r < 12; ++r) gr[r] = grad[((size_t)e * 12 + r) * P + id];
  double fs[2][3], Uc[2] = {0, 0}, Gc[2] = {0, 0};
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int c = d + 3 * h;
#pragma unroll
    for (int x = 0; x < 3; ++x) fs[h][x] = c < 5 && fso[x] >= 0 ? fstar[fso[x] + c * NN] : 0.0;
    if (c < 5 && a.mode != 0) {
      Uc[h] = a.U[((size_t)e * 5 + c) * P + id];
      Gc[h] = rk_register(a, ((size_t)e * 5 + c) * P + id);
    }
  }
  __syncthreads();
  {
    int mx[kMxCount] = {};
    auto mag2 = [](double x, double y) { return max(fx_mag(x), fx_mag(y)); };
    if (d == 0) {
      const double rho = q[0], ir = rcp_op(rho);
      const double u = q[1] * ir, v = q[2] * ir, w = q[3] * ir;
      const double kk = u * u + v * v + w * w;
      const double p = g.gm1 * fma(-0.5 * rho, kk, q[4]);
      const double bt = 0.125 * rho * rcp_op(p);   // beta / 4
      sQ[id] = u; sQ[P + id] = v; sQ[2 * P + id] = w;
      sQ[3 * P + id] = rho; sQ[4 * P + id] = bt; sQ[5 * P + id] = kk;
      const int hr = max(__double2hiint(rho), 0), hb = max(__double2hiint(bt), 0);
      mx[kMxR] = hr;
      mx[kMxRmin] = 0x7fffffff - hr;
      mx[kMxB] = hb;
      mx[kMxBmin] = 0x7fffffff - hb;
      mx[kMxU] = max(mag2(u, v), fx_mag(w));
    } else if (d == 1) {
      mx[kMxG] = max(max(mag2(gr[0], gr[1]), mag2(gr[2], gr[3])),
                     max(max(mag2(gr[4], gr[5]), mag2(gr[6], gr[7])), fx_mag(gr[8])));
      mx[kMxT] = max(mag2(gr[9], gr[10]), fx_mag(gr[11]));
    }
    __syncwarp();
    fx_maxima<kMxCount>(0, s_mx, mx);
  }
  __syncthreads();
  FxElem ex = fx_element(s_mx, ej);
  if (!ex.ok) return false;
  const int eg = ((__double2hiint(g.inv_gm1) >> 20) & 0x7ff) - 1022;
  const int ek = ((__double2hiint(g.kappa) >> 20) & 0x7ff) - 1022;
  const int q1 = 56 - ex.g - ex.e.u, q2 = 59 - ex.t - ek;   // of the viscous energy flux's two terms, + (-e_j + t_d)
  if (threadIdx.x == 3 * P - 1) {
    FxElem el = ex;
    fx_element_logs(el, s_mx, ej);
    s_al = fx_align(el.e, eg, fx_log_mantissa(__double2hiint(g.inv_gm1), 1), eD);
    s_G = fx_split(fx_from(g.inv_gm1, 62 - eg));
  }
  {
    // node data, and the viscous flux of this direction (scales as in volume_body_fx)
    const i64 xu = fx_from(sQ[id], kFxQ - ex.e.u), xv = fx_from(sQ[P + id], kFxQ - ex.e.u),
              xw = fx_from(sQ[2 * P + id], kFxQ - ex.e.u);
    if (d == 0) sN[id] = make_longlong2(fx_from(sQ[3 * P + id], kFxQ - ex.e.r), fx_from(sQ[4 * P + id], kFxQ - ex.e.b));
    else if (d == 1) sN[P + id] = make_longlong2(fx_from(sQ[5 * P + id], kFxQ - 2 - 2 * ex.e.u), xu);
    else sN[2 * P + id] = make_longlong2(xv, xw);
    reinterpret_cast<longlong2*>(sJ + d * JW)[id] = make_longlong2(Ja[0], Ja[1]);
    sJ[d * JW + 2 * P + id] = Ja[2];
    i64 G[9];
#pragma unroll
    for (int r = 0; r < 9; ++r) G[r] = fx_from(gr[r], 59 - ex.g);
    const Fx twothird{715827883, -1431655765};   // 2^62 2/3 / 2^32 and the low word of 2^62 2/3
    const i64 div = fx_mul<2>(fx_split(G[0] + G[4] + G[8]), twothird);
    const Fx t00 = fx_split(2 * G[0] - div), t11 = fx_split(2 * G[4] - div), t22 = fx_split(2 * G[8] - div);
    const Fx t01 = fx_split(G[1] + G[3]), t02 = fx_split(G[2] + G[6]), t12 = fx_split(G[5] + G[7]);
    const Fx kap = fx_split(fx_from(g.kappa, kFxQ - ek));
    const Fx J[3] = {fx_split(Ja[0]), fx_split(Ja[1]), fx_split(Ja[2])};
    FxSum f0 = fx_zero<3>(), f1 = fx_zero<3>(), f2 = fx_zero<3>(), h = fx_zero<3>(), en = fx_zero<2>();
    fx_add(f0, t00, J[0]); fx_add(f0, t01, J[1]); fx_add(f0, t02, J[2]);
    fx_add(f1, t01, J[0]); fx_add(f1, t11, J[1]); fx_add(f1, t12, J[2]);
    fx_add(f2, t02, J[0]); fx_add(f2, t12, J[1]); fx_add(f2, t22, J[2]);
#pragma unroll
    for (int l = 0; l < 3; ++l) fx_add(h, fx_split(fx_mul<4>(fx_split(fx_from(gr[9 + l], kFxQ - ex.t)), kap)), J[l]);
    const i64 v0 = fx_end<3>(f0), v1 = fx_end<3>(f1), v2 = fx_end<3>(f2);
    fx_add(en, fx_split(v0), fx_split(xu)); fx_add(en, fx_split(v1), fx_split(xv)); fx_add(en, fx_split(v2), fx_split(xw));
    i64* fv = sFv + d * 4 * P + id;
    fv[0] = v0;
    fv[P] = v1;
    fv[2 * P] = v2;
    fv[3 * P] = (fx_end<2>(en) >> fx_clamp(q1 - q2)) + (fx_end<3>(h) >> fx_clamp(q2 - q1));
  }
  __syncthreads();
  const int r = d == 0 ? ijk[0] : (d == 1 ? ijk[1] : ijk[2]);
  const int stride = d == 0 ? 1 : (d == 1 ? n : NN);
  const int line0 = id - r * stride;
  FxSum acc[5] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}, {0, 0}};
  constexpr int FULL = (n - 1) / 2;
  constexpr bool HALF = (n % 2) == 0;
  const i64* jd = sJ + d * JW;
  const longlong2* jp = reinterpret_cast<const longlong2*>(jd);
  auto pair = [&](int ia, int ib, i64 F[5]) {
    const longlong2 r0 = sN[ia], r1 = sN[ib], k0 = sN[P + ia], k1 = sN[P + ib], v0 = sN[2 * P + ia], v1 = sN[2 * P + ib];
    const longlong2 j0 = jp[ia], j1 = jp[ib];
    fx_pair(r0.x, r1.x, r0.y, r1.y, k0.y + k1.y, v0.x + v1.x, v0.y + v1.y, k0.x + k1.x, j0.x + j1.x, j0.y + j1.y,
            jd[2 * P + ia] + jd[2 * P + ib], s_G, s_al, F, FxLong());
  };
  auto put = [&](i64* xs, int at, const i64 F[5]) {
    reinterpret_cast<longlong2*>(xs)[at] = make_longlong2(F[0], F[1]);
    reinterpret_cast<longlong2*>(xs)[P + at] = make_longlong2(F[2], F[3]);
    xs[4 * P + at] = F[4];
  };
#pragma unroll 1
  for (int s = 1; s <= FULL; ++s) {
    const int m = r + s < n ? r + s : r + s - n;
    const int mid = line0 + m * stride;
    i64 F[5];
    pair(id, mid, F);
    put(sX + ((s - 1) * 3 + d) * XW, mid, F);
    const Fx D = sD[r * n + m];
#pragma unroll
    for (int c = 0; c < 5; ++c) fx_add(acc[c], D, fx_split(F[c]));
  }
  if constexpr (HALF) {
    // s = n/2: the pairs (r, r + n/2), r < n/2, on half of the direction's threads
    // (the second half for d > 0, whose warps share no sub-partition with d = 0's)
    constexpr int H = n / 2;
    const int w2 = d == 0 ? id : id - P / 2;
    if (w2 >= 0 && w2 < P / 2) {
      const int hi = w2 / stride;
      const int ia = w2 - hi * stride + stride * (hi % H + n * (hi / H));
      const int ib = ia + H * stride;
      i64 F[5];
      pair(ia, ib, F);
      i64* xh = sX + (FULL * 3 + d) * XW;
      put(xh, ia, F);
      put(xh, ib, F);
    }
  }
  // viscous line sum of direction d, with the viscous surface part in the end diagonals
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const i64* line = sFv + (d * 4 + c) * P + line0;
    FxSum s{0, 0};
#pragma unroll
    for (int m = 0; m < n; ++m) fx_add(s, sD[r * n + m], fx_split(line[m * stride]));
    if (td) fx_visc_down(s, td);
    sS[((5 + c) * 3 + d) * P + id] = make_longlong2(s.p, s.c >> 2);
  }
  __syncthreads();
  auto take_share = [&](const i64* xs, int src) {
    const Fx D = sD[r * n + src];
    const longlong2 a0 = reinterpret_cast<const longlong2*>(xs)[id], a1 = reinterpret_cast<const longlong2*>(xs)[P + id];
    fx_add(acc[0], D, fx_split(a0.x));
    fx_add(acc[1], D, fx_split(a0.y));
    fx_add(acc[2], D, fx_split(a1.x));
    fx_add(acc[3], D, fx_split(a1.y));
    fx_add(acc[4], D, fx_split(xs[4 * P + id]));
  };
#pragma unroll
  for (int s = 1; s <= FULL; ++s) take_share(sX + ((s - 1) * 3 + d) * XW, r - s >= 0 ? r - s : r - s + n);
  if constexpr (HALF) take_share(sX + (FULL * 3 + d) * XW, r >= n / 2 ? r - n / 2 : r + n / 2);
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    fx_fold(acc[c]);
    if (td) fx_shift_down(acc[c], td);
    sS[(c * 3 + d) * P + id] = make_longlong2(acc[c].p, acc[c].c);
  }
  __syncthreads();
  start_next();
  const FxAlign al = s_al;
  const int qv = kFxQD - 6 - ex.g - ex.e.j - eD, qe = (q1 < q2 ? q1 : q2) - (64 - kFxQD) - ex.e.j - eD;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int c = d + 3 * h;
    if (c >= 5) break;
    auto sum = [&](int row, i64& p, i64& f) {
      const longlong2 x = sS[row * 3 * P + id], y = sS[(row * 3 + 1) * P + id], z = sS[(row * 3 + 2) * P + id];
      p = x.x + y.x + z.x;
      f = x.y + y.y + z.y;
    };
    i64 p, f;
    sum(c, p, f);
    double R = fx_to2<32>(p, f, c == 0 ? al.q0 : (c < 4 ? al.qm : al.qe));
    if (c > 0) {
      sum(4 + c, p, f);
      R = fma(-g.mu, fx_to2<30>(p, f, c < 4 ? qv : qe), R);
    }
#pragma unroll
    for (int x = 0; x < 3; ++x)
      if (fso[x] >= 0) R = fma(fsg[x], fs[h][x], R);
    const double src = g.source == DG_SOURCE_MMS ? mms_source_lat(g, sa, ca, s_tc, c) : 0.0;
    const size_t o = ((size_t)e * 5 + c) * P + id;
    if (a.mode == 0) {
      a.Ut[o] = fma(-R, iJ, src);
    } else {
      const double gk = fma(a.A, Gc[h], a.clock[1] * fma(-R, iJ, src));
      a.Gk[o] = gk;
      a.Uw[o] = fma(a.B, gk, Uc[h]);
    }
  }
  return true;
}

// FP64 body: elements out of the fixed-point range, contexts without
// fixed-point metric terms, and Sutherland's law (whose factor every thread of a node would have to apply to the gradients).
template <int N>
constexpr size_t volume_lat_f64_bytes() {
  constexpr int n = N + 1, P = n * n * n;
  // D and its three scalings, rho, u (3), beta/4, |u|^2, J a (9), f_v . J a (12),
  // the three directions' exchange buffers (15), which also hold the partial sums
  return sizeof(double) * ((size_t)4 * n * n + 6 * P + 9 * P + 12 * P + 15 * P);
}
template <int N>
constexpr size_t volume_lat_smem_bytes() {
  return 8 * LatFx<N>::words > volume_lat_f64_bytes<N>() ? 8 * LatFx<N>::words : volume_lat_f64_bytes<N>();
}

template <int N>
__device__ __forceinline__ void volume_lat_f64(const StageArgs& a, const double* __restrict__ metrics,
                                               const double* grad, const double* fstar,
                                               const int* __restrict__ elem_face, const double* __restrict__ mms,
                                               const double* __restrict__ Dg, int E, const Gas& g, double inv_w0,
                                               unsigned char* raw, const double* s_tc) {
  using S = LatShape<N>;
  constexpr int n = S::n, P = S::P, NN = S::NN;
  double* sD = reinterpret_cast<double*>(raw);   // D, viscous surface part in the end diagonals
  double* sT0 = sD + n * n;                          // D/4, D/8, D/16 (scaled two-point fluxes)
  double* sT1 = sT0 + n * n;
  double* sT2 = sT1 + n * n;
  double* sR = sT2 + n * n;                          // rho
  double* sU = sR + P;                               // u, v, w
  double* sB = sU + 3 * P;                           // beta / 4
  double* sK = sB + P;                               // |u|^2
  double* sJ = sK + P;                               // [9][P] J a^d_l, row 3 d + l
  double* sFv = sJ + 9 * P;                          // [3][4][P] (f_v . J a^d)
  double* sX = sFv + 12 * P;                         // [3][5][P] exchange per direction, then partial sums
  const int d = threadIdx.x / P, id = threadIdx.x - d * P;
  const int e = blockIdx.x;
  for (int t = threadIdx.x; t < n * n; t += blockDim.x) {
    const double dr = Dg[t];
    sD[t] = t == 0 ? dr + inv_w0 : (t == n * n - 1 ? dr - inv_w0 : dr);
    sT0[t] = 0.25 * dr;
    sT1[t] = 0.125 * dr;
    sT2[t] = 0.0625 * dr;
  }
  const double* mt = metrics + (size_t)e * 10 * P + id;
  const double Ja0 = mt[(d * 3) * P], Ja1 = mt[(d * 3 + 1) * P], Ja2 = mt[(d * 3 + 2) * P];
  sJ[(d * 3) * P + id] = Ja0;
  sJ[(d * 3 + 1) * P + id] = Ja1;
  sJ[(d * 3 + 2) * P + id] = Ja2;
  if (d == 0) {
    const double* q = a.U + (size_t)e * 5 * P + id;
    const double rho = q[0], ir = rcp_op(rho);
    const double u = q[P] * ir, v = q[2 * P] * ir, w = q[3 * P] * ir;
    const double kk = u * u + v * v + w * w;
    const double p = g.gm1 * fma(-0.5 * rho, kk, q[4 * P]);
    sR[id] = rho; sU[id] = u; sU[P + id] = v; sU[2 * P + id] = w; sK[id] = kk;
    sB[id] = 0.125 * rho * rcp_op(p);
  }
  __syncthreads();
  const double rho = sR[id], u = sU[id], v = sU[P + id], w = sU[2 * P + id], beta = sB[id], kk = sK[id];
  {
    // viscous flux of this direction from the lifted gradients
    double gr[12];
    const double* gg = grad + (size_t)e * 12 * P + id;
#pragma unroll
    for (int r2 = 0; r2 < 12; ++r2) gr[r2] = gg[r2 * P];
    double mu = g.mu, lam = g.mu * g.kappa;
    if (g.visc_law == DG_VISC_SUTHERLAND) {
      // T = p / (rho R) with p from beta/4 = rho / (8 p)
      const double sf = visc_factor<double>(g, 0.125 * rcp_op(beta) * g.inv_R);
      mu *= sf;
      lam *= sf;
    }
    double fv[4];
    visc_flux<double>(gr, u, v, w, mu, lam, Ja0, Ja1, Ja2, fv);
#pragma unroll
    for (int c = 0; c < 4; ++c) sFv[(d * 4 + c) * P + id] = fv[c];
  }
  const int i = id % n, j = (id / n) % n, k = id / NN;
  const int ijk[3] = {i, j, k};
  const int r = ijk[d];
  const int stride = d == 0 ? 1 : (d == 1 ? n : NN);
  const int line0 = id - r * stride;
  const double* sJd = sJ + d * 3 * P;
  double* sXd = sX + d * 5 * P;
  double acc[5] = {0, 0, 0, 0, 0};
  constexpr int FULL = (n - 1) / 2;
  constexpr bool HALF = (n % 2) == 0;
  __syncthreads();
  auto take_share = [&](int src) {
    const int rm = r * n + src;
    acc[0] = fma(sT0[rm], sXd[id], acc[0]);
    acc[1] = fma(sT1[rm], sXd[P + id], acc[1]);
    acc[2] = fma(sT1[rm], sXd[2 * P + id], acc[2]);
    acc[3] = fma(sT1[rm], sXd[3 * P + id], acc[3]);
    acc[4] = fma(sT2[rm], sXd[4 * P + id], acc[4]);
  };
#pragma unroll 1
  for (int s = 1; s <= FULL; ++s) {
    const int m = r + s < n ? r + s : r + s - n;
    const int mid = line0 + m * stride;
    double F[5];
    ec_pair<double>(rho, sR[mid], beta, sB[mid], u + sU[mid], v + sU[P + mid], w + sU[2 * P + mid], kk + sK[mid],
                    0.0, Ja0 + sJd[mid], Ja1 + sJd[P + mid], Ja2 + sJd[2 * P + mid], g.inv_gm1, g, F);
    const int rm = r * n + m;
    acc[0] = fma(sT0[rm], F[0], acc[0]);
    acc[1] = fma(sT1[rm], F[1], acc[1]);
    acc[2] = fma(sT1[rm], F[2], acc[2]);
    acc[3] = fma(sT1[rm], F[3], acc[3]);
    acc[4] = fma(sT2[rm], F[4], acc[4]);
#pragma unroll
    for (int c = 0; c < 5; ++c) sXd[c * P + mid] = F[c];
    __syncthreads();
    take_share(r - s >= 0 ? r - s : r - s + n);
    __syncthreads();
  }
  if constexpr (HALF) {
    // s = n/2: the pairs (r, r + n/2), r < n/2, on the direction's first P/2 threads
    constexpr int H = n / 2;
    if (id < P / 2) {
      const int hi = id / stride;
      const int ia = id - hi * stride + stride * (hi % H + n * (hi / H));
      const int ib = ia + H * stride;
      double F[5];
      ec_pair<double>(sR[ia], sR[ib], sB[ia], sB[ib], sU[ia] + sU[ib], sU[P + ia] + sU[P + ib],
                      sU[2 * P + ia] + sU[2 * P + ib], sK[ia] + sK[ib], 0.0, sJd[ia] + sJd[ib],
                      sJd[P + ia] + sJd[P + ib], sJd[2 * P + ia] + sJd[2 * P + ib], g.inv_gm1, g, F);
#pragma unroll
      for (int c = 0; c < 5; ++c) {
        sXd[c * P + ia] = F[c];
        sXd[c * P + ib] = F[c];
      }
    }
    __syncthreads();
    take_share(r >= n / 2 ? r - n / 2 : r + n / 2);
  }
  // viscous line sum of direction d, with the viscous surface part in the end diagonals
  {
    double v0 = 0, v1 = 0, v2 = 0, v3 = 0;
#pragma unroll
    for (int m = 0; m < n; ++m) {
      const double Drm = sD[r * n + m];
      const int mid = line0 + m * stride;
      v0 = fma(Drm, sFv[(d * 4 + 0) * P + mid], v0);
      v1 = fma(Drm, sFv[(d * 4 + 1) * P + mid], v1);
      v2 = fma(Drm, sFv[(d * 4 + 2) * P + mid], v2);
      v3 = fma(Drm, sFv[(d * 4 + 3) * P + mid], v3);
    }
    acc[1] -= v0; acc[2] -= v1; acc[3] -= v2; acc[4] -= v3;
  }
  // surface integral on the face of direction d through the node
  if (r == 0 || r == N) {
    const int code = elem_face[e * 6 + 2 * d + (r == N ? 1 : 0)];
    const int fid = dg_idx(code >> 4, 3L * E, kSiteVolFace);   // F = 3 E
    const int pp = d == 0 ? j : i;
    const int qq = d == 2 ? j : k;
    const double* fsr;
    double fs_sign;
    if (code & 8) {
      fsr = fstar + (size_t)fid * 5 * NN + pp + n * qq;
      fs_sign = inv_w0;
    } else {
      int p2, q2;
      apply_flip<n>(code & 7, pp, qq, p2, q2);
      fsr = fstar + (size_t)fid * 5 * NN + p2 + n * q2;
      fs_sign = -inv_w0;
    }
#pragma unroll
    for (int c = 0; c < 5; ++c) acc[c] = fma(fs_sign, fsr[c * NN], acc[c]);
  }
  // the three directions' sums, in the order d = 0, 1, 2
  __syncthreads();
#pragma unroll
  for (int c = 0; c < 5; ++c) sXd[c * P + id] = acc[c];
  __syncthreads();
  const double iJ = mt[9 * P];
  double sa = 0.0, ca = 0.0;
  if (g.source == DG_SOURCE_MMS) {
    sa = mms[((size_t)e * 2) * P + id];
    ca = mms[((size_t)e * 2 + 1) * P + id];
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int c = d + 3 * h;
    if (c >= 5) break;
    const double tot = (sX[c * P + id] + sX[(5 + c) * P + id]) + sX[(10 + c) * P + id];
    const double src = g.source == DG_SOURCE_MMS ? mms_source_lat(g, sa, ca, s_tc, c) : 0.0;
    const size_t o = ((size_t)e * 5 + c) * P + id;
    if (a.mode == 0) {
      a.Ut[o] = fma(-tot, iJ, src);
    } else {
      const double gk = fma(a.A, rk_register(a, o), a.clock[1] * fma(-tot, iJ, src));
      a.Gk[o] = gk;
      a.Uw[o] = fma(a.B, gk, a.U[o]);
    }
  }
}

template <int N, bool STRETCH>
__global__ void __launch_bounds__(LatShape<N>::THREADS, 2)
k_volume_lat(StageArgs a, const double* __restrict__ metrics, const i64* __restrict__ jx,
             const float4* __restrict__ ejx, const double* __restrict__ grad, const double* __restrict__ fstar,
             const int* __restrict__ elem_face, const double* __restrict__ mms, const double* __restrict__ Dg, int E,
             Gas g, double inv_w0) {
  extern __shared__ __align__(16) unsigned char lat_raw[];
  __shared__ double s_tc[2];
  if (g.visc_law != DG_VISC_SUTHERLAND && jx != nullptr) {
    if (volume_lat_fx<N, STRETCH>(a, metrics, jx, ejx, grad, fstar, elem_face, mms, Dg, E, g, inv_w0, lat_raw, s_tc)) return;
    __syncthreads();
  } else {
    wait_previous();
    if (threadIdx.x == 0 && g.source == DG_SOURCE_MMS)
      sincospi(a.clock[0] + a.c_stage * a.clock[1], &s_tc[0], &s_tc[1]);
  }
  volume_lat_f64<N>(a, metrics, after_previous(grad), after_previous(fstar), elem_face, mms, Dg, E, g, inv_w0, lat_raw,
                    s_tc);
}

// ---------------------------------------------------------------------------
// Face flux with the LLF Riemann flux: two threads per face node, one per
// side (even lane: master, odd lane: slave), each forming its side's
// primitives, Euler flux, wave speed and viscous flux; the partner's values
// come by warp shuffle, and the even lane writes the mass and momentum
// components of F*, the odd lane the energy component:
//   F* = (1/2 (f_L + f_R) . n - 1/2 lambda_max (q_R - q_L) - 1/2 (f_v,L + f_v,R) . n) sJ.
template <int N>
__global__ void __launch_bounds__(64)
k_face_lat(const double* __restrict__ U_, const double* __restrict__ grad_, const FaceInfo* __restrict__ faces,
           const double* __restrict__ facegeo, double* __restrict__ fstar, int F, Gas g) {
  constexpr int n = N + 1, P = n * n * n, NN = n * n;
  const long gid = ((long)blockIdx.x * blockDim.x + threadIdx.x) >> 1;
  const int side = threadIdx.x & 1;
  const bool live = gid < (long)F * NN;
  const long gsafe = live ? gid : 0;
  const int f = (int)(gsafe / NN), pq = (int)(gsafe % NN);
  const int p = pq % n, q = pq / n;
  const FaceInfo fi = faces[f];
  int e, lf, pp = p, qq = q;
  if (side == 0) {
    e = dg_idx(fi.master >> 3, F / 3, kSiteFaceElems);   // F = 3 E
    lf = fi.master & 7;
  } else {
    e = dg_idx(fi.slave >> 3, F / 3, kSiteFaceElems);
    lf = fi.slave & 7;
    apply_flip<n>(fi.flip, p, q, pp, qq);
  }
  const int node = face_node<n>(lf, pp, qq);
  const double* fg = facegeo + (size_t)f * 4 * NN + pq;
  const double nv[3] = {fg[0], fg[NN], fg[2 * NN]}, sJ = fg[3 * NN];
  wait_previous();
  const double* qp = after_previous(U_) + (size_t)e * 5 * P + node;
  const double* gs = after_previous(grad_) + (size_t)e * 12 * P + node;
  double qs[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) qs[v] = qp[v * P];
  const double nx = nv[0], ny = nv[1], nz = nv[2];
  const double ir = rcp_op(qs[0]);
  const double us[3] = {qs[1] * ir, qs[2] * ir, qs[3] * ir};
  const double pr = g.gm1 * (qs[4] - 0.5 * (qs[1] * us[0] + qs[2] * us[1] + qs[3] * us[2]));
  const bool suth = g.visc_law == DG_VISC_SUTHERLAND;
  const double sf = suth ? visc_factor<double>(g, pr * ir * g.inv_R) : 1.0;
  double fv[4];
  if (!face_visc_fx<1>(gs, gs, P, sf, sf, suth, us, us, nv, g.kappa, fv)) {
    double a[12];
#pragma unroll
    for (int r = 0; r < 12; ++r) a[r] = gs[r * P];
    visc_flux<double>(a, us[0], us[1], us[2], sf, g.kappa * sf, nx, ny, nz, fv);
  }
  const double un = us[0] * nx + us[1] * ny + us[2] * nz;
  const double lam = fabs(un) + sqrt_op(g.gamma * pr * ir);
  // f . n - mu f_v . n: one value per component to exchange
  const double fa[5] = {qs[0] * un, fma(-g.mu, fv[0], fma(qs[1], un, pr * nx)), fma(-g.mu, fv[1], fma(qs[2], un, pr * ny)),
                        fma(-g.mu, fv[2], fma(qs[3], un, pr * nz)), fma(-g.mu, fv[3], (qs[4] + pr) * un)};
  start_next();
  double qo[5], fo[5];
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    qo[c] = __shfl_xor_sync(0xffffffffu, qs[c], 1);
    fo[c] = __shfl_xor_sync(0xffffffffu, fa[c], 1);
  }
  const double lamo = __shfl_xor_sync(0xffffffffu, lam, 1);
  if (!live) return;
  // left = master (even lane), right = slave (odd lane)
  const double lL = side ? lamo : lam, lR = side ? lam : lamo;
  const double lmax = lR > lL ? lR : lL, half = 0.5 * sJ;
  double* out = fstar + (size_t)f * 5 * NN + pq;
  const int c0 = side ? 3 : 0, c1 = side ? 5 : 3;
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    if (c < c0 || c >= c1) continue;
    const double jump = side ? qs[c] - qo[c] : qo[c] - qs[c];
    out[(size_t)c * NN] = half * fma(-lmax, jump, fa[c] + fo[c]);
  }
}

// ---------------------------------------------------------------------------
template <int N>
static cudaError_t lat_setup() {
  cudaError_t e = cudaFuncSetAttribute(k_lift_lat<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)lift_lat_smem_bytes<N>());
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_volume_lat<N, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)volume_lat_smem_bytes<N>());
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_volume_lat<N, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)volume_lat_smem_bytes<N>());
  // one split of L1 for the three, so that blocks of two of them fit on an SM at a time
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_lift_lat<N>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_face_lat<N>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_volume_lat<N, false>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_volume_lat<N, true>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  return e;
}

cudaError_t setup_latency(int N) {
  switch (N) {
    case 1: return lat_setup<1>();
    case 2: return lat_setup<2>();
    case 3: return lat_setup<3>();
    default: return cudaSuccess;
  }
}

// Whether the context takes the latency kernels: FP64, LGL nodes, N <= 3 and
// at most kLatencyNodes nodes.  They pay where the one-thread-per-node kernels
// leave sub-partitions idle and lose where the mesh fills the GPU (Taylor-Green,
// us per stage, one-thread-per-node -> these: 4^3 N = 1 32.1 -> 15.1, N = 2 35.8
// -> 15.0, N = 3 32.5 -> 16.6; 6^3 N = 3 32.7 -> 24.1; 7^3 36.9 -> 33.7; but 8^3
// 39.2 -> 40.1, 11^3 N = 2 46.0 -> 45.0, 16^3 N = 1 43.8 -> 57.9).
bool use_latency_kernels(const Ctx& c) {
  return c.prm.precision == DG_FP64 && c.prm.nodes == DG_NODES_LGL && c.N <= 3 && c.M == 0 &&
         (long)c.E * c.P <= kLatencyNodes;
}

// Launch that may start before the stream's previous kernel has ended.  Only for
// meshes of up to 8 warps per SM: there a stage takes 2 to 3 us less (4^3: N = 1
// 17.4 -> 15.1, 2 17.3 -> 15.1, 3 18.8 -> 16.3; 5^3 N = 3 19.0 -> 18.6), with more
// the waiting blocks keep the running kernel's out (8^3 N = 2 23.8 -> 27.1).
constexpr int kEarlyWarpsPerSM = 8, kSMs = 152;
template <int N>
static bool early_launch(const Ctx& c) {
  return (long)c.E * ((LatShape<N>::THREADS + 31) / 32) <= (long)kEarlyWarpsPerSM * kSMs;
}
template <int N, typename... P, typename... A>
static cudaError_t launch_lat(const Ctx& c, void (*kernel)(P...), bool early, int grid, int block, size_t smem,
                              cudaStream_t s, A... args) {
  cudaLaunchAttribute at[1] = {};
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = early && early_launch<N>(c) ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

template <int N>
static cudaError_t lift_lat_N(const Ctx& c, const double* U, cudaStream_t s, bool early) {
  return launch_lat<N>(c, k_lift_lat<N>, early, c.E, LatShape<N>::THREADS, lift_lat_smem_bytes<N>(), s, U, c.d_metrics,
                       c.d_elem_nbr, c.d_elem_face, c.d_D, (double*)c.d_grad, c.E, c.gas, 1.0 / c.w[0]);
}

template <int N>
static cudaError_t volume_lat_N(const Ctx& c, const StageArgs& a, cudaStream_t s) {
  return launch_lat<N>(c, c.fx_stretch ? k_volume_lat<N, true> : k_volume_lat<N, false>, true, c.E, LatShape<N>::THREADS, volume_lat_smem_bytes<N>(), s, a, c.d_metrics,
                       c.d_jx, c.d_ejx, (const double*)c.d_grad, (const double*)c.d_fstar, c.d_elem_face, c.d_mms, c.d_D,
                       c.E, c.gas, 1.0 / c.w[0]);
}

cudaError_t launch_lift_lat(const Ctx& c, const double* U, cudaStream_t s, bool early) {
  switch (c.N) {
    case 1: return lift_lat_N<1>(c, U, s, early);
    case 2: return lift_lat_N<2>(c, U, s, early);
    case 3: return lift_lat_N<3>(c, U, s, early);
    default: return cudaErrorInvalidValue;
  }
}

template <int N>
static cudaError_t face_lat_N(const Ctx& c, const double* U, cudaStream_t s) {
  const long threads = 2L * c.nfaces * (N + 1) * (N + 1);
  return launch_lat<N>(c, k_face_lat<N>, true, (int)((threads + 63) / 64), 64, 0, s, U, (const double*)c.d_grad, c.d_faces,
                       c.d_facegeo, (double*)c.d_fstar, c.nfaces, c.gas);
}

cudaError_t launch_face_lat(const Ctx& c, const double* U, cudaStream_t s) {
  switch (c.N) {
    case 1: return face_lat_N<1>(c, U, s);
    case 2: return face_lat_N<2>(c, U, s);
    case 3: return face_lat_N<3>(c, U, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_volume_lat(const Ctx& c, const StageArgs& a, cudaStream_t s) {
  switch (c.N) {
    case 1: return volume_lat_N<1>(c, a, s);
    case 2: return volume_lat_N<2>(c, a, s);
    case 3: return volume_lat_N<3>(c, a, s);
    default: return cudaErrorInvalidValue;
  }
}

// Host reader of this file's bounds-check error word (0 in normal builds).
DG_BOUNDS_READER(bounds_word_latency)

}  // namespace dg
