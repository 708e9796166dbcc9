// Lifting body of the FP64 operator in block fixed point (dg_fixed.cuh): the
// same terms as lift_body<N, double>.  The primitives (14 FP64 operations a
// node, and as many a face point) stay FP64 and run beside the integer work;
// the jumps, line sums, metric products and the scaling by 1/J are integer.
//
// Bound and measured: lift_body<N, double> held the FP64 pipe 93 % busy (150
// FP64 instructions a node at N = 7); here about 25 are left, and the integer
// part takes some 1300 issue slots a node.  Two 512-thread blocks per SM (64
// registers, a word spilled) at N = 7: three (42 registers) 251 us, one 331.
// Manufactured solution, 16^3 elements, us per launch before -> now: N = 1 18 ->
// 17, 2 42 -> 29, 3 73 -> 39, 4 144 -> 70, 5 250 -> 104, 6 415 -> 189, 7 627 ->
// 243, 8 970 -> 472, 9 1393 -> 639.
#pragma once

#include "dg_fx_metrics.cuh"
#include "dg_stage.cuh"

namespace dg {

template <int N, int EPB>
constexpr size_t lift_fx_smem_bytes() {
  // D, [EPB][2][P] pairs (u, v), (w, T), [EPB][6][4][n^2] face jumps
  return 8 * ((((N + 1) * (N + 1) + 1) & ~1) + (size_t)EPB * (4 * (N + 1) * (N + 1) * (N + 1) + 24 * (N + 1) * (N + 1)));
}

// MORTAR as in lift_body.  Elements outside the fixed-point range (a
// non-finite state, velocity or temperature outside 2^kFxLow to 2^90, e_j = 1000) get lift_body's FP64
// arithmetic from the same block.
template <int N, int EPB, bool MORTAR = false>
__device__ __forceinline__ void lift_body_fx(const double* __restrict__ U, const double* __restrict__ metrics,
                                             const i64* __restrict__ jx, const float4* __restrict__ ejx,
                                             const int* __restrict__ elem_nbr, const int* __restrict__ elem_face,
                                             const double* __restrict__ Dg, double* __restrict__ grad, int E,
                                             const Gas& g, double inv_w0, int blk,
                                             const double* __restrict__ mvirt = nullptr, int n_mortar = 0) {
  using S = Shape<N, EPB>;
  constexpr int n = S::n, P = S::P, NN = S::NN, NF = 6 * NN, eD = fx_eD(N);
  constexpr int NI = (EPB * NF + S::THREADS - 1) / S::THREADS;
  extern __shared__ __align__(16) unsigned char lift_raw[];
  Fx* sD = reinterpret_cast<Fx*>(lift_raw);
  longlong2* sphi = reinterpret_cast<longlong2*>(reinterpret_cast<i64*>(lift_raw) + ((n * n + 1) & ~1));   // [EPB][2][P]
  i64* sjmp = reinterpret_cast<i64*>(sphi + EPB * 2 * P);                                                   // [EPB][6][4][NN]
  __shared__ int s_mx[EPB][2];                  // high words of the largest velocity component and temperature
  const int le = threadIdx.x / P, id = threadIdx.x % P;
  const int e = blk * EPB + le;
  const bool active = e < E;
  auto load_nbr = [&](int t, double qv[5]) {
    const int le2 = t / NF, r2 = t - le2 * NF;
    const int e2 = blk * EPB + le2;
    if (t < EPB * NF && e2 < E) {
      const int f = r2 / NN, pq = r2 - f * NN;
      const int code = elem_face[e2 * 6 + f], nb = elem_nbr[e2 * 6 + f];
      if constexpr (MORTAR) {
        if (nb < 0) {
          const double* q = mvirt + (size_t)dg_idx(-1 - nb, 5L * n_mortar, kSiteMortar) * 5 * NN + pq;
#pragma unroll
          for (int v = 0; v < 5; ++v) qv[v] = q[v * NN];
          return;
        }
      }
      int p2, q2;
      apply_flip<n>(code & 7, pq % n, pq / n, p2, q2);
      const int enb = dg_idx(nb >> 3, E, kSiteLiftNbr);
      const double* q = U + (size_t)enb * 5 * P + face_node<n>(nb & 7, p2, q2);
#pragma unroll
      for (int v = 0; v < 5; ++v) qv[v] = q[v * P];
    }
  };
  // (u, v, w, T) of a conservative state
  auto lifted = [&](const double q[5], double phi[4]) {
    const double ir = rcp_op(q[0]);
    phi[0] = q[1] * ir;
    phi[1] = q[2] * ir;
    phi[2] = q[3] * ir;
    const double p = g.gm1 * (q[4] - 0.5 * (q[1] * phi[0] + q[2] * phi[1] + q[3] * phi[2]));
    phi[3] = p * ir * g.inv_R;
  };
  auto mag = [](double x) { return __double2hiint(x) & 0x7fffffff; };
  double phi[4] = {0, 0, 0, 0};
  double qn[5] = {1, 0, 0, 0, 0};
  if constexpr (NI == 1) load_nbr(threadIdx.x, qn);
  for (int t = threadIdx.x; t < n * n; t += blockDim.x) sD[t] = fx_split(fx_round(Dg[t], kFxQD - eD));
  for (int t = threadIdx.x; t < EPB * 2; t += blockDim.x) s_mx[t >> 1][t & 1] = 0;
  if (active) {
    double q[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) q[v] = U[((size_t)e * 5 + v) * P + id];
    lifted(q, phi);
  }
  __syncthreads();
  auto maxima = [&](int el, const double f[4]) {   // into s_mx[el], lanes of one element together
    const unsigned lanes = __match_any_sync(__activemask(), el);
    const unsigned a = __reduce_max_sync(lanes, (unsigned)max(max(mag(f[0]), mag(f[1])), mag(f[2])));
    const unsigned b = __reduce_max_sync(lanes, (unsigned)mag(f[3]));
    if ((int)(threadIdx.x & 31) == __ffs(lanes) - 1) {
      atomicMax(&s_mx[el][0], (int)a);
      atomicMax(&s_mx[el][1], (int)b);
    }
  };
  if (active) maxima(le, phi);
  // the neighbours' values at the face points, whole warps over them
#pragma unroll 1
  for (int it = 0; it < NI; ++it) {
    const int t = threadIdx.x + it * S::THREADS;
    const int le2 = t / NF, r2 = t - le2 * NF;
    if constexpr (NI > 1) load_nbr(t, qn);
    if (t < EPB * NF && blk * EPB + le2 < E) {
      const int f = r2 / NN, pq = r2 - f * NN;
      double o[4];
      lifted(qn, o);
      maxima(le2, o);
#pragma unroll
      for (int a = 0; a < 4; ++a) sjmp[((le2 * 6 + f) * 4 + a) * NN + pq] = __double_as_longlong(o[a]);
    }
  }
  __syncthreads();
  // exponents of velocity and temperature; range of the element
  const int eu = fx_expo(s_mx[le][0]), et = fx_expo(s_mx[le][1]);
  const float4 ej = active ? ejx[e] : make_float4(1000.0f, 0.0f, 0.0f, 0.0f);
  const bool ok = fx_in_range(s_mx[le][0], 90) && fx_in_range(s_mx[le][1], 90) && ej.x < 90.0f;
  if (active) {
    if (ok) {
      sphi[le * 2 * P + id] = make_longlong2(fx_from(phi[0], kFxQ - eu), fx_from(phi[1], kFxQ - eu));
      sphi[(le * 2 + 1) * P + id] = make_longlong2(fx_from(phi[2], kFxQ - eu), fx_from(phi[3], kFxQ - et));
    } else {
      sphi[le * 2 * P + id] = make_longlong2(__double_as_longlong(phi[0]), __double_as_longlong(phi[1]));
      sphi[(le * 2 + 1) * P + id] = make_longlong2(__double_as_longlong(phi[2]), __double_as_longlong(phi[3]));
    }
  }
  __syncthreads();
  // face jumps (phi_nbr - phi)/2 (+-1/w_0)
#pragma unroll 1
  for (int it = 0; it < NI; ++it) {
    const int t = threadIdx.x + it * S::THREADS;
    const int le2 = t / NF, r2 = t - le2 * NF;
    if (t < EPB * NF && blk * EPB + le2 < E) {
      const int f = r2 / NN, pq = r2 - f * NN;
      const int node = face_node<n>(f, pq % n, pq / n);
      const double hs = (f & 1) ? 0.5 * inv_w0 : -0.5 * inv_w0;
      i64* sj = sjmp + (le2 * 6 + f) * 4 * NN + pq;
      const longlong2 p0 = sphi[le2 * 2 * P + node], p1 = sphi[(le2 * 2 + 1) * P + node];
      const i64 own[4] = {p0.x, p0.y, p1.x, p1.y};
      const int eu2 = fx_expo(s_mx[le2][0]), et2 = fx_expo(s_mx[le2][1]);
      if (fx_in_range(s_mx[le2][0], 90) && fx_in_range(s_mx[le2][1], 90) && ejx[blk * EPB + le2].x < 90.0f) {
        const Fx hx = fx_split(fx_round(hs, kFxQD - eD));
#pragma unroll
        for (int a = 0; a < 4; ++a)
          sj[a * NN] = fx_mul<0>(fx_split(fx_from(__longlong_as_double(sj[a * NN]), kFxQ - (a < 3 ? eu2 : et2)) - own[a]), hx);
      } else {
#pragma unroll
        for (int a = 0; a < 4; ++a)
          sj[a * NN] = __double_as_longlong((__longlong_as_double(sj[a * NN]) - __longlong_as_double(own[a])) * hs);
      }
    }
  }
  __syncthreads();
  if (!active) return;
  const int i = id % n, j = (id / n) % n, k = id / NN;
  const longlong2* ph = sphi + le * 2 * P;
  double* go = grad + (size_t)e * 12 * P + id;
  if (!ok) {
    // FP64 arithmetic, as lift_body
    auto val = [&](int a, int node) {
      const longlong2 v = ph[(a >> 1) * P + node];
      return __longlong_as_double((a & 1) ? v.y : v.x);
    };
    const double* mt = metrics + (size_t)e * 10 * P + id;
    const double iJ = mt[9 * P];
#pragma unroll 1
    for (int a = 0; a < 4; ++a) {
      double dd[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const int r = d == 0 ? i : (d == 1 ? j : k), stride = d == 0 ? 1 : (d == 1 ? n : NN);
        double s = 0.0;
        if (r == 0 || r == N)
          s = __longlong_as_double(sjmp[((le * 6 + 2 * d + (r == N ? 1 : 0)) * 4 + a) * NN + (d == 0 ? j : i) +
                                        n * (d == 2 ? j : k)]);
#pragma unroll 1
        for (int m = 0; m < n; ++m) s += Dg[r * n + m] * val(a, id + (m - r) * stride);
        dd[d] = s;
      }
#pragma unroll
      for (int l = 0; l < 3; ++l)
        go[(a * 3 + l) * P] = (mt[l * P] * dd[0] + mt[(3 + l) * P] * dd[1] + mt[(6 + l) * P] * dd[2]) * iJ;
    }
    return;
  }
  // line sums D phi + jump
  i64 dd[4][3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int r = d == 0 ? i : (d == 1 ? j : k), stride = d == 0 ? 1 : (d == 1 ? n : NN);
    const i64* jm = sjmp + (le * 6 + 2 * d + (r == N ? 1 : 0)) * 4 * NN + (d == 0 ? j : i) + n * (d == 2 ? j : k);
    const bool edge = r == 0 || r == N;
    FxSum s[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) s[a] = fx_lift_start(edge ? jm[a * NN] : 0);
    const longlong2* line = ph + id - r * stride;
#pragma unroll
    for (int m = 0; m < n; ++m) {
      const Fx D = sD[r * n + m];
      const longlong2 p0 = line[m * stride], p1 = line[P + m * stride];
      fx_add(s[0], D, fx_split(p0.x));
      fx_add(s[1], D, fx_split(p0.y));
      fx_add(s[2], D, fx_split(p1.x));
      fx_add(s[3], D, fx_split(p1.y));
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) dd[a][d] = fx_lift_line(s[a]);
  }
  // g_l = (1/J) sum_d Ja^d_l dd_d
  const i64* mt = jx + (size_t)e * 10 * P + id;
  const Fx iJ = fx_split(mt[9 * P]);
  const FxMetricShifts sh = fx_shifts(ej);
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    const int c = sh.c(l), qg = fx_lift_bits(eD, (int)ej.x - c, (int)ej.z);   // less e
    const Fx J[3] = {fx_split(fx_up(mt[l * P], c)), fx_split(fx_up(mt[(3 + l) * P], c)),
                     fx_split(fx_up(mt[(6 + l) * P], c))};
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const Fx x[3] = {fx_split(dd[a][0]), fx_split(dd[a][1]), fx_split(dd[a][2])};
      go[(a * 3 + l) * P] = fx_to(fx_lift_gradient(J, x, iJ), qg - (a < 3 ? eu : et));
    }
  }
}

// Shared memory of the lifting body in either operator type.
template <int N, typename R, int EPB>
constexpr size_t lift_op_smem_bytes() {
  if constexpr (sizeof(R) == 8) return lift_fx_smem_bytes<N, EPB>();
  else return lift_smem_bytes<N, R, EPB>();
}

}  // namespace dg
