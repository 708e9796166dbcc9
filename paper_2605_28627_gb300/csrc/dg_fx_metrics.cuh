// Fixed-point data that do not depend on the state: the scale of the
// differentiation matrix, and the metric terms as integers.
#pragma once

#include "dg_check.cuh"
#include "dg_fixed.cuh"

namespace dg {

// |D| < 2^e_D for the differentiation matrix (and with the surface term in its
// corners), per degree: at most 0.5, 2.0, 4.05, 6.76, 10.2, 14.3, 19.0, 24.4, 30.5.
constexpr int fx_eD(int N) { return N == 1 ? 0 : (N == 2 ? 2 : (N <= 4 ? 3 : (N <= 6 ? 4 : 5))); }

// |x| < 2^e from the high word of the largest |x|; a quantity that is zero all
// over the element gets kFxLow.
constexpr int kFxLow = -200;
__host__ __device__ __forceinline__ int fx_expo(int h) {
  const int e = (h >> 20) - 1022;
  return e > kFxLow ? e : kFxLow;
}
// Whether fixed point may hold the quantity: zero, or 2^kFxLow <= 2^e < 2^high
// (scaled below 2^kFxLow it would lose digits).
__host__ __device__ __forceinline__ bool fx_in_range(int h, int high) {
  constexpr int low = (kFxLow + 1022) << 20;
  return ((unsigned)(h - low) < (unsigned)((high - kFxLow) << 20)) | (h == 0);
}
__device__ __forceinline__ int fx_mag(double x) { return __double2hiint(x) & 0x7fffffff; }
// maxima of v[0..C) over the lanes of element el of this warp, into mx[0..C)
template <int C>
__device__ __forceinline__ void fx_maxima(int el, int* mx, const int v[C]) {
  const unsigned lanes = __match_any_sync(__activemask(), el);
  const bool first = (int)(threadIdx.x & 31) == __ffs(lanes) - 1;
#pragma unroll
  for (int c = 0; c < C; ++c) {
    const unsigned r = __reduce_max_sync(lanes, (unsigned)v[c]);
    if (first) atomicMax(&mx[c], (int)r);
  }
}

// logarithm (base 2) less the exponent e of a positive double with high word
// h, from below (up = 0) or above (up = 1); in -1..0 for e of fx_element
__device__ __forceinline__ float fx_log_mantissa(int h, int up) {
  return __log2f(__int_as_float((((h & 0xfffff) + up) << 3) + 0x3f800000)) - 1.0f + (up ? 1e-5f : -1e-5f);
}
// Shifts of one element's metric terms, packed with their exponents (ej.w of
// k_fx_metrics): jx holds all rows with 60 - e_j bits; a direction's three rows
// are shifted up by t for the volume terms (its largest sum over l is 2^t to
// 2^(t+1) below the largest direction's; 0 for cells of ratio below 2, so that
// those skip the shifts), a column's three (component l of every direction) by c
// for the lifting: to the column's own exponent on LGL nodes, like t on Gauss
// nodes; order: the directions by falling t.
struct FxMetricShifts {
  int w;
  __device__ int t(int d) const { return (w >> (4 * d)) & 15; }
  __device__ int c(int l) const { return (w >> (12 + 4 * l)) & 15; }
  __device__ int order(int x) const { return (w >> (24 + 2 * x)) & 3; }
  // the directions' order (2 bits each) and by how much the sums move down after
  // each (4 bits each, from bit 8)
  __device__ int walk() const {
    const int a = t(order(0)), b = t(order(1)), c = t(order(2));
    return (w >> 24 & 63) | (a - b) << 8 | (b - c) << 12 | c << 16;
  }
};
__device__ __forceinline__ FxMetricShifts fx_shifts(float4 ej) { return FxMetricShifts{__float_as_int(ej.w)}; }
// (p + c 2^-32) / 2^k, c in [0, 2^32), 0 <= k <= 31
__device__ __forceinline__ void fx_shift_down(FxSum& s, int k) {
  const unsigned lo = (unsigned)(u64)s.p;
  s.c = (i64)__funnelshift_r((unsigned)(u64)s.c, lo, k);
  s.p >>= k;
}
// A fixed-point element's directions differ by less than 2^(kFxStretch + 1) in
// size, the nodes of one direction by kFxVary.  Beyond, the exponents that the
// directions share in the fields cost digits: of a small velocity across long
// faces, and by the pressure's rounding in the other momenta.  Error of R(U) over
// the FP64 kernels', rms, boundary-layer flows on cells of ratio A: at most 1.1 to
// 1.2 for A = 3.9 (1.0 to 1.1 for cubic cells), 1.6 to 2.4 for A = 15.
constexpr int kFxStretch = 1;
constexpr double kFxVary = 16.0;

// Once per context: metric terms and 1/J as integers (jx [E][10][P]): rows
// 0..8 with 60 - e_j bits, e_j of the element's largest sum over l of |J
// a^d_l|; row 9 with 62 - e_i bits.  ej [E]: e_j, the logarithm of the largest
// sum less e_j (rounded up), e_i, FxMetricShifts.  An element with exponents out
// of range, with 1/J varying by more than 2^8 or stretched beyond kFxStretch gets
// e_j = 1000: FP64 only; so does every element if there is no jx (null).
// With facegeo (Gauss nodes, whose face points are not nodes) e_j and c cover
// the surface elements of the element's faces too.  *stretch: set if any element
// in range has a t (on Gauss nodes a t or a c) other than 0.
template <int N>
__global__ void __launch_bounds__(256) k_fx_metrics(const double* __restrict__ metrics, i64* __restrict__ jx,
                                                    float4* __restrict__ ej, const double* __restrict__ facegeo,
                                                    const int* __restrict__ elem_face, int F, int* __restrict__ stretch) {
  constexpr int P = (N + 1) * (N + 1) * (N + 1), NN = (N + 1) * (N + 1);
  // largest sum, 1/J and its complement; per direction the largest sum and the
  // complement of the smallest; per column the largest term
  __shared__ unsigned s_max[3], s_row[3], s_rowmin[3], s_col[3];
  const double* mt = metrics + (size_t)blockIdx.x * 10 * P;
  if (threadIdx.x < 3) s_max[threadIdx.x] = s_row[threadIdx.x] = s_rowmin[threadIdx.x] = s_col[threadIdx.x] = 0;
  __syncthreads();
  auto above = [](double x) { return (unsigned)__double2hiint(fabs(x)) + 1u; };   // NaN stays above all
  for (int id = threadIdx.x; id < P; id += blockDim.x) {
    for (int d = 0; d < 3; ++d) {
      const double j[3] = {mt[(d * 3) * P + id], mt[(d * 3 + 1) * P + id], mt[(d * 3 + 2) * P + id]};
      const unsigned h = above(fabs(j[0]) + fabs(j[1]) + fabs(j[2]));
      atomicMax(&s_row[d], h);
      atomicMax(&s_rowmin[d], 0x7fffffffu - (h - 1u));
      for (int l = 0; l < 3; ++l) atomicMax(&s_col[l], above(j[l]));
    }
    const unsigned h = (unsigned)__double2hiint(mt[9 * P + id]);
    atomicMax(&s_max[1], h);
    atomicMax(&s_max[2], 0x7fffffffu - h);
  }
  if (facegeo != nullptr)
    for (int t = threadIdx.x; t < 6 * NN; t += blockDim.x) {
      const int fid = dg_idx(elem_face[blockIdx.x * 6 + t / NN] >> 4, F, kSiteGeomFace);
      const double* fg = facegeo + (size_t)fid * 4 * NN + t % NN;
      const double sJ = fg[3 * NN];
      atomicMax(&s_max[0], above(sJ));
      for (int l = 0; l < 3; ++l) atomicMax(&s_col[l], above(sJ * fg[l * NN]));
    }
  __syncthreads();
  auto expo = [](unsigned h) { return (int)(h >> 20) - 1022; };
  auto size = [](unsigned h) { return __hiloint2double((int)h, 0); };
  const unsigned most = max(s_row[0], max(s_row[1], s_row[2])), h = max(most, s_max[0]);
  const int e = expo(h), ei = expo(s_max[1]), emin = expo(0x7fffffffu - s_max[2]);
  bool fine = jx != nullptr && e > -90 && e < 90 && ei > -90 && ei < 90 && ei - emin <= 8;
  int t[3], w = 0;
  for (int d = 0; d < 3; ++d) {
    t[d] = expo(most) - expo(s_row[d]);
    if (t[d] > 0 && size(s_row[d] + (t[d] << 20)) > size(most)) --t[d];
    fine = fine && t[d] <= kFxStretch && size(s_row[d]) <= kFxVary * size(0x7fffffffu - s_rowmin[d]);
    int c = e - expo(s_col[d]);
    if (facegeo != nullptr && c > 0 && size(s_col[d] + (c << 20)) > size(h)) --c;
    w |= t[d] << (4 * d) | min(c, 15) << (12 + 4 * d);
  }
  if (threadIdx.x == 0 && fine && (w & (facegeo != nullptr ? 0xffffff : 0xfff)) != 0) atomicOr(stretch, 1);
  for (int d = 0; d < 3; ++d) {   // place of direction d among the falling t
    int place = 0;
    for (int x = 0; x < 3; ++x) place += x != d && (t[x] > t[d] || (t[x] == t[d] && x < d));
    w |= d << (24 + 2 * place);
  }
  if (threadIdx.x == 0)
    ej[blockIdx.x] = make_float4(fine ? (float)e : 1000.0f, fx_log_mantissa((int)h, 1), (float)ei, __int_as_float(fine ? w : 0));
  for (int x = threadIdx.x; jx != nullptr && x < 10 * P; x += blockDim.x)
    jx[(size_t)blockIdx.x * 10 * P + x] = fine ? fx_from(mt[x], x < 9 * P ? kFxQ - e : 62 - ei) : 0;
}

}  // namespace dg
