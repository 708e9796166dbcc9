// Fixed-point data that do not depend on the state: the scale of the
// differentiation matrix, and the metric terms as integers.
#pragma once

#include "dg_check.cuh"
#include "dg_fixed.cuh"

namespace dg {

// |D| < 2^e_D for the differentiation matrix (and with the surface term in its
// corners), per degree: at most 0.5, 2.0, 4.05, 6.76, 10.2, 14.3, 19.0, 24.4, 30.5.
constexpr int fx_eD(int N) { return N == 1 ? 0 : (N == 2 ? 2 : (N <= 4 ? 3 : (N <= 6 ? 4 : 5))); }

__device__ __forceinline__ int fx_expo(int h) {   // |x| < 2^e from the high word of the largest |x|
  const int e = (h >> 20) - 1022;
  return e > -90 ? e : -90;
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
// Once per context: metric terms and 1/J as integers (jx [E][10][P]): rows
// 0..8 with 60 - e_j bits, e_j of the element's largest sum over l of |J
// a^d_l|; row 9 with 62 - e_i bits.  ej [E]: e_j, the logarithm of the largest
// sum less e_j (rounded up), e_i.  An element with exponents out of range, or
// with 1/J varying by more than 2^8, gets e_j = 1000: FP64 only.
// With facegeo (Gauss nodes, whose face points are not nodes) e_j covers the
// surface elements of the element's faces too.
template <int N>
__global__ void __launch_bounds__(256) k_fx_metrics(const double* __restrict__ metrics, i64* __restrict__ jx,
                                                    float4* __restrict__ ej, const double* __restrict__ facegeo,
                                                    const int* __restrict__ elem_face, int F) {
  constexpr int P = (N + 1) * (N + 1) * (N + 1), NN = (N + 1) * (N + 1);
  __shared__ unsigned s_max[3];
  const double* mt = metrics + (size_t)blockIdx.x * 10 * P;
  if (threadIdx.x < 3) s_max[threadIdx.x] = 0;
  __syncthreads();
  for (int id = threadIdx.x; id < P; id += blockDim.x) {
    for (int d = 0; d < 3; ++d) {
      const double s = fabs(mt[(d * 3) * P + id]) + fabs(mt[(d * 3 + 1) * P + id]) + fabs(mt[(d * 3 + 2) * P + id]);
      atomicMax(&s_max[0], (unsigned)__double2hiint(s) + 1u);   // above the sum; NaN stays above all
    }
    const unsigned h = (unsigned)__double2hiint(mt[9 * P + id]);
    atomicMax(&s_max[1], h);
    atomicMax(&s_max[2], 0x7fffffffu - h);
  }
  if (facegeo != nullptr)
    for (int t = threadIdx.x; t < 6 * NN; t += blockDim.x) {
      const int fid = dg_idx(elem_face[blockIdx.x * 6 + t / NN] >> 4, F, kSiteGeomFace);
      atomicMax(&s_max[0], (unsigned)__double2hiint(facegeo[((size_t)fid * 4 + 3) * NN + t % NN]) + 1u);
    }
  __syncthreads();
  const int h = (int)s_max[0], e = (h >> 20) - 1022, ei = (int)(s_max[1] >> 20) - 1022,
            emin = (int)((0x7fffffffu - s_max[2]) >> 20) - 1022;
  const bool fine = e > -90 && e < 90 && ei > -90 && ei < 90 && ei - emin <= 8;
  if (threadIdx.x == 0)
    ej[blockIdx.x] = make_float4(fine ? (float)e : 1000.0f, fx_log_mantissa(h, 1), (float)ei, 0.0f);
  for (int t = threadIdx.x; t < 10 * P; t += blockDim.x)
    jx[(size_t)blockIdx.x * 10 * P + t] = fine ? fx_from(mt[t], t < 9 * P ? kFxQ - e : 62 - ei) : 0;
}

}  // namespace dg
