// Sums of a warp's lanes for the inner products of the vector kernels, in the vectors' own precision or in
// float32 pairs that keep what float32 rounds off.
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"

namespace swm {

// A float32 sum h and the part l of it that float32 could not hold.
struct FPair {
  float h, l;
};

// s + e = a + b exactly (D. E. Knuth, The Art of Computer Programming, vol. 2, 4.2.2, theorem B)
__host__ __device__ __forceinline__ FPair two_sum(float a, float b) {
  FPair r;
  r.h = a + b;
  const float t = r.h - a;
  r.l = (a - (r.h - t)) + (b - t);
  return r;
}
__host__ __device__ __forceinline__ FPair operator+(FPair a, FPair b) {
  FPair r = two_sum(a.h, b.h);
  r.l += a.l + b.l;
  return r;
}
// (a sum that has left float32's range has no remainder: h is the infinity or NaN itself)
__host__ __device__ __forceinline__ double widen(FPair a) {
  const double s = (double)a.h + (double)a.l;
  return s - s == 0.0 ? s : (double)a.h;
}
__host__ __device__ __forceinline__ double widen(float a) { return a; }
__host__ __device__ __forceinline__ double widen(double a) { return a; }

__device__ __forceinline__ FPair lane_xor(FPair a, int o) {
  return FPair{__shfl_xor_sync(0xffffffffu, a.h, o), __shfl_xor_sync(0xffffffffu, a.l, o)};
}
__device__ __forceinline__ float lane_xor(float a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ double lane_xor(double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }

// Sums over the warp of eight values: lanes 4 i .. 4 i + 3 return that of v[i].  Each of the first three
// exchanges halves the number of values a lane carries (9 additions for 8 sums; one sum after the other
// takes 40, which in float64 cost half as much as reading the rows).
template <typename T>
__device__ __forceinline__ T warp_sum8(const T (&v)[8], int lane) {
  const bool h = lane & 16, m = lane & 8, l = lane & 4;
  T p[4], q[2];
#pragma unroll
  for (int i = 0; i < 4; ++i) p[i] = (h ? v[i + 4] : v[i]) + lane_xor(h ? v[i] : v[i + 4], 16);
#pragma unroll
  for (int i = 0; i < 2; ++i) q[i] = (m ? p[i + 2] : p[i]) + lane_xor(m ? p[i] : p[i + 2], 8);
  T k = (l ? q[1] : q[0]) + lane_xor(l ? q[0] : q[1], 4);
  k = k + lane_xor(k, 2);
  return k + lane_xor(k, 1);
}

// sum_k conj(v_k) x_k over a lane's KR rows, re and im.  As pairs: four float32 sums of every fourth row,
// joined without rounding, so that no more than KR / 4 rows are added in float32 alone.
template <int KR, typename T>
__device__ __forceinline__ void lane_dot(const cplx<T> (&v)[KR], const cplx<T> (&x)[KR], T* o) {
  T re = T(0), im = T(0);
#pragma unroll
  for (int k = 0; k < KR; ++k) {
    re = fma(v[k].re, x[k].re, fma(v[k].im, x[k].im, re));
    im = fma(v[k].re, x[k].im, fma(-v[k].im, x[k].re, im));
  }
  o[0] = re;
  o[1] = im;
}
template <int KR>
__device__ __forceinline__ void lane_dot(const c64 (&v)[KR], const c64 (&x)[KR], FPair* o) {
  static_assert(KR % 4 == 0, "rows in fours");
  float re[4], im[4];
#pragma unroll
  for (int k = 0; k < KR; ++k) {
    const float r0 = k < 4 ? 0.f : re[k & 3], i0 = k < 4 ? 0.f : im[k & 3];
    re[k & 3] = fmaf(v[k].re, x[k].re, fmaf(v[k].im, x[k].im, r0));
    im[k & 3] = fmaf(v[k].re, x[k].im, fmaf(-v[k].im, x[k].re, i0));
  }
  o[0] = two_sum(re[0], re[1]) + two_sum(re[2], re[3]);
  o[1] = two_sum(im[0], im[1]) + two_sum(im[2], im[3]);
}

}  // namespace swm
