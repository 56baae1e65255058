// Element operations of the Householder QR and Jacobi kernels.
#pragma once
#include "common.cuh"

namespace ttfit {

// The df32 square root and reciprocal start from the FP32 result of the high
// word and take one Newton step in df32 arithmetic, which doubles the number
// of correct bits (Dekker, Numer. Math. 18 (1971); Karp and Markstein, ACM
// TOMS 23 (1997)): sqrt(x) = s + (x - s^2) / (2 s), 1/x = r + r (1 - x r).
__device__ __forceinline__ float qsqrt(float x) { return sqrtf(x); }
__device__ __forceinline__ double qsqrt(double x) { return sqrt(x); }
__device__ __forceinline__ df32 qsqrt(df32 x) {
  if (!(x.hi > 0.0f)) return df32(0.0f, 0.0f);
  const float s = sqrtf(x.hi);
  const df32 e = madd(df32(-s, 0.0f), df32(s, 0.0f), x);  // x - s^2
  return two_sum(s, e.hi * (0.5f / s));
}
// 1/sqrt(x): FP32 from the hardware estimate and one Newton step (r (3 - x r^2) / 2)
__device__ __forceinline__ float qrsqrt(float x) {
  const float r = rsqrtf(x);
  return r * fmaf(-0.5f * x * r, r, 1.5f);
}
__device__ __forceinline__ double qrsqrt(double x) { return 1.0 / sqrt(x); }
__device__ __forceinline__ float qrcp(float x) { return 1.0f / x; }
__device__ __forceinline__ double qrcp(double x) { return 1.0 / x; }
__device__ __forceinline__ df32 qrcp(df32 x) {
  const df32 r(1.0f / x.hi, 0.0f);
  const df32 e = madd(-x, r, df32(1.0f, 0.0f));  // 1 - x r
  return madd(r, e, r);
}
__device__ __forceinline__ df32 qrsqrt(df32 x) { return qrcp(qsqrt(x)); }
__device__ __forceinline__ bool qneg(float x) { return x < 0.0f; }
__device__ __forceinline__ bool qneg(double x) { return x < 0.0; }
__device__ __forceinline__ bool qneg(df32 x) { return x.hi < 0.0f; }  // a normalised pair has the sign of hi
__device__ __forceinline__ bool qpos(float x) { return x > 0.0f; }
__device__ __forceinline__ bool qpos(double x) { return x > 0.0; }
__device__ __forceinline__ bool qpos(df32 x) { return x.hi > 0.0f; }
template <typename C>
__device__ __forceinline__ C qshfl_xor(C v, int m) {
  return __shfl_xor_sync(0xffffffffu, v, m);
}
template <>
__device__ __forceinline__ df32 qshfl_xor<df32>(df32 v, int m) {
  return df32(__shfl_xor_sync(0xffffffffu, v.hi, m), __shfl_xor_sync(0xffffffffu, v.lo, m));
}
template <typename C>
__device__ __forceinline__ C qshfl(C v, int src) {
  return __shfl_sync(0xffffffffu, v, src);
}
template <>
__device__ __forceinline__ df32 qshfl<df32>(df32 v, int src) {
  return df32(__shfl_sync(0xffffffffu, v.hi, src), __shfl_sync(0xffffffffu, v.lo, src));
}

// 1/sqrt(x) for x in [1, 2]: the hardware estimate refined by one Newton step
// r <- r + r (1 - x r^2) / 2, so that cs^2 + sn^2 = cs^2 (1 + t^2) is 1 to the
// FP32 rounding. An estimate left unrefined makes every rotation a rotation
// times sqrt(cs^2 + sn^2), and the accumulated right factor drifts away from
// orthonormal over the thousands of rotations of a decomposition.
__device__ __forceinline__ float rot_rsqrt(float x) {
  const float r = rsqrtf(x);
  return fmaf(0.5f * r, fmaf(-x * r, r, 1.f), r);
}

// x 2^s by the bits; zero below the normal numbers
__device__ __forceinline__ double shift_bits(double x, int s) {
  const int hi = __double2hiint(x), f = (hi >> 20) & 0x7FF, g = f + s;
  if (f == 0x7FF || s == 0) return x;
  if (f == 0 || g <= 0) return 0.0;
  if (g >= 0x7FF) return __hiloint2double((hi & (int)0x80000000) | 0x7FF00000, 0);
  return __hiloint2double(hi + (int)((unsigned)s << 20), __double2loint(x));
}

}  // namespace ttfit
