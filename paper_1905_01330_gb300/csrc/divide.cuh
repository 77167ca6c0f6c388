// Division by a scale that many numbers share, rounded as the division itself:
// the quotient by the rounded reciprocal, q = x r, corrected once by its
// residual, fma(fma(-q, s, x), r, q), is x / s rounded to nearest (Markstein,
// IBM J. Res. Dev. 34, 1990) unless the scale's mantissa is all ones, the
// quotient is not a normal number or the residual is not exact. It takes two
// FMAs and a product where the division takes about ten instructions; numbers
// near the ends of the exponent range, infinities and NaN are divided, out of
// line. (A negative zero comes out as zero.)
#pragma once

#include <cuda_runtime.h>

namespace tn {

static __device__ __noinline__ float divide_slow(float x, float s) { return __fdiv_rn(x, s); }

__device__ __forceinline__ float divide_corrected(float x, float s, float r) {
  const float q = x * r;
  return fmaf(fmaf(-q, s, x), r, q);
}

__device__ __forceinline__ bool full_mantissa(float s) { return (__float_as_uint(s) & 0x7FFFFFu) == 0x7FFFFFu; }

// v / s for |v| <= s, the scale the same in the whole warp. Quotients down to
// 2^-40 of a scale in (2^-60, 2^60): |v| > 2^-100, so a residual's last bit,
// at 2^-47 |v|, is not lost.
template <int N>
__device__ __forceinline__ void divide_by_max(float (&v)[N], float s) {
  const float r = __frcp_rn(s);
  bool plain = s > 0x1p-60f && s < 0x1p60f && !full_mantissa(s);
#pragma unroll
  for (int j = 0; j < N; ++j) plain = plain && (fabsf(v[j] * r) > 0x1p-40f || v[j] == 0.0f);
  if (__all_sync(__activemask(), plain)) {
#pragma unroll
    for (int j = 0; j < N; ++j) v[j] = divide_corrected(v[j], s, r);
  } else {
#pragma unroll
    for (int j = 0; j < N; ++j) v[j] = divide_slow(v[j], s);
  }
}

// v[i][:] / s[i]: scales in (2^-24, 2^24) and 0 or 2^-100 < |v| < 2^100, so
// quotients are normal and residuals exact. BOUNDED: no |v| is above its scale.
// The whole warp calls it; eight neighbouring lanes have the same scales and
// share out their reciprocals.
template <bool BOUNDED, int R, int N>
__device__ __forceinline__ void divide_rows(float (&v)[R][N], const float (&s)[R]) {
  static_assert(R == 2 || R == 4 || R == 8, "rows");
  const int lane = threadIdx.x & 31;
  // row lane % R's scale, by bits of the lane (an indexed choice goes through
  // local memory)
  float pick[R];
#pragma unroll
  for (int i = 0; i < R; ++i) pick[i] = s[i];
#pragma unroll
  for (int n = R / 2, bit = 1; n > 0; n /= 2, bit *= 2)
#pragma unroll
    for (int i = 0; i < n; ++i) pick[i] = (lane & bit) ? pick[2 * i + 1] : pick[2 * i];
  const float mine = pick[0];
  bool plain = mine > 0x1p-24f && mine < 0x1p24f && !full_mantissa(mine);
  unsigned least = 0xFFFFFFFFu;  // of the values without their signs, times 2, less 1: zeros come last
  float most = 0.0f;
#pragma unroll
  for (int i = 0; i < R; ++i)
#pragma unroll
    for (int j = 0; j < N; ++j) {
      least = min(least, __float_as_uint(v[i][j]) * 2u - 1u);
      if (!BOUNDED) most = fmaxf(most, fabsf(v[i][j]));
    }
  plain = plain && least >= 2u * __float_as_uint(0x1p-100f) && most < 0x1p100f;
  if (__all_sync(0xffffffffu, plain)) {
    const float mr = __frcp_rn(mine);
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const float r = __shfl_sync(0xffffffffu, mr, (lane & 24) | i);
#pragma unroll
      for (int j = 0; j < N; ++j) v[i][j] = divide_corrected(v[i][j], s[i], r);
    }
  } else {
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
      for (int j = 0; j < N; ++j) v[i][j] = divide_slow(v[i][j], s[i]);
  }
}

}  // namespace tn
