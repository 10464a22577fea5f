// The division of the absorbing layer as a product and two corrections.  Plain
// C++ as well, so that it can be compared with a division on the host.
#pragma once

#include <math.h>

#ifdef __CUDACC__
#define TP_HD __host__ __device__ __forceinline__
#else
#define TP_HD inline
#endif

namespace tp {

// n / b, b = 1 + a of the absorbing layer, with inv = 1 / b correctly rounded:
// two residual corrections give the correctly rounded quotient (Markstein 1990)
// while the residual does not underflow.  The values ahead of a wave are tiny
// over most of a layer; they are divided scaled by 2^96, and a subnormal result,
// then rounded a second time, moves to its other neighbour where the first
// rounding had made a tie.  Bit for bit n / b, but for the sign of a zero.  (A
// plain division, with its slow branch for zeros and tiny values, took 13 us of a
// 17 us step: 601 x 201, 16 shots.)
TP_HD float quotient(float n, float b, float inv) {
  const bool tiny = fabsf(n) < 0x1p-60f;
  if (tiny) n *= 0x1p96f;
  float q = n * inv;
  q = fmaf(fmaf(-q, b, n), inv, q);
  const float r = fmaf(-q, b, n);
  q = fmaf(r, inv, q);
  if (tiny) {
    const float s = q, d = s * 0x1p-96f, diff = fmaf(d, -0x1p96f, s);
    q = d;
    if (fabsf(diff) == 0x1p-54f && fmaf(-s, b, n) * diff > 0.f) q += copysignf(0x1p-149f, diff);
  }
  return fabsf(n) <= 3.402823466e38f ? q : n;  // infinities and NaN: no residual
}

}  // namespace tp
