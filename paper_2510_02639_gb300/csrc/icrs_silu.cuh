// SiLU z / (1 + e^-z) and its derivative, N values at a time.
//
// The SiLU bounds the inference kernel, and a division costs more than the rest
// of it.  For |z| < 80 (1 + e^-z below 2^126, where the hardware's approximate
// reciprocal r of d = 1 + e^-z has a relative error of at most 2^-23) the quotient is
// q = z r, corrected once by its remainder, q + r (z - q d) (Markstein, IBM J.
// Res. Dev. 34, 111, 1990); the reciprocal itself by one Newton step, r + r (1 -
// d r).  Both corrections multiply the error, below 2^-22, by that of r, so what the
// last rounding sees is off by less than 2^-44 of itself: the result is within
// an ulp of the rounded division, and differs from it only where the quotient
// lies within 2^-20 ulp of the middle between two floats.  Where one of the N
// values is larger, infinite included, the division itself.  (NaN compares
// as not larger; the arithmetic keeps it.)
//
// Inference of 2^20 queries 343 us, with the division everywhere 499; a training
// step over 8192 samples 84.6 us and 95.3.  (Paired operations around the two
// exponentials were slower: 356 us against 341.)
#pragma once

#include "icrs_common.cuh"

namespace icrs {

constexpr float SILU_FAST_MAX = 80.0f;

template <int N>
__device__ __forceinline__ bool silu_all_fast(const float* z) {
  float m = 0.0f;
#pragma unroll
  for (int j = 0; j < N; ++j) m = fmaxf(m, fabsf(z[j]));
  return m < SILU_FAST_MAX;
}

// z[j] <- SiLU(z[j])
template <int N>
__device__ __forceinline__ void silu_n(float* z) {
  if (silu_all_fast<N>(z)) {
#pragma unroll
    for (int j = 0; j < N; ++j) {
      const float d = 1.0f + expf(-z[j]), r = rcp_fast(d), q = z[j] * r;
      z[j] = fmaf(fmaf(-q, d, z[j]), r, q);
    }
  } else {
#pragma unroll
    for (int j = 0; j < N; ++j) z[j] = z[j] / (1.0f + expf(-z[j]));
  }
}

// v[j] <- v[j] SiLU'(z[j]), SiLU' = s (1 + z (1 - s)), s = 1 / (1 + e^-z)
template <int N>
__device__ __forceinline__ void silu_prime_n(const float* z, float* v) {
  if (silu_all_fast<N>(z)) {
#pragma unroll
    for (int j = 0; j < N; ++j) {
      const float d = 1.0f + expf(-z[j]), r = rcp_fast(d), s = fmaf(fmaf(-d, r, 1.0f), r, r);
      v[j] *= s * (1.0f + z[j] * (1.0f - s));
    }
  } else {
#pragma unroll
    for (int j = 0; j < N; ++j) {
      const float s = 1.0f / (1.0f + expf(-z[j]));
      v[j] *= s * (1.0f + z[j] * (1.0f - s));
    }
  }
}

}  // namespace icrs
