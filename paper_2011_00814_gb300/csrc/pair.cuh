// pair.cuh -- phi as an FP32 high/low pair: the sums of the compensated
// accumulation.
//
// Every sum and product that carries rounding is taken with its error: two-sum
// (Knuth) for sums, the fused multiply-add (Dekker's product) for products.  What
// is lost is the rounding of the new low part, half an ulp of it, which the
// same sum taken in FP64 and stored as a pair loses too; the terms past the
// first two orders add 2^-70 of the largest summand.  So the pair is never
// further from the exact sum than an FP64 sum's would be, whatever the sizes of
// phi and its increment.
// GB300's FP64 pipe is 64 times narrower than its FP32 one: with this sum in
// FP64 the last CH stage of 101 x 75 x 130 took 42 us, the stages before it 24.
#pragma once

#include <cmath>

#ifdef __CUDACC__
#define GPE2P_HD __host__ __device__ __forceinline__
#else
#define GPE2P_HD inline  // (a host compiler must not contract: -ffp-contract=off)
#endif

namespace gpe2p {

// sums and products that are not to be fused
GPE2P_HD float rn_add(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fadd_rn(a, b);
#else
  return a + b;
#endif
}
GPE2P_HD float rn_mul(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fmul_rn(a, b);
#else
  return a * b;
#endif
}

// s + e = a + b exactly
GPE2P_HD void two_sum(float a, float b, float& s, float& e) {
  const float r = rn_add(a, b), t = rn_add(r, -a);
  e = rn_add(rn_add(a, -rn_add(r, -t)), rn_add(b, -t));
  s = r;
}

// ph + q + the terms y + tail as a pair (y: terms of second order, at most half an ulp of
// ph or q each; tail: of third).  The last sum needs no two-sum: where t is not the
// larger summand it is what a cancellation left, a multiple of an ulp of ph or
// q and so of any ulp of s, and the shorter form (Dekker) is exact as well.
template <int N>
GPE2P_HD void pair_sum(float ph, float q, const float (&y)[N], float tail, float& hi, float& low) {
  float t, s, e;
  two_sum(ph, q, t, s);
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int i = 0; i < N; ++i) {
    two_sum(s, y[i], s, e);
    tail = rn_add(tail, e);
  }
  hi = rn_add(t, s);
  low = rn_add(rn_add(s, -rn_add(hi, -t)), tail);
}

// ph + lo + (a + d) / 2
GPE2P_HD void pair_half(float ph, float lo, float a, float d, float& hi, float& low) {
  float s, se;
  two_sum(a, d, s, se);
  const float y[2] = {lo, rn_mul(0.5f, se)};
  pair_sum(ph, rn_mul(0.5f, s), y, 0.0f, hi, low);
}

// ph + lo + (a + d) / 6, the sixth as three floats
GPE2P_HD void pair_sixth(float ph, float lo, float a, float d, float& hi, float& low) {
  constexpr float c0 = (float)(1.0 / 6.0), c1 = (float)(1.0 / 6.0 - (double)c0);
  constexpr float c2 = (float)((1.0 - 6.0 * ((double)c0 + (double)c1)) / 6.0);
  float s, se;
  two_sum(a, d, s, se);
  const float p0 = rn_mul(s, c0), p1 = rn_mul(s, c1), p2 = rn_mul(se, c0);
  const float y[4] = {lo, fmaf(s, c0, -p0), p1, p2};
  const float tail = fmaf(s, c2, fmaf(se, c1, rn_add(fmaf(s, c1, -p1), fmaf(se, c0, -p2))));
  pair_sum(ph, p0, y, tail, hi, low);
}

}  // namespace gpe2p
