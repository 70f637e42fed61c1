// The bound the bucket-pruned searches share.  The objective D(s, P) = P^2/s + (T-P)^2/(n-s) of Algorithm 1 is jointly
// convex in (s, P).  While a split moves through a bucket (count c, sum S, values in [vlo, vhi)), (s, P) stays within a
// parallelogram whose corners are the bucket's two edges and two inner points, so D is largest at one of the four.
// Edges and inner corners are evaluated in fp32 from exact fp64 coordinates; a bucket is kept if its largest value
// reaches the best edge value times prune_margin.
#pragma once

#include "common.cuh"

namespace dab {

// Objective in fp32 from fp64 coordinates: every input is rounded once (relative 2^-24), both terms are
// non-negative, the two quotients are good to 2 ulp: the result is within 1e-6 relative of the exact value for
// results inside the normal fp32 range.  s = 0 and s = n stand for the limits (P = 0 resp. P = T there).
__device__ __forceinline__ float objective_bound(double s, double P, double T, double nd) {
  const float Pf = (float)P, Qf = (float)(T - P), sf = (float)s, rf = (float)(nd - s);
  const float a = sf > 0.0f ? __fdividef(Pf * Pf, sf) : 0.0f;
  const float b = rf > 0.0f ? __fdividef(Qf * Qf, rf) : 0.0f;
  return a + b;
}

// A candidate is kept if its fp32 value reaches best * prune_margin: with both sides within 1e-6 of their exact
// values, anything whose exact bound reaches the exact best edge value is kept.
constexpr float prune_margin = 0.99998f;

// Buckets that are ranges of bit patterns of the magnitude: [pattern << SHIFT, (pattern + 1) << SHIFT), the one next to
// zero (i = 0) from 0 on.  Value bounds of bucket i and the reciprocal of its width: exact for i > 0 (the width is a power
// of two), good to 2e-14 relative for i = 0.
template <int SHIFT>
__device__ __forceinline__ void bucket_range(int i, int pattern, bool negative, double& vlo, double& vhi, double& inv_width) {
  const float lo = i ? __uint_as_float((uint32_t)pattern << SHIFT) : 0.0f;
  const float hi = __uint_as_float((uint32_t)(pattern + 1) << SHIFT);
  vlo = negative ? -(double)hi : (double)lo;
  vhi = negative ? -(double)lo : (double)hi;
  const int biased = pattern >> (23 - SHIFT);  // exponent field of lo; the width is 2^(exponent - (23 - SHIFT))
  const double r = i ? (double)__int_as_float((254 + (23 - SHIFT) - biased) << 23) : (double)__fdividef(1.0f, hi);
  // one Newton step: leaves the exact reciprocals as they are and takes 1 / hi from 2 ulp of fp32 to 2e-14 relative
  inv_width = __dmul_rn(r, __dsub_rn(2.0, __dmul_rn(vhi - vlo, r)));
}

// Larger of the objective's values at the two inner corners of a bucket with c >= 2 values of sum S, s0 elements with sum
// P0 before it.
template <int SHIFT>
__device__ __forceinline__ float bucket_corner_bound(int i, int pattern, bool negative, int s0, int c, double P0, double S,
                                                     double T, double nd) {
  double vlo, vhi, inv_width;
  bucket_range<SHIFT>(i, pattern, negative, vlo, vhi, inv_width);
  const double cd = (double)c;
  double jl = (cd * vhi - S) * inv_width;
  jl = fmin(fmax(jl, 0.0), cd);
  const double ju = cd - jl;
  return fmaxf(objective_bound((double)s0 + jl, P0 + jl * vlo, T, nd), objective_bound((double)s0 + ju, P0 + ju * vhi, T, nd));
}

// Smallest and largest order_key of bucket b (buckets 0 .. NB-1 negative, descending magnitude; NB .. positive); base:
// pattern of i = 0.  Zero itself lies in neither of the two buckets next to it.
template <int SHIFT>
__device__ __forceinline__ uint32_t bucket_first_key(int b, int NB, int base) {
  if (b < NB) return order_key(-__uint_as_float((uint32_t)(NB - 1 - b + base + 1) << SHIFT)) + 1u;
  return b == NB ? 0x80000001u : order_key(__uint_as_float((uint32_t)(b - NB + base) << SHIFT));
}
template <int SHIFT>
__device__ __forceinline__ uint32_t bucket_last_key(int b, int NB, int base) {
  if (b < NB) return b == NB - 1 ? 0x7FFFFFFFu : order_key(-__uint_as_float((uint32_t)(NB - 1 - b + base) << SHIFT));
  return order_key(__uint_as_float((uint32_t)(b - NB + base + 1) << SHIFT)) - 1u;
}

}  // namespace dab
