// Sign coding of one row by one warp: rows of a matrix, patches that are coded one by one.
#pragma once

#include "common.cuh"

namespace dab {

// Sign code of a row by one warp; value(i) returns element i.
template <typename Value>
__device__ __forceinline__ void warp_sign_row(Value value, int n, int ld, int lane, int32_t* K_out, float* gamma_out,
                                              float* delta_out, uint32_t* flags_out, uint32_t* __restrict__ mrow) {
  double sum = 0.0;
  int ones = 0, bad = 0;
  uint32_t mine = 0;
  const int words = (n + 31) >> 5;
  for (int k = 0; k < words; ++k) {
    const int i = k * 32 + lane;
    float x = -1.0f;  // lanes beyond n contribute a 0 bit
    if (i < n) {
      x = value(i);
      bad |= is_nonfinite(x);
      sum += fabs((double)x);
    }
    const uint32_t word = __ballot_sync(0xFFFFFFFFu, i < n && x >= 0.0f);
    ones += __popc(word);
    if ((k & 31) == lane) mine = word;
    if ((k & 31) == 31 || k == words - 1) {  // a batch of up to 32 words is complete: one coalesced store
      const int w = (k & ~31) + lane;
      if (w <= k) mrow[w] = mine;
    }
  }
  for (int w = words + lane; w < ld; w += 32) mrow[w] = 0u;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, off);
  bad = __any_sync(0xFFFFFFFFu, bad);
  if (bad) {  // flagged rows: empty mask, NaN scales
    __syncwarp();
    for (int w = lane; w < ld; w += 32) mrow[w] = 0u;
  }
  if (lane == 0) {
    const float g = bad ? __uint_as_float(0x7FC00000u) : (float)(sum / (double)n);
    *K_out = bad ? 0 : ones;
    *gamma_out = g;
    *delta_out = -g;
    if (flags_out) *flags_out = bad ? DAB_ROW_NONFINITE : 0u;
  }
}

}  // namespace dab
