// Test-only kernel: the bounded barrier wait of the tensor-core kernels (tc::mbar_wait) made to run out.
// One thread initialises an mbarrier that nothing ever arrives on and waits on it with a limit of a few
// thousand cycles; the wait must return false, set the caller's `dead` flag, bump the failure counter once per
// waiting thread, make later waits return at once, and the kernel must end.  No tensor-core instruction is used.
#include <cuda_runtime.h>
#include <stdint.h>

#include "tc.cuh"

__global__ void wait_timeout_kernel(long long limit, unsigned int* failures, int* out) {
  __shared__ __align__(8) unsigned long long bar;
  const uint32_t bar_addr = dab::tc::smem_u32(&bar);
  if (threadIdx.x == 0) dab::tc::mbar_init(bar_addr, 1);
  __syncthreads();
  bool dead = false;
  const long long t0 = clock64();
  const bool first = dab::tc::mbar_wait(bar_addr, 0, dead, failures, limit);
  const long long waited = clock64() - t0;
  const bool second = dab::tc::mbar_wait(bar_addr, 0, dead, failures, limit);  // must not wait again
  __syncthreads();  // every thread still reaches the barriers that follow a failed wait
  if (threadIdx.x == 0) {
    out[0] = first ? 1 : 0;
    out[1] = second ? 1 : 0;
    out[2] = dead ? 1 : 0;
    out[3] = waited >= limit ? 1 : 0;
  }
}

// The hand-over of two alternating stages from producer warps to a consumer warp (tc::stage_handover), on barriers that no product
// ever completes: from its third stage on every producer's wait runs out.  The consumer is slower than the producers; it must
// still meet each of them exactly once per stage, and the kernel must end.  out[stage]: producers that had filled exactly that
// stage when the consumer took it.
__global__ void handover_timeout_kernel(int stages, long long limit, unsigned int* failures, int* out) {
  __shared__ __align__(8) unsigned long long bars[2];
  __shared__ int filled[2][32];
  const int producers = (int)blockDim.x - 32, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t bar0 = dab::tc::smem_u32(&bars[0]);
  if (threadIdx.x == 0)
    for (int b = 0; b < 2; ++b) dab::tc::mbar_init(bar0 + 8 * b, 1);
  __syncthreads();
  if (warp == producers / 32) {
    for (int c = 0; c < stages; ++c) {
      for (const long long t0 = clock64(); clock64() - t0 < 500;) {}  // (well within `limit`)
      dab::tc::bar_sync(1 + (c & 1), producers + 32);
      const bool here = lane < producers / 32 && filled[c & 1][lane] == c;
      const unsigned who = __ballot_sync(0xFFFFFFFFu, here);
      if (lane == 0) out[c] = __popc(who);
    }
  } else {
    bool dead = false;
    for (int c = 0; c < stages; ++c) {
      if (c >= 2) dab::tc::mbar_wait(bar0 + 8 * (c & 1), (uint32_t)(c / 2 - 1) & 1u, dead, failures, limit);
      if (lane == 0) filled[c & 1][warp] = c;
      __syncwarp();
      dab::tc::stage_handover(1 + (c & 1), producers + 32, dead);
    }
  }
}

extern "C" int run_handover_timeout(int producer_warps, int stages, long long limit, unsigned int* d_failures, int* d_out) {
  handover_timeout_kernel<<<1, 32 * producer_warps + 32>>>(stages, limit, d_failures, d_out);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return (int)e;
  return (int)cudaDeviceSynchronize();
}

extern "C" int run_wait_timeout(long long limit, int threads, unsigned int* d_failures, int* d_out) {
  wait_timeout_kernel<<<1, threads>>>(limit, d_failures, d_out);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return (int)e;
  return (int)cudaDeviceSynchronize();
}
