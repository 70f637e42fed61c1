// Training-side weight binarization (Algorithm 2, steps 4-13) and the gradient factor of Theorem 4, a CTA per filter.
//
// Forward: MeanCenter (the mean of a filter's n weights, summed in fp64, is subtracted) and Clamp to [-1, 1] happen as
// the row coder of rowbucket.cuh stages the row, the dense two-level filter W~ = alpha e + beta (1 - e) of Corollary 1 is
// written while the row is still staged.  Backward: the l1 norms of the two partitions, then the printed expression
// element by element.  A layer has a few hundred filters of a few MB: bound by the latency of one row's chain of passes,
// so a row gets a CTA (the coder 64 to 256 threads by row length, the backward pass 256) and every launch counts.
// Measured on 512 x 4608: forward 0.145 ms in three launches (sorting coder) -> 0.027 ms in one; backward with a warp per row 0.045
// -> 0.010 ms.
#include "rowbucket.cuh"

namespace dab {
namespace {

template <int T>
__device__ __forceinline__ double block_sum(double v, double* s_part) {  // s_part: T / 32 doubles; the same result in every thread
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v = __dadd_rn(v, __shfl_xor_sync(0xFFFFFFFFu, v, off));
  if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = v;
  __syncthreads();
  double sum = 0.0;
#pragma unroll
  for (int w = 0; w < T / 32; ++w) sum = __dadd_rn(sum, s_part[w]);
  return sum;
}

// A filter on its way through the row coder: staged as Wc = clamp(fp32(w - mean), -1, 1), which is also stored.
struct TrainRow {
  const float* w;
  float* c;
  float* t;  // dense filter, may be null
  int n;
  template <int T>
  __device__ __forceinline__ uint32_t stage(float* vals, int quads, BlockShared<T>* bs) const {
    double sum = 0.0;
#pragma unroll 8
    for (int i = threadIdx.x; i < n; i += T) {
      const float v = w[i];
      vals[i] = v;
      sum = __dadd_rn(sum, (double)v);
    }
    const double mean = __ddiv_rn(block_sum<T>(sum, bs->wsum), (double)n);
    uint32_t top = 0u;
#pragma unroll 4
    for (int i = threadIdx.x; i < 4 * quads; i += T) {
      float v = 0.0f;
      if (i < n) {
        v = fminf(fmaxf((float)__dsub_rn((double)vals[i], mean), -1.0f), 1.0f);
        c[i] = v;
      }
      vals[i] = v;
      top = max(top, magnitude_bits(v));
    }
    return top;
  }
  template <int T>
  __device__ __forceinline__ void restage(float* vals, int quads) const {  // (a thread reads what it wrote)
    for (int i = threadIdx.x; i < 4 * quads; i += T) vals[i] = i < n ? c[i] : 0.0f;
  }
  template <int T>
  __device__ __forceinline__ void finish(const float* vals, const RowResult& res) const {
    if (!t) return;
    const bool flip = res.mode == 1, none = res.mode == 2;
    const float tv = key_value(res.tkey);
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += T) t[i] = !none && ((vals[i] >= tv) != flip) ? res.alpha : res.beta;
  }
};

template <int T>
__global__ void __launch_bounds__(T, 1024 / T) train_forward_kernel(const float* W, int32_t n, int64_t ld_W, float* Wc, int64_t ld_Wc,
                                                                    float* Wt, int64_t ld_Wt, const RowOut out) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  for (int64_t row = blockIdx.x; row < out.rows; row += gridDim.x) {
    const TrainRow r{W + row * ld_W, Wc + row * ld_Wc, Wt ? Wt + row * ld_Wt : nullptr, n};
    block_code_row<T>(r, n, smem_raw, out, row);
    __syncthreads();
  }
}

template <int T>
cudaError_t launch_forward(const float* W, int32_t n, int64_t ld_W, float* Wc, int64_t ld_Wc, float* Wt, int64_t ld_Wt,
                           const RowOut& out, cudaStream_t stream) {
  auto kern = train_forward_kernel<T>;
  const size_t smem = block_row_bytes<T>(n);
  cudaError_t e = ensure_dynamic_smem(kern, smem);
  if (e != cudaSuccess) return e;
  kern<<<(unsigned)(out.rows < (1 << 20) ? out.rows : (1 << 20)), T, smem, stream>>>(W, n, ld_W, Wc, ld_Wc, Wt, ld_Wt, out);
  return cudaGetLastError();
}

// Theorem 4.  G_i = 1/|part| + (l1 norm of the part / |part|) * STE(W_i), the part being the side of the mask element i
// is on; grad_W_i = grad_Wt_i * G_i.
constexpr int kBackThreads = 256;

__global__ void __launch_bounds__(kBackThreads) train_backward_kernel(const float* __restrict__ Wc, int64_t ld_Wc,
                                                                      const uint32_t* __restrict__ mask, int32_t ld_mask,
                                                                      const int32_t* __restrict__ K, int64_t rows, int32_t n,
                                                                      const float* __restrict__ gWt, int64_t ld_g,
                                                                      float* __restrict__ gW, int64_t ld_gw) {
  __shared__ double s_sel[kBackThreads / 32], s_rest[kBackThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31;
  for (int64_t row = blockIdx.x; row < rows; row += gridDim.x) {
    const float* w = Wc + row * ld_Wc;
    const uint32_t* m = mask + row * (int64_t)ld_mask;
    const int k = K[row];
    double l1_sel = 0.0, l1_rest = 0.0;
#pragma unroll 8
    for (int i = tid; i < n; i += kBackThreads) {
      const double a = fabs((double)__ldg(w + i));
      const bool sel = (__ldg(m + (i >> 5)) >> lane) & 1u;
      l1_sel = __dadd_rn(l1_sel, sel ? a : 0.0);
      l1_rest = __dadd_rn(l1_rest, sel ? 0.0 : a);
    }
    l1_sel = block_sum<kBackThreads>(l1_sel, s_sel);
    l1_rest = block_sum<kBackThreads>(l1_rest, s_rest);
    const bool coded = k > 0 && k < n;
    const double inv_sel = coded ? __ddiv_rn(1.0, (double)k) : 0.0, inv_rest = coded ? __ddiv_rn(1.0, (double)(n - k)) : 0.0;
    const double s_sel1 = coded ? __ddiv_rn(l1_sel, (double)k) : 0.0, s_rest1 = coded ? __ddiv_rn(l1_rest, (double)(n - k)) : 0.0;
    const float* g = gWt + row * ld_g;
    float* out = gW + row * ld_gw;
#pragma unroll 4
    for (int i = tid; i < n; i += kBackThreads) {
      const double wi = (double)__ldg(w + i);
      const double ste = fabs(wi) <= 1.0 ? wi : 0.0;
      const bool sel = (__ldg(m + (i >> 5)) >> lane) & 1u;
      const double G = __dadd_rn(sel ? inv_sel : inv_rest, __dmul_rn(sel ? s_sel1 : s_rest1, ste));
      out[i] = (float)__dmul_rn((double)__ldg(g + i), coded ? G : 0.0);
    }
    __syncthreads();  // the partial sums are free again
  }
}

}  // namespace

cudaError_t launch_train_forward(const float* W, int64_t rows, int32_t n, int64_t ld_W, float* Wc, int64_t ld_Wc,
                                 float* Wt, int64_t ld_Wt, int32_t* K, float* alpha, float* beta, uint32_t* mask,
                                 int32_t ld_mask, uint32_t* flags, cudaStream_t stream) {
  const RowOut out{K, alpha, beta, flags, mask, ld_mask, rows};
  if (n <= BucketShape<64>::kMaxN) return launch_forward<64>(W, n, ld_W, Wc, ld_Wc, Wt, ld_Wt, out, stream);
  if (n <= BucketShape<128>::kMaxN) return launch_forward<128>(W, n, ld_W, Wc, ld_Wc, Wt, ld_Wt, out, stream);
  return launch_forward<256>(W, n, ld_W, Wc, ld_Wc, Wt, ld_Wt, out, stream);
}

cudaError_t launch_train_backward(const float* Wc, int64_t ld_Wc, const uint32_t* mask, int32_t ld_mask,
                                  const int32_t* K, int64_t rows, int32_t n, const float* gWt, int64_t ld_g, float* gW,
                                  int64_t ld_gw, cudaStream_t stream) {
  train_backward_kernel<<<(unsigned)(rows < (1 << 20) ? rows : (1 << 20)), kBackThreads, 0, stream>>>(
      Wc, ld_Wc, mask, ld_mask, K, rows, n, gWt, ld_g, gW, ld_gw);
  return cudaGetLastError();
}

}  // namespace dab
