// Training-side weight binarization (Algorithm 2, steps 4-13) and the gradient factor of Theorem 4, a CTA per filter.
//
// Forward: MeanCenter (the mean of a filter's n weights, summed in fp64, is subtracted) and Clamp to [-1, 1] happen as
// the row coder of rowbucket.cuh stages the row, the dense two-level filter W~ = alpha e + beta (1 - e) of Corollary 1 is
// written while the row is still staged.  Backward: the l1 norms of the two partitions, then the printed expression
// element by element.  A layer has a few hundred filters of a few MB: bound by the latency of one row's chain of passes,
// so a row gets a CTA (the coder 64 to 256 threads by row length, the backward pass 256) and every launch counts.  Short filters, and
// many of them, get a warp each.
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

// Filters of up to 256 weights, a warp each: centred in shared memory, coded by the sorting coder of rowcode.cuh.  Many of them have
// nothing to gain from more threads, and few neither: 512 x 64 7.6 us with two warps per row in the search below -> 5.1, 65536 x 64
// 187 -> 107, 16384 x 128 53 -> 33.
template <int R>
__global__ void __launch_bounds__(kWarpsPerCta * 32) train_forward_short_kernel(const float* W, int32_t n, int64_t ld_W, float* Wc, int64_t ld_Wc,
                                                                               float* Wt, int64_t ld_Wt, const RowOut out) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* const rcp = reinterpret_cast<double*>(smem_raw);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t* const scratch = reinterpret_cast<uint32_t*>(rcp + rcp_table_slots(n)) + warp * (64 * R);
  float* const vals = reinterpret_cast<float*>(scratch + 32 * R);
  fill_reciprocals(rcp, n, threadIdx.x, blockDim.x);
  __syncthreads();
  for (int64_t row = (int64_t)blockIdx.x * kWarpsPerCta + warp; row < out.rows; row += (int64_t)gridDim.x * kWarpsPerCta) {
    const float* const w = W + row * ld_W;
    float v[R];
    double sum = 0.0;
#pragma unroll
    for (int k = 0; k < R; ++k) {
      v[k] = k * 32 + lane < n ? w[DAB_IDX(k * 32 + lane, n)] : 0.0f;
      sum = __dadd_rn(sum, (double)v[k]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum = __dadd_rn(sum, __shfl_xor_sync(0xFFFFFFFFu, sum, o));
    const double mean = __ddiv_rn(sum, (double)n);
    float* const c = Wc + row * ld_Wc;
#pragma unroll
    for (int k = 0; k < R; ++k)
      if (k * 32 + lane < n) {
        v[k] = fminf(fmaxf((float)__dsub_rn((double)v[k], mean), -1.0f), 1.0f);
        c[k * 32 + lane] = vals[k * 32 + lane] = v[k];
      }
    __syncwarp();
    uint32_t kreg[R];
    auto keyof = [vals](int i) { return order_key(vals[i]); };
    const RowResult res = warp_code_row<R, false>(keyof, n, lane, scratch, rcp, kreg);
    if (lane == 0 && DAB_IN_BOUNDS(row, out.rows)) {
      out.K[row] = res.K;
      out.alpha[row] = res.alpha;
      out.beta[row] = res.beta;
      if (out.flags) out.flags[row] = res.flags;
    }
    const uint32_t mine = warp_mask_words<R, false>(kreg, n, lane, res);
    for (int i = lane; i < out.ld; i += 32)
      if (DAB_IN_BOUNDS(row * out.ld + i, out.rows * out.ld)) out.mask[row * out.ld + i] = i < 32 ? mine : 0u;
    if (Wt) {
      float* const t = Wt + row * ld_Wt;
#pragma unroll
      for (int k = 0; k < R; ++k)
        if (k * 32 + lane < n) t[k * 32 + lane] = res.mode != 2 && (kreg[k] >= res.tkey) != (res.mode == 1) ? res.alpha : res.beta;
    }
    __syncwarp();  // the staged values are free again
  }
}

template <int R>
cudaError_t launch_forward_short(const float* W, int32_t n, int64_t ld_W, float* Wc, int64_t ld_Wc, float* Wt, int64_t ld_Wt,
                                 const RowOut& out, cudaStream_t stream) {
  const size_t smem = sizeof(double) * rcp_table_slots(n) + sizeof(uint32_t) * 64 * R * kWarpsPerCta;
  cudaError_t e = ensure_dynamic_smem(train_forward_short_kernel<R>, smem);
  if (e != cudaSuccess) return e;
  const int64_t blocks = (out.rows + kWarpsPerCta - 1) / kWarpsPerCta, most = (int64_t)sm_count() * 16;
  train_forward_short_kernel<R><<<(unsigned)(blocks < most ? blocks : most), kWarpsPerCta * 32, smem, stream>>>(W, n, ld_W, Wc, ld_Wc, Wt, ld_Wt, out);
  return cudaGetLastError();
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
// THREADS of them work on a row, 256 / THREADS rows side by side in a CTA.
constexpr int kBackThreads = 256;

template <int THREADS>
__global__ void __launch_bounds__(kBackThreads) train_backward_kernel(const float* __restrict__ Wc, int64_t ld_Wc,
                                                                      const uint32_t* __restrict__ mask, int32_t ld_mask,
                                                                      const int32_t* __restrict__ K, int64_t rows, int32_t n,
                                                                      const float* __restrict__ gWt, int64_t ld_g,
                                                                      float* __restrict__ gW, int64_t ld_gw) {
  static_assert(THREADS == 32 || THREADS == kBackThreads, "a warp or the CTA per row");
  constexpr int ROWS = kBackThreads / THREADS;
  __shared__ double s_sel[kBackThreads / 32], s_rest[kBackThreads / 32];
  const int tid = threadIdx.x % THREADS, lane = tid & 31;
  auto row_sum = [&](double v, double* part) {
    if (THREADS == kBackThreads) return block_sum<kBackThreads>(v, part);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v = __dadd_rn(v, __shfl_xor_sync(0xFFFFFFFFu, v, off));
    return v;
  };
  for (int64_t row = (int64_t)blockIdx.x * ROWS + threadIdx.x / THREADS; row < rows; row += (int64_t)gridDim.x * ROWS) {
    const float* w = Wc + row * ld_Wc;
    const uint32_t* m = mask + row * (int64_t)ld_mask;
    const int k = K[row];
    double l1_sel = 0.0, l1_rest = 0.0;
#pragma unroll 8
    for (int i = tid; i < n; i += THREADS) {
      const double a = fabs((double)__ldg(w + i));
      const bool sel = (__ldg(m + (i >> 5)) >> lane) & 1u;
      l1_sel = __dadd_rn(l1_sel, sel ? a : 0.0);
      l1_rest = __dadd_rn(l1_rest, sel ? 0.0 : a);
    }
    l1_sel = row_sum(l1_sel, s_sel);
    l1_rest = row_sum(l1_rest, s_rest);
    const bool coded = k > 0 && k < n;
    const double inv_sel = coded ? __ddiv_rn(1.0, (double)k) : 0.0, inv_rest = coded ? __ddiv_rn(1.0, (double)(n - k)) : 0.0;
    const double s_sel1 = coded ? __ddiv_rn(l1_sel, (double)k) : 0.0, s_rest1 = coded ? __ddiv_rn(l1_rest, (double)(n - k)) : 0.0;
    const float* g = gWt + row * ld_g;
    float* out = gW + row * ld_gw;
#pragma unroll 4
    for (int i = tid; i < n; i += THREADS) {
      const double wi = (double)__ldg(w + i);
      const double ste = fabs(wi) <= 1.0 ? wi : 0.0;
      const bool sel = (__ldg(m + (i >> 5)) >> lane) & 1u;
      const double G = __dadd_rn(sel ? inv_sel : inv_rest, __dmul_rn(sel ? s_sel1 : s_rest1, ste));
      out[i] = (float)__dmul_rn((double)__ldg(g + i), coded ? G : 0.0);
    }
    if (THREADS == kBackThreads) __syncthreads();  // the partial sums are free again
  }
}

}  // namespace

cudaError_t launch_train_forward(const float* W, int64_t rows, int32_t n, int64_t ld_W, float* Wc, int64_t ld_Wc,
                                 float* Wt, int64_t ld_Wt, int32_t* K, float* alpha, float* beta, uint32_t* mask,
                                 int32_t ld_mask, uint32_t* flags, cudaStream_t stream) {
  const RowOut out{K, alpha, beta, flags, mask, ld_mask, rows};
  if (n <= 256) return launch_forward_short<8>(W, n, ld_W, Wc, ld_Wc, Wt, ld_Wt, out, stream);
  if (many_short_rows(rows, n)) return launch_forward<32>(W, n, ld_W, Wc, ld_Wc, Wt, ld_Wt, out, stream);
  if (n <= BucketShape<64>::kMaxN) return launch_forward<64>(W, n, ld_W, Wc, ld_Wc, Wt, ld_Wt, out, stream);
  if (n <= BucketShape<128>::kMaxN) return launch_forward<128>(W, n, ld_W, Wc, ld_Wc, Wt, ld_Wt, out, stream);
  return launch_forward<256>(W, n, ld_W, Wc, ld_Wc, Wt, ld_Wt, out, stream);
}

cudaError_t launch_train_backward(const float* Wc, int64_t ld_Wc, const uint32_t* mask, int32_t ld_mask,
                                  const int32_t* K, int64_t rows, int32_t n, const float* gWt, int64_t ld_g, float* gW,
                                  int64_t ld_gw, cudaStream_t stream) {
  // A warp per row: 16384 rows of 128 43 -> 9.6 us, 4096 of 1024 20 -> 12; but 512 of 4608, where a warp's chain is the longer one, 6.4 -> 13.7
  if (rows >= n + n / 8) {
    const int64_t blocks = (rows + 7) / 8;
    train_backward_kernel<32><<<(unsigned)(blocks < (1 << 20) ? blocks : (1 << 20)), kBackThreads, 0, stream>>>(Wc, ld_Wc, mask, ld_mask, K, rows, n, gWt, ld_g, gW, ld_gw);
  } else {
    train_backward_kernel<kBackThreads><<<(unsigned)(rows < (1 << 20) ? rows : (1 << 20)), kBackThreads, 0, stream>>>(Wc, ld_Wc, mask, ld_mask, K, rows, n, gWt, ld_g, gW, ld_gw);
  }
  return cudaGetLastError();
}

}  // namespace dab
