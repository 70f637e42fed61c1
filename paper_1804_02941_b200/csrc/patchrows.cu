// Patches through the bucket-pruned search of rowbucket.cuh, a CTA per patch whose values are gathered straight from the
// image: layers with too few patches for the tile coders to fill the device (batch 1, fully connected layers; a chain
// of three mostly idle kernels before), and the patches that the tile coder marked (a sort of 8 warps each
// before).  Latency bounds the first use, the search of rowbucket.cuh the second.  Measured, before -> this: the
// Sketch-A-Net-shaped network at batch 1 581 -> 334 us, its fully connected layer of 12544 values 209 -> 53 us; the
// marked patches of the AlexNet-shaped network at batch 32 3.0 -> 0.43 ms.
#include "rowbucket.cuh"

namespace dab {
namespace {

struct PatchRowArgs {
  dab_conv_desc d;
  int32_t Ho, Wo, n;
  uint32_t magic_khw, magic_kw;  // ceil(2^32 / d): floor(i / d) = umulhi(i, magic) for i < 2^16; 0 if d == 1
  const float* x;
  RowOut out;
  int32_t run;  // patch slots a CTA of the marked kernel scans at a time
};

struct PatchRow {
  const float* img;  // the image
  int hb, wb;        // first row and column of the window
  const PatchRowArgs& a;
  __device__ __forceinline__ PatchRow(const PatchRowArgs& args, int64_t patch) : a(args) {
    const int wo = (int)(patch % a.Wo), ho = (int)((patch / a.Wo) % a.Ho);
    img = a.x + patch / ((int64_t)a.Wo * a.Ho) * a.d.C * a.d.H * a.d.W;
    hb = ho * a.d.stride_h - a.d.pad_h;
    wb = wo * a.d.stride_w - a.d.pad_w;
  }
  __device__ __forceinline__ float value(int i) const {
    const int c = a.magic_khw ? (int)__umulhi((unsigned)i, a.magic_khw) : i, rs = i - c * a.d.kh * a.d.kw;
    const int r = a.magic_kw ? (int)__umulhi((unsigned)rs, a.magic_kw) : rs, s = rs - r * a.d.kw;
    const int h = hb + r, w = wb + s;
    if ((unsigned)h >= (unsigned)a.d.H || (unsigned)w >= (unsigned)a.d.W) return 0.0f;
    return __ldg(img + DAB_IDX(((int64_t)c * a.d.H + h) * a.d.W + w, (int64_t)a.d.C * a.d.H * a.d.W));
  }
  template <int T>
  __device__ __forceinline__ uint32_t stage(float* vals, int quads, BlockShared<T>*) const {
    uint32_t top = 0u;
#pragma unroll 8
    for (int i = threadIdx.x; i < 4 * quads; i += T) {
      const float v = i < a.n ? value(i) : 0.0f;
      vals[i] = v;
      top = max(top, magnitude_bits(v));
    }
    return top;
  }
  template <int T>
  __device__ __forceinline__ void restage(float* vals, int quads) const { stage<T>(vals, quads, nullptr); }
  template <int T>
  __device__ __forceinline__ void finish(const float*, const RowResult&) const {}
};

template <int T>
__global__ void __launch_bounds__(T, 1024 / T) binarize_patches_bucket_kernel(const PatchRowArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  for (int64_t p = blockIdx.x; p < a.out.rows; p += gridDim.x) {
    block_code_row<T>(PatchRow(a, p), a.n, smem_raw, a.out, p);
    __syncthreads();
  }
}

// The patches with K = kRowMark.
template <int T>
__global__ void __launch_bounds__(T, 1024 / T) binarize_patches_marked_kernel(const PatchRowArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint16_t queue[256];
  __shared__ int queued;
  for (int64_t chunk = (int64_t)blockIdx.x * a.run; chunk < a.out.rows; chunk += (int64_t)gridDim.x * a.run) {
    if (threadIdx.x == 0) queued = 0;
    __syncthreads();
#pragma unroll 4
    for (int s = threadIdx.x; s < a.run; s += T)
      if (chunk + s < a.out.rows && a.out.K[DAB_IDX(chunk + s, a.out.rows)] == kRowMark) queue[atomicAdd(&queued, 1)] = (uint16_t)s;
    __syncthreads();
    const int count = queued;
    for (int q = 0; q < count; ++q) {
      block_code_row<T>(PatchRow(a, chunk + queue[q]), a.n, smem_raw, a.out, chunk + queue[q]);
      __syncthreads();
    }
    __syncthreads();
  }
}

template <int T>
cudaError_t launch(PatchRowArgs& a, bool marked_only, cudaStream_t stream) {
  const size_t smem = block_row_bytes<T>(a.n);
  cudaError_t e;
  if (!marked_only) {
    if ((e = ensure_dynamic_smem(binarize_patches_bucket_kernel<T>, smem)) != cudaSuccess) return e;
    binarize_patches_bucket_kernel<T><<<(unsigned)(a.out.rows < (1 << 20) ? a.out.rows : (1 << 20)), T, smem, stream>>>(a);
    return cudaGetLastError();
  }
  if ((e = ensure_dynamic_smem(binarize_patches_marked_kernel<T>, smem)) != cudaSuccess) return e;
  // short runs spread the marked patches of a small layer over all SMs
  const int64_t resident = (int64_t)sm_count() * (1024 / T);
  a.run = 256;
  while (a.run > 8 && (a.out.rows + a.run - 1) / a.run < resident) a.run >>= 1;
  const int64_t blocks = (a.out.rows + a.run - 1) / a.run;
  binarize_patches_marked_kernel<T><<<(unsigned)(blocks < resident ? blocks : resident), T, smem, stream>>>(a);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_binarize_patches_bucket(const dab_conv_desc& d, int32_t Ho, int32_t Wo, const float* x, int32_t* pK,
                                           float* pgamma, float* pdelta, uint32_t* pmask, int32_t ldp, uint32_t* pflags,
                                           bool marked_only, cudaStream_t stream) {
  PatchRowArgs a;
  a.d = d; a.Ho = Ho; a.Wo = Wo; a.n = d.C * d.kh * d.kw;
  const int64_t khw = (int64_t)d.kh * d.kw;
  a.magic_khw = khw > 1 ? (uint32_t)((0x100000000ll + khw - 1) / khw) : 0u;
  a.magic_kw = d.kw > 1 ? (uint32_t)((0x100000000ll + d.kw - 1) / d.kw) : 0u;
  a.x = x;
  a.out = RowOut{pK, pgamma, pdelta, pflags, pmask, ldp, (int64_t)d.N * Ho * Wo};
  a.run = 0;
  if (a.n <= BucketShape<64>::kMaxN) return launch<64>(a, marked_only, stream);
  if (a.n <= BucketShape<128>::kMaxN) return launch<128>(a, marked_only, stream);
  return launch<256>(a, marked_only, stream);
}

}  // namespace dab
