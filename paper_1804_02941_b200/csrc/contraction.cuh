// What the two contraction kernels share: the arguments, the rescale and the elementwise layers a network hangs on to a
// convolution's outputs.
#pragma once

#include "common.cuh"

namespace dab {

// Elementwise layers that follow a layer of a network, applied to its outputs as they are stored: a tensor is not written and
// read again for each (a ResNet-18-shaped network at batch 32 spent 0.7 of 4.6 ms on those passes).  The arithmetic is that of the
// layers by themselves, operation for operation.
constexpr int kMaxPostOps = 8;
enum PostKind : int32_t { kPostAffine, kPostRelu, kPostAdd, kPostStore };
struct PostOp {
  int32_t kind;
  const float* a;   // scale per channel; the tensor to add
  const float* b;   // shift per channel
  float* to;        // where the value so far is stored as well (a remembered or inspected tensor)
};
struct PostOps {
  int32_t count = 0;
  PostOp op[kMaxPostOps];
};

// One rounding of the exact scale * v + shift (in fp64 the sum was rounded twice, and the three conversions cost more than the store).
__device__ __forceinline__ float post_affine(const PostOp& o, float v, int channel) {
  return __fmaf_rn(__ldg(o.a + channel), v, __ldg(o.b + channel));
}

// at: the element's place in the tensor (all tensors of the chain have one shape); extent: elements of it.
__device__ __forceinline__ float apply_post_op(const PostOp& o, float v, int channel, int64_t at, int64_t extent = INT64_MAX) {
  if (o.kind == kPostAffine) v = post_affine(o, v, channel);
  else if (o.kind == kPostRelu) v = v > 0.0f ? v : 0.0f;
  else if (o.kind == kPostAdd) v = __fadd_rn(v, o.a[DAB_IDX(at, extent)]);
  else if (DAB_IN_BOUNDS(at, extent)) o.to[at] = v;
  return v;
}
__device__ __forceinline__ float apply_post(const PostOps& ops, float v, int channel, int64_t at, int64_t extent = INT64_MAX) {
#pragma unroll 1
  for (int k = 0; k < ops.count; ++k) v = apply_post_op(ops.op[k], v, channel, at, extent);
  return v;
}

// The sum of the four terms alpha gamma p11 + alpha delta p10 + beta gamma p01 + beta delta p00 of the four counts
// (p10 = Ke - p11, p01 = Kf - p11, p00 = n - Ke - Kf + p11) in fp64, one rounding to fp32, gathered by what depends on the pair:
//   (gamma - delta) ((alpha - beta) p11 + beta Kf) + delta (alpha Ke + beta (n - Ke))
// Five fp64 operations per output instead of the fifteen of the four terms, which kept the fp64 pipe busy longer than the
// counting where rows are short.  A product of a value and a count is exact in fp64 and the fused additions round once.  What is
// rounded on the way stays below 2^-50 of the terms' magnitudes if |alpha| >= |beta| and |gamma| >= |delta|, as in every code that
// the coders write: then no part of the gathered sum is larger than the terms.  Other scales (the contraction entry points take
// any) could cancel in it: alpha = 1, beta = 0, gamma = 1e-12, delta = 3, p11 = Ke = 100 comes out 9e-5 off.  An output of which
// either row is not gathers() is formed by rescale_terms, term by term.  Every kernel that rescales does it in exactly these
// operations.
struct RescaleSide {  // of a weight row: d = alpha - beta, b = beta, c = alpha Ke + beta (n - Ke); of an activation row: d = gamma -
  double d, b, c;     // delta, b = Kf, c = delta
};
__device__ __forceinline__ RescaleSide rescale_weight(double alpha, double beta, int Ke, int n) {
  return {__dsub_rn(alpha, beta), beta, __dadd_rn(__dmul_rn(alpha, int_to_double(Ke)), __dmul_rn(beta, int_to_double(n - Ke)))};
}
__device__ __forceinline__ RescaleSide rescale_activation(double gamma, double delta, int Kf) {
  return {__dsub_rn(gamma, delta), int_to_double(Kf), delta};
}
__device__ __forceinline__ float rescale(int p11, double wd, double wb, double wc, double ad, double ab, double ac) {
  const double t = __fma_rn(wd, int_to_double(p11), __dmul_rn(wb, ab));
  return (float)__fma_rn(ad, t, __dmul_rn(ac, wc));
}
__device__ __forceinline__ float rescale(int p11, const RescaleSide& w, const RescaleSide& a) {
  return rescale(p11, w.d, w.b, w.c, a.d, a.b, a.c);
}
// Values of the set and the clear bits of a row that the gathered form is good for: finite, the first no smaller in magnitude.
__device__ __forceinline__ bool gathers(float set, float clear) { return fabsf(clear) <= fabsf(set) && !is_nonfinite(set); }
// The four terms by themselves, every operation rounded, in the order above.
__device__ __forceinline__ float rescale_terms(int p11, int Ke, int Kf, int n, double alpha, double beta, double gamma, double delta) {
  double y = __dmul_rn(__dmul_rn(alpha, gamma), int_to_double(p11));
  y = __dadd_rn(y, __dmul_rn(__dmul_rn(alpha, delta), int_to_double(Ke - p11)));
  y = __dadd_rn(y, __dmul_rn(__dmul_rn(beta, gamma), int_to_double(Kf - p11)));
  return (float)__dadd_rn(y, __dmul_rn(__dmul_rn(beta, delta), int_to_double(n - Ke - Kf + p11)));
}

// Where an output element (row i of the activation side, column j of the weight side) is stored:
//   offset = (i / inner) * outer_stride + (i % inner) * row_stride + j * col_stride
// Row-major M x N: inner = M (never wraps), row_stride = ldc, col_stride = 1.
// NCHW conv output: inner = Ho*Wo, outer_stride = Cout*Ho*Wo, row_stride = 1, col_stride = Ho*Wo.
struct OutMap {
  int64_t inner, outer_stride, row_stride, col_stride;
};

struct GemmArgs {
  int64_t M, N;
  int32_t n, words;  // words = ceil(n/32) rounded up to a multiple of 4 (<= lda, ldb)
  const uint32_t* A;
  int32_t lda;
  const int32_t* KA;
  const float* gamma;
  const float* delta;
  const uint32_t* B;
  int32_t ldb;
  const int32_t* KB;
  const float* alpha;
  const float* beta;
  float* C;
  OutMap map;
  int64_t c_extent;  // elements from C to the end of the output it addresses (last offset of the map + 1)
  int32_t* p11;
  int64_t ldp;
  PostOps post;      // applied to every output (convolutions only: column j = channel j)
};

// Output of activation row i and weight row j with p11 common bits: gathered if both rows are, else term by term.
__device__ __forceinline__ float rescale_any(const GemmArgs& g, int p11, int64_t i, int64_t j) {
  const float alpha = g.alpha[DAB_IDX(j, g.N)], beta = g.beta[DAB_IDX(j, g.N)], gamma = g.gamma[DAB_IDX(i, g.M)], delta = g.delta[DAB_IDX(i, g.M)];
  const int Ke = g.KB[DAB_IDX(j, g.N)], Kf = g.KA[DAB_IDX(i, g.M)];
  if (gathers(alpha, beta) && gathers(gamma, delta))
    return rescale(p11, rescale_weight((double)alpha, (double)beta, Ke, g.n), rescale_activation((double)gamma, (double)delta, Kf));
  return rescale_terms(p11, Ke, Kf, g.n, (double)alpha, (double)beta, (double)gamma, (double)delta);
}

cudaError_t launch_gemm(const GemmArgs& args, bool lanes_along_rows, cudaStream_t stream);
// Tensor-core contraction; lanes_along_rows as for launch_gemm.  See gemm_mma.cu.
cudaError_t launch_gemm_mma(const GemmArgs& args, bool lanes_along_rows, cudaStream_t stream);

// dab_binary_conv with the layers of `post` behind it.
dab_status binary_conv(const dab_conv_desc* desc, const float* d_x, const uint32_t* d_wmask, int32_t ldw, const int32_t* d_wK,
                       const float* d_walpha, const float* d_wbeta, float* d_y, void* d_workspace, size_t workspace_bytes,
                       const PostOps& post, void* stream);

}  // namespace dab
