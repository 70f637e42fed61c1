// Whole-network inference (Section 5.1: Sketch-A-Net, ResNet-18 and GoogLeNet with all but the first (and last)
// layer binarized): the full-precision layers around the binarized ones as small kernels of their own, and
// dab_network_forward, which queues every layer of a chain on one stream without synchronising.
//
// Elementwise layers (per-channel affine, ReLU, shortcuts and the copies that remember them) run in the kernel of the layer before
// them, on its outputs; what has no such layer before it runs as one pass.  Pooling is its plain definition, one thread per
// output.  The dense convolution sums its products in fp64 in element order (c, kh, kw), each product and sum
// rounded on its own, and rounds once to fp32, so that its result does not depend on the launch shape.
#include "contraction.cuh"

namespace dab {

namespace {

constexpr int kGlueThreads = 256;

inline unsigned glue_blocks(int64_t count) {
  int64_t b = (count + kGlueThreads - 1) / kGlueThreads;
  const int64_t cap = (int64_t)sm_count() * 32;
  return (unsigned)(b < 1 ? 1 : (b > cap ? cap : b));
}

// Full-precision convolution as an implicit matrix product on the fp64 pipe.  A CTA owns 32*PX output positions (of
// all images, flattened) and 8*CO filters: a warp takes CO filters, a lane PX positions, so that a value of x serves CO
// products and a weight (the same address for the whole warp) 32*PX.  Chunks of TAPS taps of both operands are
// staged in shared memory, the next chunk travels in registers meanwhile; weights are staged as fp64 (converted once
// per CTA), positions as fp32 (a conversion per PX products of a lane).
// The order of the sum is (c, kh, kw), as ever.  The product of two fp32 values has 48 significant bits and is exact in
// fp64, so the fused multiply-add rounds exactly where a multiplication and an addition would.
// Bound by the fp64 pipe (64 per clock and SM), of which it keeps about half busy.  Measured at batch 32, one thread per
// output without reuse -> this: 7x7 stem, 3 -> 64 filters on 224^2 (3.8 G products, 0.20 ms at the pipe's rate)
// 4.2 -> 0.44 ms; 11x11 stride 4, 3 -> 96 (3.4 G) 2.5 -> 0.45 ms; 4096 -> 250 fully connected 0.80 -> 0.13 ms.
struct __align__(16) DenseTap {
  int64_t offset;   // in the image, from the window's origin
  int row, column;  // in the window
};

template <int PX, int CO, int TAPS>
__global__ void __launch_bounds__(256, 2) conv_dense_kernel(dab_conv_desc d, int Ho, int Wo, int co_tiles, const float* __restrict__ x,
                                                         const float* __restrict__ w, const float* __restrict__ bias,
                                                         float* __restrict__ y, const PostOps post) {
  constexpr int PT = 32 * PX, CT = 8 * CO;                 // positions and filters of a CTA
  constexpr int XL = TAPS * PT / 256;                // staged values per thread and chunk: positions ...
  constexpr int WL = (TAPS * CT + 255) / 256;        // ... and weights
  __shared__ float s_x[2][TAPS][PT + (PX == 1)];          // (+ 1: see below)
  __shared__ __align__(16) double s_w[2][TAPS][CT + 2];  // + 2: fewer bank conflicts between taps
  __shared__ DenseTap s_tap[2][TAPS];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int khw = d.kh * d.kw, n = d.C * khw;
  const int64_t HoWo = (int64_t)Ho * Wo, positions = (int64_t)d.N * HoWo;
  const int64_t p0 = (int64_t)(blockIdx.x / (unsigned)co_tiles) * PT;
  const int co0 = (int)(blockIdx.x % (unsigned)co_tiles) * CT;

  // The position this thread stages, and the first of the taps it stages there.  Behind 1 x 1 outputs (fully connected
  // layers) every position is another image and its taps are contiguous: there neighbouring threads stage neighbouring
  // taps of one position (32 images read 32 cache lines per load otherwise: 166 us for 4096 -> 250 at batch 32).
  const bool along_taps = PX == 1 && HoWo == 1;
  const int sp = along_taps ? tid / TAPS : tid % PT, st0 = along_taps ? tid % TAPS : tid / PT;
  constexpr int ST = 256 / PT;                             // taps staged side by side
  const int64_t gp = p0 + sp;
  const bool live = gp < positions;
  const int img = live ? (int)(gp / HoWo) : 0;
  const int rem = live ? (int)(gp % HoWo) : 0;
  const int hb = rem / Wo * d.stride_h - d.pad_h, wb = rem % Wo * d.stride_w - d.pad_w;
  const float* const xpos = x + (int64_t)img * d.C * d.H * d.W + (int64_t)hb * d.W + wb;  // may lie before the image: taps outside it are not read

  auto tap_table = [&](int b, int k0) {
    if (tid >= TAPS) return;
    const int k = k0 + tid, c = k / khw, rs = k - c * khw, r = rs / d.kw, q = rs - r * d.kw;
    s_tap[b][tid] = DenseTap{((int64_t)c * d.H + r) * d.W + q, k < n ? r : 0x3FFFFFFF, q};  // (a row no image has)
  };
  float xr[XL], wr[WL];
  auto fetch = [&](int b, int k0) {
    if (along_taps) {
      const DenseTap t = s_tap[b][st0];
      const bool in = (unsigned)(t.row - d.pad_h) < (unsigned)d.H && (unsigned)(t.column - d.pad_w) < (unsigned)d.W;
#pragma unroll
      for (int j = 0; j < XL; ++j) {
        const int64_t p = p0 + sp + j * (256 / TAPS);
        xr[j] = in && p < positions ? __ldg(x + p * d.C * d.H * d.W - (int64_t)d.pad_h * d.W - d.pad_w + t.offset) : 0.0f;
      }
    } else
#pragma unroll
    for (int j = 0; j < XL; ++j) {
      const DenseTap t = s_tap[b][st0 + j * ST];
      const bool in = live && (unsigned)(hb + t.row) < (unsigned)d.H && (unsigned)(wb + t.column) < (unsigned)d.W;
      xr[j] = in ? __ldg(xpos + t.offset) : 0.0f;
    }
#pragma unroll
    for (int j = 0; j < WL; ++j) {
      const int e = tid + j * 256, k = k0 + e % TAPS, co = co0 + e / TAPS;
      wr[j] = (e < TAPS * CT && k < n && co < d.Cout) ? __ldg(w + (int64_t)co * n + k) : 0.0f;
    }
  };
  auto stage = [&](int b) {
#pragma unroll
    for (int j = 0; j < XL; ++j) {
      if (along_taps) s_x[b][st0][sp + j * (256 / TAPS)] = xr[j];
      else s_x[b][st0 + j * ST][sp] = xr[j];
    }
#pragma unroll
    for (int j = 0; j < WL; ++j) {
      const int e = tid + j * 256;
      if (e < TAPS * CT) s_w[b][e % TAPS][e / TAPS] = (double)wr[j];
    }
  };

  double acc[PX][CO];
#pragma unroll
  for (int i = 0; i < PX; ++i)
#pragma unroll
    for (int j = 0; j < CO; ++j) acc[i][j] = 0.0;

  auto taps = [&](int b, int count) {
#pragma unroll(PX == 1 ? 8 : 2)
    for (int k = 0; k < count; ++k) {
      double xv[PX], wv[CO];
#pragma unroll
      for (int i = 0; i < PX; ++i) xv[i] = (double)s_x[b][k][i * 32 + lane];
#pragma unroll
      for (int j = 0; j < CO; ++j) wv[j] = s_w[b][k][warp * CO + j];
#pragma unroll
      for (int i = 0; i < PX; ++i)
#pragma unroll
        for (int j = 0; j < CO; ++j) acc[i][j] = __fma_rn(xv[i], wv[j], acc[i][j]);
    }
  };

  tap_table(0, 0);
  tap_table(1, TAPS);
  __syncthreads();
  fetch(0, 0);
  stage(0);
  __syncthreads();
  int b = 0;
  for (int k0 = 0; k0 < n; k0 += TAPS, b ^= 1) {
    if (k0 + TAPS < n) {
      tap_table(b, k0 + 2 * TAPS);  // (its readers were done before the last barrier)
      fetch(b ^ 1, k0 + TAPS);
      taps(b, TAPS);
      stage(b ^ 1);
      __syncthreads();
    } else {
      taps(b, n - k0);
    }
  }

#pragma unroll
  for (int i = 0; i < PX; ++i) {
    const int64_t p = p0 + i * 32 + lane;
    if (p >= positions) continue;
    const int64_t at = (p / HoWo) * d.Cout * HoWo + p % HoWo;
    const int first = co0 + warp * CO;
    float out[CO];
#pragma unroll
    for (int j = 0; j < CO; ++j) {
      double v = acc[i][j];
      if (bias && first + j < d.Cout) v = __dadd_rn(v, (double)__ldg(bias + first + j));
      out[j] = (float)v;
    }
    for (int k = 0; k < post.count; ++k) {
      const PostOp o = post.op[k];
#pragma unroll
      for (int j = 0; j < CO; ++j)
        if (first + j < d.Cout) out[j] = apply_post_op(o, out[j], first + j, at + (first + j) * HoWo);
    }
#pragma unroll
    for (int j = 0; j < CO; ++j)
      if (first + j < d.Cout) y[at + (first + j) * HoWo] = out[j];
  }
}

// A thread per output, for one or two filters of few taps: there is nothing to share.
__global__ void __launch_bounds__(kGlueThreads) conv_dense_direct_kernel(dab_conv_desc d, int Ho, int Wo, const float* __restrict__ x,
                                                                         const float* __restrict__ w, const float* __restrict__ bias,
                                                                         float* __restrict__ y, const PostOps post) {
  const int64_t outputs = (int64_t)d.N * d.Cout * Ho * Wo;
  const int n = d.C * d.kh * d.kw;
  for (int64_t oi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; oi < outputs; oi += (int64_t)gridDim.x * blockDim.x) {
    const int wo = (int)(oi % Wo);
    const int64_t line = oi / Wo, plane = line / Ho;
    const int ho = (int)(line % Ho), co = (int)(plane % d.Cout);
    const float* const wrow = w + (int64_t)co * n;
    const float* const ximg = x + plane / d.Cout * d.C * d.H * d.W;
    const int hb = ho * d.stride_h - d.pad_h, wb = wo * d.stride_w - d.pad_w;
    double acc = 0.0;
    int k = 0;
    for (int c = 0; c < d.C; ++c)
      for (int r = 0; r < d.kh; ++r)
        for (int s = 0; s < d.kw; ++s, ++k) {
          const int h = hb + r, q = wb + s;
          const float v = (unsigned)h < (unsigned)d.H && (unsigned)q < (unsigned)d.W ? __ldg(ximg + ((int64_t)c * d.H + h) * d.W + q) : 0.0f;
          acc = __fma_rn((double)v, (double)__ldg(wrow + k), acc);
        }
    if (bias) acc = __dadd_rn(acc, (double)__ldg(bias + co));
    const float v = (float)acc;
    y[oi] = post.count > 0 ? apply_post(post, v, co, oi) : v;
  }
}

// 128 positions x 64 filters (or 48, where that wastes fewer) where that gives the device work for every SM; otherwise
// (batch 1, fully connected layers, where a chain of n dependent additions is what counts) 32 positions x 16 filters in
// chunks of 64 taps, one memory latency each.  Layers of few filters take tiles of 8 or 16 of them.  Measured, 48 filters, this, and a
// thread per output: 8 x 3 x 224 x 224 3 x 3, 8 filters 90, 46 and 107 us, 4 filters 89, 46 and 56, one filter 87, 46 and 18; 64 channels
// 1 x 1 on 16 x 56 x 56, one filter 27, 14 and 26.
cudaError_t launch_conv_dense(const dab_conv_desc& d, int Ho, int Wo, const float* x, const float* w, const float* bias, float* y,
                              const PostOps& post, cudaStream_t stream) {
  const int64_t positions = (int64_t)d.N * Ho * Wo;
  auto run = [&](auto kernel, int pt, int ct) {
    const int co_tiles = (d.Cout + ct - 1) / ct;
    const int64_t blocks = (positions + pt - 1) / pt * co_tiles;
    if (blocks > 0x7FFFFFFF) return cudaErrorInvalidValue;
    kernel<<<(unsigned)blocks, 256, 0, stream>>>(d, Ho, Wo, co_tiles, x, w, bias, y, post);
    return cudaGetLastError();
  };
  const bool large = ((positions + 127) / 128) * ((d.Cout + 63) / 64) >= sm_count();
  const bool by48 = (d.Cout + 47) / 48 * 48 < (d.Cout + 63) / 64 * 64;
  if (!large) return run(conv_dense_kernel<1, 2, 64>, 32, 16);
  if (d.Cout <= 2 && d.C * d.kh * d.kw <= 32) {
    conv_dense_direct_kernel<<<glue_blocks(positions * d.Cout), kGlueThreads, 0, stream>>>(d, Ho, Wo, x, w, bias, y, post);
    return cudaGetLastError();
  }
  if (d.Cout <= 16) return d.Cout <= 8 ? run(conv_dense_kernel<4, 1, 16>, 128, 8) : run(conv_dense_kernel<4, 2, 16>, 128, 16);
  return by48 ? run(conv_dense_kernel<4, 6, 16>, 128, 48) : run(conv_dense_kernel<4, 8, 16>, 128, 64);
}

// Elementwise layers with no layer before them that could take them along: one pass, four elements a thread (VEC) where the
// planes and pointers allow.  magic: ceil(2^32 / units of a plane), 0 where a 32-bit quotient would not be exact.
template <int VEC>
__global__ void __launch_bounds__(kGlueThreads) glue_kernel(const float* __restrict__ x, int64_t units, int C, int64_t plane_units,
                                                            uint32_t magic, const PostOps post, float* __restrict__ y) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < units; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t plane = magic ? (int64_t)__umulhi((unsigned)i, magic) : i / plane_units;
    const int channel = magic ? (int)((unsigned)plane % (unsigned)C) : (int)(plane % C);
    float v[VEC];
    if (VEC == 4) {
      const float4 f = *reinterpret_cast<const float4*>(x + 4 * i);
      v[0] = f.x; v[VEC > 1 ? 1 : 0] = f.y; v[VEC > 2 ? 2 : 0] = f.z; v[VEC > 3 ? 3 : 0] = f.w;
    } else {
      v[0] = x[i];
    }
    for (int k = 0; k < post.count; ++k) {
      const PostOp o = post.op[k];
      if (VEC == 4 && o.kind == kPostStore) {
        *reinterpret_cast<float4*>(o.to + 4 * i) = make_float4(v[0], v[VEC > 1 ? 1 : 0], v[VEC > 2 ? 2 : 0], v[VEC > 3 ? 3 : 0]);
      } else if (VEC == 4 && o.kind == kPostAdd) {
        const float4 f = *reinterpret_cast<const float4*>(o.a + 4 * i);
        const float w[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
        for (int j = 0; j < VEC; ++j) v[j] = __fadd_rn(v[j], w[j]);
      } else {
#pragma unroll
        for (int j = 0; j < VEC; ++j) v[j] = apply_post_op(o, v[j], channel, VEC * i + j);
      }
    }
    if (VEC == 4) *reinterpret_cast<float4*>(y + 4 * i) = make_float4(v[0], v[VEC > 1 ? 1 : 0], v[VEC > 2 ? 2 : 0], v[VEC > 3 ? 3 : 0]);
    else y[i] = v[0];
  }
}

cudaError_t launch_glue(const float* x, int32_t N, int32_t C, int64_t plane, const PostOps& post, float* y, cudaStream_t stream) {
  uintptr_t bits = reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(y);
  for (int k = 0; k < post.count; ++k)
    bits |= post.op[k].kind == kPostAdd ? reinterpret_cast<uintptr_t>(post.op[k].a) : reinterpret_cast<uintptr_t>(post.op[k].to);
  const int vec = plane % 4 == 0 && (bits & 15) == 0 ? 4 : 1;
  const int64_t per_plane = plane / vec, units = (int64_t)N * C * per_plane;
  // floor(i / d) = umulhi(i, ceil(2^32 / d)) for i * d < 2^32
  const uint32_t magic = per_plane > 1 && units * per_plane < 0x100000000ll ? (uint32_t)((0x100000000ull + per_plane - 1) / per_plane) : 0u;
  if (vec == 4) glue_kernel<4><<<glue_blocks(units), kGlueThreads, 0, stream>>>(x, units, C, per_plane, magic, post, y);
  else glue_kernel<1><<<glue_blocks(units), kGlueThreads, 0, stream>>>(x, units, C, per_plane, magic, post, y);
  return cudaGetLastError();
}

// i / d: by multiply-high where the magic number is exact for the whole range (0: it is not).
__host__ inline uint32_t magic_for(int64_t count, int64_t d) { return d > 1 && count * d < 0x100000000ll ? (uint32_t)((0x100000000ull + d - 1) / d) : 0u; }
__device__ __forceinline__ int64_t divide(int64_t i, int d, uint32_t magic) { return magic ? (int64_t)__umulhi((unsigned)i, magic) : i / d; }

// K x K windows unrolled, all loads of an output in flight together (K = 0: any window, four loads at a time).  The first value of the window
// counts as it is and a later one if it is larger, in this order.
// 32 x 64 x 112 x 112, 3 x 3 stride 2, is 130 MB, 20 us at the memory's rate: 51 us (with 64-bit divisions and a
// load at a time 104); 32 x 96 x 55 x 55 18 (37).  Windows of K = 0, the values beyond the last four one at a time: 32 x 64 x 56 x 56 5 x 5
// stride 2 pad 2 40.4 (42.0; with loads of all fours, masked, 44.0), 4 x 32 x 64 x 64 9 x 9 pad 4 32.3 (33.8; 36.3).
template <int K>
__global__ void __launch_bounds__(kGlueThreads) maxpool_kernel(dab_conv_desc d, int Ho, int Wo, uint32_t magic_wo, uint32_t magic_ho, uint32_t magic_c,
                                                               const float* __restrict__ x, const PostOps post, float* __restrict__ y) {
  const int64_t outputs = (int64_t)d.N * d.C * Ho * Wo;
  const int kh = K ? K : d.kh, kw = K ? K : d.kw;
  for (int64_t oi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; oi < outputs; oi += (int64_t)gridDim.x * blockDim.x) {
    const int64_t line = divide(oi, Wo, magic_wo), plane = divide(line, Ho, magic_ho);
    const int h0 = (int)(line - plane * Ho) * d.stride_h - d.pad_h, w0 = (int)(oi - line * Wo) * d.stride_w - d.pad_w;
    const float* const xp = x + plane * d.H * d.W + (int64_t)h0 * d.W + w0;
    bool seen = false;
    float best = 0.0f;
    auto inside = [&](int s) { return (unsigned)(w0 + s) < (unsigned)d.W; };
    auto take = [&](float v, bool in) {
      if (in && (!seen || v > best)) best = v;
      seen = seen || in;
    };
    if (K) {
      float v[K ? K * K : 1];
      bool in[K ? K * K : 1];
#pragma unroll
      for (int i = 0; i < K * K; ++i) {
        const int r = i / (K ? K : 1), s = i % (K ? K : 1);
        in[i] = (unsigned)(h0 + r) < (unsigned)d.H && (unsigned)(w0 + s) < (unsigned)d.W;
        v[i] = in[i] ? __ldg(xp + (int64_t)r * d.W + s) : 0.0f;
      }
#pragma unroll
      for (int i = 0; i < K * K; ++i) take(v[i], in[i]);
    } else {
      for (int r = 0; r < kh; ++r) {
        if ((unsigned)(h0 + r) >= (unsigned)d.H) continue;
        const float* const row = xp + (int64_t)r * d.W;
        int s = 0;
        for (; s + 4 <= kw; s += 4) {
          float v[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) v[j] = inside(s + j) ? __ldg(row + s + j) : 0.0f;
#pragma unroll
          for (int j = 0; j < 4; ++j) take(v[j], inside(s + j));
        }
        for (; s < kw; ++s)
          if (inside(s)) take(__ldg(row + s), true);
      }
    }
    if (post.count > 0) best = apply_post(post, best, (int)(plane - divide(plane, d.C, magic_c) * d.C), oi);
    y[oi] = best;
  }
}

cudaError_t launch_maxpool(const dab_conv_desc& d, int Ho, int Wo, const float* x, const PostOps& post, float* y, cudaStream_t stream) {
  const int64_t planes = (int64_t)d.N * d.C, outputs = planes * Ho * Wo;
  const uint32_t magic_wo = Wo > 1 ? magic_for(outputs, Wo) : 0u, magic_ho = magic_for(planes * Ho, Ho), magic_c = magic_for(planes, d.C);
  auto run = [&](auto kernel) {
    kernel<<<glue_blocks(outputs), kGlueThreads, 0, stream>>>(d, Ho, Wo, magic_wo, magic_ho, magic_c, x, post, y);
    return cudaGetLastError();
  };
  if (d.kh == 3 && d.kw == 3) return run(maxpool_kernel<3>);
  if (d.kh == 2 && d.kw == 2) return run(maxpool_kernel<2>);
  return run(maxpool_kernel<0>);
}

inline size_t round_up(size_t v, size_t a) { return (v + a - 1) / a * a; }
constexpr size_t kAlign = 256;

struct Shape {
  int32_t C, H, W;
  int64_t count(int32_t N) const { return (int64_t)N * C * H * W; }
};

// Geometry of layer `L` applied to a tensor of shape `in`; false if it cannot be applied.
bool layer_desc(const dab_layer& L, int32_t N, const Shape& in, dab_conv_desc* d, Shape* out) {
  d->N = N; d->C = in.C; d->H = in.H; d->W = in.W;
  d->Cout = L.kind == DAB_LAYER_MAXPOOL ? in.C : L.Cout;
  d->kh = L.kh; d->kw = L.kw; d->stride_h = L.stride_h; d->stride_w = L.stride_w; d->pad_h = L.pad_h; d->pad_w = L.pad_w;
  // (the row-length limit of the binarized layers does not apply to pooling and full-precision layers)
  if (d->Cout < 1 || d->kh < 1 || d->kw < 1 || d->stride_h < 1 || d->stride_w < 1 || d->pad_h < 0 || d->pad_w < 0) return false;
  const int64_t eh = (int64_t)d->H + 2 * (int64_t)d->pad_h - d->kh, ew = (int64_t)d->W + 2 * (int64_t)d->pad_w - d->kw;
  if (eh < 0 || ew < 0) return false;
  out->C = d->Cout; out->H = (int32_t)(eh / d->stride_h + 1); out->W = (int32_t)(ew / d->stride_w + 1);
  return true;
}

struct Plan {
  int64_t max_count = 0;   // largest tensor of the chain, elements
  size_t conv_scratch = 0; // largest scratch of a binarized layer
  Shape out{0, 0, 0};
};

// Walks the chain on the host: shapes, argument checks, sizes.  Returns DAB_OK or the status to report.
dab_status plan_network(const dab_layer* layers, int32_t count, int32_t N, Shape in, Plan* plan) {
  if (!layers || count < 1 || N < 1 || in.C < 1 || in.H < 1 || in.W < 1) return DAB_ERR_INVALID_ARG;
  Shape cur = in, saved{0, 0, 0};
  plan->max_count = cur.count(N);
  for (int32_t i = 0; i < count; ++i) {
    const dab_layer& L = layers[i];
    Shape& t = L.on_saved ? saved : cur;
    if (L.on_saved && saved.C == 0) return DAB_ERR_INVALID_ARG;  // nothing was saved
    dab_conv_desc d;
    Shape out = t;
    switch (L.kind) {
      case DAB_LAYER_CONV_DENSE:
        if (!L.d_weights || L.Cout < 1 || !layer_desc(L, N, t, &d, &out)) return DAB_ERR_INVALID_ARG;
        break;
      case DAB_LAYER_CONV_BINARY: {
        if (!L.d_wmask || !L.d_wK || !L.d_walpha || !L.d_wbeta || L.Cout < 1 || L.on_saved) return DAB_ERR_INVALID_ARG;
        if ((int64_t)t.C * L.kh * L.kw > DAB_MAX_N) return DAB_ERR_UNSUPPORTED;
        if (!layer_desc(L, N, t, &d, &out)) return DAB_ERR_INVALID_ARG;
        const size_t s = dab_binary_conv_workspace(&d);
        if (s == 0) return DAB_ERR_INVALID_ARG;
        if (s > plan->conv_scratch) plan->conv_scratch = s;
        break;
      }
      case DAB_LAYER_AFFINE:
        if (!L.d_scale || !L.d_shift) return DAB_ERR_INVALID_ARG;
        break;
      case DAB_LAYER_RELU:
        break;
      case DAB_LAYER_MAXPOOL:
        if (!layer_desc(L, N, t, &d, &out)) return DAB_ERR_INVALID_ARG;
        break;
      case DAB_LAYER_SAVE:
        if (L.on_saved) return DAB_ERR_INVALID_ARG;
        saved = cur;
        continue;
      case DAB_LAYER_ADD:
        if (L.on_saved || saved.C != cur.C || saved.H != cur.H || saved.W != cur.W) return DAB_ERR_INVALID_ARG;
        break;
      default:
        return DAB_ERR_INVALID_ARG;
    }
    t = out;
    if (out.count(N) > plan->max_count) plan->max_count = out.count(N);
  }
  plan->out = cur;
  return DAB_OK;
}

}  // namespace
}  // namespace dab

using namespace dab;

extern "C" {

dab_status dab_network_output_shape(const dab_layer* layers, int32_t count, int32_t N, int32_t C, int32_t H, int32_t W,
                                    int32_t* Cout, int32_t* Ho, int32_t* Wo) {
  if (!Cout || !Ho || !Wo) return DAB_ERR_INVALID_ARG;
  Plan plan;
  dab_status s = plan_network(layers, count, N, Shape{C, H, W}, &plan);
  if (s != DAB_OK) return s;
  *Cout = plan.out.C; *Ho = plan.out.H; *Wo = plan.out.W;
  return DAB_OK;
}

size_t dab_network_workspace(const dab_layer* layers, int32_t count, int32_t N, int32_t C, int32_t H, int32_t W) {
  Plan plan;
  if (plan_network(layers, count, N, Shape{C, H, W}, &plan) != DAB_OK) return 0;
  return 4 * round_up((size_t)plan.max_count * sizeof(float), kAlign) + round_up(plan.conv_scratch, kAlign);
}

dab_status dab_network_forward(const dab_layer* layers, int32_t count, int32_t N, int32_t C, int32_t H, int32_t W,
                               const float* d_x, float* d_y, void* d_workspace, size_t workspace_bytes,
                               float* const* h_layer_outputs, void* stream) {
  Plan plan;
  dab_status st = plan_network(layers, count, N, Shape{C, H, W}, &plan);
  if (st != DAB_OK) return st;
  if (!d_x || !d_y) return DAB_ERR_INVALID_ARG;
  const size_t buf = round_up((size_t)plan.max_count * sizeof(float), kAlign);
  if (!d_workspace || (reinterpret_cast<uintptr_t>(d_workspace) % kAlign) || workspace_bytes < 4 * buf + round_up(plan.conv_scratch, kAlign))
    return DAB_ERR_WORKSPACE;
  cudaStream_t cs = static_cast<cudaStream_t>(stream);
  char* ws = static_cast<char*>(d_workspace);
  float* pool[4] = {reinterpret_cast<float*>(ws), reinterpret_cast<float*>(ws + buf), reinterpret_cast<float*>(ws + 2 * buf),
                    reinterpret_cast<float*>(ws + 3 * buf)};
  void* scratch = ws + 4 * buf;
  // buffers 0/1 alternate for the running tensor, 2/3 for the remembered one
  const float* cur = d_x;
  const float* saved = nullptr;
  int cur_next = 0, saved_next = 2;
  Shape cs_shape{C, H, W}, sv_shape{0, 0, 0};
  auto kept = [&](int32_t i) { return h_layer_outputs ? h_layer_outputs[i] : nullptr; };  // the caller wants this layer's output
  auto to_saved = [&]() {
    float* const slot = pool[saved_next];
    saved_next = saved_next == 2 ? 3 : 2;
    return slot;
  };
  for (int32_t i = 0; i < count;) {
    const dab_layer& L = layers[i];
    const bool on_saved = L.on_saved != 0;
    Shape& shp = on_saved ? sv_shape : cs_shape;
    const float* const src = on_saved ? saved : cur;
    const bool own_kernel = L.kind == DAB_LAYER_CONV_DENSE || L.kind == DAB_LAYER_CONV_BINARY || L.kind == DAB_LAYER_MAXPOOL;
    dab_conv_desc d;
    Shape out = shp;
    if (own_kernel) layer_desc(L, N, shp, &d, &out);
    // the elementwise layers that follow on the same tensor (or that begin here), as far as they fit
    PostOps post;
    auto add = [&](int32_t kind, const float* a, const float* b, float* to) { post.op[post.count++] = PostOp{kind, a, b, to}; };
    int32_t last = own_kernel ? i : i - 1;
    while (last + 1 < count && post.count + 3 <= kMaxPostOps) {
      const dab_layer& E = layers[last + 1];
      if ((E.on_saved != 0) != on_saved || E.kind < DAB_LAYER_AFFINE || E.kind == DAB_LAYER_MAXPOOL) break;
      // (a SAVE's kept output is stored with it)
      if (last >= i && layers[last].kind != DAB_LAYER_SAVE && kept(last)) add(kPostStore, nullptr, nullptr, kept(last));
      ++last;
      if (E.kind == DAB_LAYER_AFFINE) add(kPostAffine, E.d_scale, E.d_shift, nullptr);
      else if (E.kind == DAB_LAYER_RELU) add(kPostRelu, nullptr, nullptr, nullptr);
      else if (E.kind == DAB_LAYER_ADD) add(kPostAdd, saved, nullptr, nullptr);
      else {
        // the remembered tensor is a copy (the running buffers are overwritten two layers on)
        float* const slot = to_saved();
        add(kPostStore, nullptr, nullptr, slot);
        saved = slot;
        sv_shape = out;
        if (kept(last)) break;
      }
    }
    const bool ends_saved = layers[last].kind == DAB_LAYER_SAVE;
    if (ends_saved && kept(last)) add(kPostStore, nullptr, nullptr, kept(last));
    cudaError_t e = cudaSuccess;
    bool copies = !own_kernel;  // nothing but a SAVE: the running tensor stays where it is
    for (int32_t k = 0; k < post.count; ++k) copies = copies && post.op[k].kind == kPostStore;
    if (copies) {
      const size_t bytes = (size_t)shp.count(N) * sizeof(float);
      for (int32_t k = 0; k < post.count && e == cudaSuccess; ++k) e = cudaMemcpyAsync(post.op[k].to, src, bytes, cudaMemcpyDeviceToDevice, cs);
      if (e != cudaSuccess) return DAB_ERR_CUDA;
      i = last + 1;
      continue;
    }
    float* dst;
    if (!ends_saved && kept(last)) dst = kept(last);
    else if (on_saved) dst = to_saved();
    else if (last == count - 1) dst = d_y;
    else { dst = pool[cur_next]; cur_next ^= 1; }
    switch (own_kernel ? L.kind : DAB_LAYER_RELU) {
      case DAB_LAYER_CONV_DENSE:
        e = launch_conv_dense(d, out.H, out.W, src, L.d_weights, L.d_bias, dst, post, cs);
        break;
      case DAB_LAYER_CONV_BINARY: {
        const dab_status s = binary_conv(&d, src, L.d_wmask, L.ldw, L.d_wK, L.d_walpha, L.d_wbeta, dst, scratch,
                                         round_up(plan.conv_scratch, kAlign), post, stream);
        if (s != DAB_OK) return s;
        break;
      }
      case DAB_LAYER_MAXPOOL:
        e = launch_maxpool(d, out.H, out.W, src, post, dst, cs);
        break;
      default:
        e = launch_glue(src, N, out.C, (int64_t)out.H * out.W, post, dst, cs);
        break;
    }
    if (e != cudaSuccess) return DAB_ERR_CUDA;
    shp = out;
    if (on_saved) saved = dst;
    else cur = dst;
    i = last + 1;
  }
  if (cur != d_y &&
      cudaMemcpyAsync(d_y, cur, (size_t)cs_shape.count(N) * sizeof(float), cudaMemcpyDeviceToDevice, cs) != cudaSuccess)
    return DAB_ERR_CUDA;
  return DAB_OK;
}

}  // extern "C"
