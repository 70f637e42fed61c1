// Sign coding (the paper's XNOR-structured FBin inputs): mask bit = [x >= 0], gamma = mean |x|, delta = -gamma.
//
// Patches: everything that does not depend on the patch is done once per staged pixel of a CTA's tile of output
// positions.  A row of input pixels of one channel becomes one word of sign bits (a ballot, lane = pixel), and a thread sums
// |x| over the channels of its pixel in fp64.  A patch is then a lane: 32 channels fill exactly kh*kw of its mask words,
// each channel and window row adding kw bits taken from the ballot word by a rotation, so that a warp assembles 32
// patches at once; gamma is the sum of kh*kw pixel sums.  The words go through shared memory, where the patches of an
// output row are contiguous, as they are in the output.
// Floor: HBM, one read of x and one write of the codes.  Bound by memory latency and issue (half of the slots).  Measured
// on 256 x 128 x 28 x 28, 3 x 3: 495 us with every patch element gathered by a warp per patch -> 72 us (1.8 TB/s).
#include <cmath>

#include "signrow.cuh"

namespace dab {
namespace {

constexpr int kSignWarps = 8, kSignThreads = kSignWarps * 32;

struct SignArgs {
  dab_conv_desc d;
  int32_t Ho, Wo, n;
  int32_t TH, TW, tiles_h, tiles_w;   // output positions per tile
  int32_t in_h, in_w;                 // staged rows and columns (in_w <= 32)
  int32_t rows_per_ballot, groups;    // whole rows in 32 lanes; ballots per channel
  int32_t c_pitch;                    // words per row of sign bits: channels rounded up to 32, a multiple of 4 but not of 8
  int32_t pitch;                      // words per assembled patch (odd)
  uint32_t magic_ldp;                 // ceil(2^32 / ldp)
  const float* x;
  int32_t* pK;
  float* pgamma;
  float* pdelta;
  uint32_t* pflags;  // may be null
  uint32_t* pmask;
  int32_t ldp;
};

// Bits 0 .. q-1 of `low`, the others of `high`; q is a compile-time constant wherever this is used on a hot path.
__device__ __forceinline__ uint32_t join_bits(uint32_t low, uint32_t high, int q) {
  const uint32_t m = q ? 0xFFFFFFFFu >> (32 - q) : 0u;
  return (low & m) | (high & ~m);
}

// KHW 9: 3 x 3 windows, fully unrolled; 0: any window of up to 32 columns.
template <int KHW>
__global__ void __launch_bounds__(kSignThreads, 4) sign_patches_kernel(const SignArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int C = a.d.C, kh = a.d.kh, kw = a.d.kw, khw = kh * kw, in_h = a.in_h, in_w = a.in_w, groups = a.groups;
  double* const pixel = reinterpret_cast<double*>(smem_raw);                       // [group][32] sum of |x| over the channels
  uint32_t* const bits = reinterpret_cast<uint32_t*>(pixel + groups * 32);         // [in_h][c_pitch] sign bits of a row
  double* const psum = reinterpret_cast<double*>(bits + in_h * a.c_pitch);         // [warp][group][32] partial sums, later
  uint32_t* const words = bits + in_h * a.c_pitch;                                 // [patch][pitch]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

  int t = blockIdx.x;
  const int tw_i = t % a.tiles_w;
  t /= a.tiles_w;
  const int ho0 = (t % a.tiles_h) * a.TH, wo0 = tw_i * a.TW, img = t / a.tiles_h;
  const int h0 = ho0 * a.d.stride_h - a.d.pad_h, w0 = wo0 * a.d.stride_w - a.d.pad_w;
  const int th = min(a.TH, a.Ho - ho0), tw = min(a.TW, a.Wo - wo0), npatch = th * tw;
  const int64_t plane = (int64_t)a.d.H * a.d.W;

  // ---- sign bits of every staged row and channel, partial sums of |x| ----
  const int lr = lane / in_w, lc = lane - lr * in_w;  // this lane's row of a ballot and column (rows_per_ballot and on: idle)
  for (int g = 0; g < groups; ++g) {
    const int r = g * a.rows_per_ballot + lr, h = h0 + r, w = w0 + lc;
    const bool staged = lr < a.rows_per_ballot && r < in_h;
    const bool inside = staged && (unsigned)h < (unsigned)a.d.H && (unsigned)w < (unsigned)a.d.W;
    const float* src = a.x + ((int64_t)img * C + warp) * plane + (inside ? (int64_t)h * a.d.W + w : 0);
    double sum = 0.0;
    uint32_t* const out = bits + r * a.c_pitch;
#pragma unroll 8
    for (int c = warp; c < C; c += kSignWarps, src += kSignWarps * plane) {
      const float v = inside ? __ldg(src) : 0.0f;
      sum = __dadd_rn(sum, fabs((double)v));
      const uint32_t b = __ballot_sync(0xFFFFFFFFu, v >= 0.0f);
      if (staged && lc == 0) out[c] = b >> lane;  // (bits of further rows behind this one's are never looked at)
    }
    psum[(warp * groups + g) * 32 + lane] = sum;
  }
  const int c32 = (C + 31) & ~31;  // the bits of channels that do not exist are 0
  for (int i = threadIdx.x; i < in_h * (c32 - C); i += kSignThreads) bits[(i / (c32 - C)) * a.c_pitch + C + i % (c32 - C)] = 0u;
  __syncthreads();
  for (int i = threadIdx.x; i < groups * 32; i += kSignThreads) {
    double s = psum[i];
#pragma unroll
    for (int w = 1; w < kSignWarps; ++w) s = __dadd_rn(s, psum[w * groups * 32 + i]);
    pixel[i] = s;
  }
  __syncthreads();

  // ---- mask words: a lane per patch, a unit of work per 32 patches and 32 channels ----
  const int pgroups = (npatch + 31) >> 5, cblocks = c32 >> 5;
  for (int u = warp; u < pgroups * cblocks; u += kSignWarps) {
    const int cb = u / pgroups, p = (u - cb * pgroups) * 32 + lane;
    const int pl = p < npatch ? p : 0, lh = pl / tw, lw = pl - lh * tw;
    const int sw = lw * a.d.stride_w;
    const uint32_t* const src = bits + lh * a.d.stride_h * a.c_pitch + cb * 32;
    uint32_t* const dst = words + pl * a.pitch + cb * khw;
    const int room = p < npatch ? a.pitch - cb * khw : 0;  // words of the patch from dst on
    if (KHW == 9) {
      uint32_t acc = 0u;
#pragma unroll
      for (int c4 = 0; c4 < 8; ++c4) {
        uint4 q[3];
#pragma unroll
        for (int r = 0; r < 3; ++r) q[r] = *reinterpret_cast<const uint4*>(src + r * a.c_pitch + c4 * 4);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
#pragma unroll
          for (int r = 0; r < 3; ++r) {
            const uint32_t w = c == 0 ? q[r].x : c == 1 ? q[r].y : c == 2 ? q[r].z : q[r].w;
            constexpr int kRow = 3;
            const int at = (c4 * 4 + c) * 9 + r * kRow, b = at & 31, k = at >> 5;  // first bit of the three, its word
            const uint32_t s = __funnelshift_r(w, w, sw), rot = __funnelshift_l(s, s, b);
            acc = join_bits(acc, rot, b);
            if (b + kRow >= 32) {  // the word is full; the rotated bits that did not fit start the next one
              if (k < room) dst[k] = acc;
              acc = rot;
            }
          }
        }
      }
    } else {
      uint32_t acc = 0u;
      int b = 0, k = 0;
      for (int c = 0; c < 32; ++c) {
        for (int r = 0; r < kh; ++r) {
          const uint32_t w = src[r * a.c_pitch + c], s = __funnelshift_r(w, w, sw), rot = __funnelshift_l(s, s, b);
          acc = join_bits(acc, rot, b);
          b += kw;
          if (b >= 32) {
            if (k < room) dst[k] = acc;
            ++k;
            b -= 32;
            acc = rot;
          }
        }
      }
    }
  }
  __syncthreads();

  // ---- K, gamma, delta: a thread per patch ----
  for (int p = threadIdx.x; p < npatch; p += kSignThreads) {
    const int lh = p / tw, lw = p - lh * tw, r0 = lh * a.d.stride_h, s0 = lw * a.d.stride_w;
    double sum = 0.0;
    for (int r = 0; r < kh; ++r) {
      const int g = (r0 + r) / a.rows_per_ballot, base = g * 32 + ((r0 + r) - g * a.rows_per_ballot) * in_w + s0;
      for (int s = 0; s < kw; ++s) sum = __dadd_rn(sum, pixel[base + s]);
    }
    const bool bad = !(sum <= 1.7976931348623157e308);  // a NaN or an infinity among the values
    uint32_t* const row = words + p * a.pitch;
    const int live = (a.n + 31) >> 5;
    int ones = 0;
    for (int k = 0; k < live; ++k) {
      if (bad) row[k] = 0u;
      ones += __popc(row[k]);
    }
    for (int k = live; k < a.ldp; ++k) row[k] = 0u;
    const int64_t pi = ((int64_t)img * a.Ho + ho0 + lh) * a.Wo + wo0 + lw;
    const float gm = bad ? __uint_as_float(0x7FC00000u) : (float)(sum / (double)a.n);
    a.pK[pi] = ones;
    a.pgamma[pi] = gm;
    a.pdelta[pi] = -gm;
    if (a.pflags) a.pflags[pi] = bad ? DAB_ROW_NONFINITE : 0u;
  }
  __syncthreads();
  // ---- the words of an output row of the tile are contiguous ----
  const int per_row = tw * a.ldp;
  for (int lh = 0; lh < th; ++lh) {
    uint32_t* const out = a.pmask + (((int64_t)img * a.Ho + ho0 + lh) * a.Wo + wo0) * a.ldp;
    const uint32_t* const src = words + lh * tw * a.pitch;
    for (int i = threadIdx.x; i < per_row; i += kSignThreads) {
      const int p = (int)__umulhi((unsigned)i, a.magic_ldp);
      out[i] = src[p * a.pitch + (i - p * a.ldp)];
    }
  }
}

__global__ void __launch_bounds__(256) sign_rows_kernel(const float* __restrict__ values, int64_t rows, int32_t n,
                                                        int64_t ld_values, int32_t* K, float* alpha, float* beta,
                                                        uint32_t* mask, int32_t ld_mask, uint32_t* flags) {
  const int lane = threadIdx.x & 31;
  const int64_t warp0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t row = warp0; row < rows; row += nwarps) {
    const float* v = values + row * ld_values;
    auto value = [v](int i) { return __ldg(v + i); };
    warp_sign_row(value, n, ld_mask, lane, K + row, alpha + row, beta + row, flags ? flags + row : nullptr,
                  mask + row * (int64_t)ld_mask);
  }
}


// Windows of more than 32 columns (no word of 32 pixels holds one): a warp per patch, values straight from the image.
__global__ void __launch_bounds__(kSignThreads) sign_wide_patches_kernel(const SignArgs a) {
  const int lane = threadIdx.x & 31, khw = a.d.kh * a.d.kw;
  const int64_t patches = (int64_t)a.d.N * a.Ho * a.Wo;
  for (int64_t pi = (int64_t)blockIdx.x * kSignWarps + (threadIdx.x >> 5); pi < patches; pi += (int64_t)gridDim.x * kSignWarps) {
    const int wo = (int)(pi % a.Wo), ho = (int)((pi / a.Wo) % a.Ho);
    const float* img = a.x + pi / ((int64_t)a.Wo * a.Ho) * a.d.C * a.d.H * a.d.W;
    const int hb = ho * a.d.stride_h - a.d.pad_h, wb = wo * a.d.stride_w - a.d.pad_w;
    auto value = [&](int i) {
      const int c = i / khw, rs = i - c * khw, r = rs / a.d.kw, h = hb + r, w = wb + rs - r * a.d.kw;
      return (unsigned)h < (unsigned)a.d.H && (unsigned)w < (unsigned)a.d.W ? __ldg(img + ((int64_t)c * a.d.H + h) * a.d.W + w) : 0.0f;
    };
    warp_sign_row(value, a.n, a.ldp, lane, a.pK + pi, a.pgamma + pi, a.pdelta + pi, a.pflags ? a.pflags + pi : nullptr,
                  a.pmask + pi * (int64_t)a.ldp);
  }
}

// Rows of output positions per tile: the number whose estimated cycles over the whole layer are fewest.  A ballot of a
// channel costs a warp about 10 instructions, 32 channels of 32 patches about 38 per window position (the proportions
// matter, not the scale); tiles share the halo of kh - stride rows, and a small layer needs enough of them.
// *us_out: what that tile's estimate comes to, a generic window's rows at 500 instructions each.
bool choose_sign_tile(SignArgs* a, size_t* smem_out, double* us_out) {
  const dab_conv_desc& d = a->d;
  if (d.kw > 32) return false;
  const int widest = (32 - d.kw) / d.stride_w + 1;
  a->tiles_w = (a->Wo + widest - 1) / widest;
  a->TW = (a->Wo + a->tiles_w - 1) / a->tiles_w;
  a->in_w = (a->TW - 1) * d.stride_w + d.kw;
  a->rows_per_ballot = 32 / a->in_w;
  const int c32 = (d.C + 31) & ~31;
  a->c_pitch = c32 + 4;
  a->pitch = a->ldp | 1;
  double best = 0.0;
  for (int th = 1; th <= 16 && th <= a->Ho; ++th) {
    const int in_h = (th - 1) * d.stride_h + d.kh, groups = (in_h + a->rows_per_ballot - 1) / a->rows_per_ballot;
    const size_t partials = sizeof(double) * kSignThreads * groups, words = sizeof(uint32_t) * (size_t)th * a->TW * a->pitch;
    const size_t smem = sizeof(double) * 32 * groups + sizeof(uint32_t) * (size_t)in_h * a->c_pitch + (partials > words ? partials : words);
    if (smem > 227 * 1024) break;
    int ctas = (int)(228 * 1024 / (smem + 1024));
    if (ctas > 4) ctas = 4;
    const int64_t tiles = (int64_t)((a->Ho + th - 1) / th) * a->tiles_w * d.N, slots = (int64_t)sm_count() * ctas;
    const int units = (th * a->TW + 31) / 32 * (c32 / 32);
    const double cost = (double)((tiles + slots - 1) / slots) * sqrt((double)ctas) *  // (the passes are latency-bound: residents add up)
                        (1500.0 + 10.0 * groups * ((d.C + 7) / 8) * 8 + 38.0 * d.kh * d.kw * ((units + 7) / 8) * 8);
    if (best == 0.0 || cost < best) {
      best = cost;
      a->TH = th; a->in_h = in_h; a->groups = groups;
      *smem_out = smem;
      const double unit = d.kh == 3 && d.kw == 3 ? 342.0 : 500.0 * d.kh * (d.stride_h * d.stride_w > 1 ? 2.0 : 1.0);
      *us_out = 3.0 + (double)((tiles + slots - 1) / slots) * sqrt((double)ctas) *
                          (1500.0 + 10.0 * groups * ((d.C + 7) / 8) * 8 + unit * ((units + 7) / 8) * 8) / 3000.0;
    }
  }
  if (best == 0.0) return false;
  a->tiles_h = (a->Ho + a->TH - 1) / a->TH;
  return (int64_t)a->tiles_h * a->tiles_w * d.N <= 0x7FFFFFFF;
}

}  // namespace

cudaError_t launch_sign_rows(const float* values, int64_t rows, int32_t n, int64_t ld_values, int32_t* K, float* alpha,
                             float* beta, uint32_t* mask, int32_t ld_mask, uint32_t* flags, cudaStream_t stream) {
  int64_t blocks = (rows + 7) / 8;
  if (blocks > sm_count() * 16) blocks = sm_count() * 16;
  sign_rows_kernel<<<(unsigned)blocks, 256, 0, stream>>>(values, rows, n, ld_values, K, alpha, beta, mask, ld_mask,
                                                        flags);
  return cudaGetLastError();
}

cudaError_t launch_sign_patches(const dab_conv_desc& d, int32_t Ho, int32_t Wo, const float* x, int32_t* pK,
                                float* pgamma, float* pdelta, uint32_t* pmask, int32_t ldp, uint32_t* pflags,
                                cudaStream_t stream) {
  SignArgs a;
  a.d = d; a.Ho = Ho; a.Wo = Wo; a.n = d.C * d.kh * d.kw;
  a.x = x; a.pK = pK; a.pgamma = pgamma; a.pdelta = pdelta; a.pflags = pflags; a.pmask = pmask; a.ldp = ldp;
  a.magic_ldp = (uint32_t)((0x100000000ull + (uint64_t)ldp - 1) / (uint64_t)ldp);
  size_t smem = 0;
  double us = 0.0;
  const double patches = (double)d.N * Ho * Wo;
  // The other coder: a warp's chain of n / 32 words, and per patch what it reads and stages.  It is ahead for few channels with wide
  // windows, strides and small layers.  Measured, that one and this: 128 x 3 x 64 x 64 11 x 11 stride 4 32 and 132 us, 128 x 2 x 80 x 80 31 x 31
  // stride 5 106 and 823, 1024 channels 1 x 1 on 7 x 7 11 and 24; 128 x 8 x 56 x 56 7 x 7 285 and 125, 128 x 128 x 28 x 28 3 x 3 215 and 33.
  const double staged = 3.0 + 0.0037 * a.n + patches * (0.25 + 0.0015 * a.n + 0.002 * d.C * d.stride_h * d.stride_w) / 1000.0;
  const bool tiled = choose_sign_tile(&a, &smem, &us);
  if (!tiled || staged < us) {
    const cudaError_t e = launch_sign_patches_staged(d, Ho, Wo, x, pK, pgamma, pdelta, pmask, ldp, pflags, stream);
    if (e != cudaErrorInvalidValue) return e;
  }
  if (!tiled) {
    const int64_t blocks = ((int64_t)patches + kSignWarps - 1) / kSignWarps;
    sign_wide_patches_kernel<<<(unsigned)(blocks < sm_count() * 16 ? blocks : sm_count() * 16), kSignThreads, 0, stream>>>(a);
    return cudaGetLastError();
  }
  auto kern = d.kh == 3 && d.kw == 3 ? sign_patches_kernel<9> : sign_patches_kernel<0>;
  cudaError_t e = ensure_dynamic_smem(kern, smem);
  if (e != cudaSuccess) return e;
  kern<<<(unsigned)(a.tiles_h * a.tiles_w * d.N), kSignThreads, smem, stream>>>(a);
  return cudaGetLastError();
}

}  // namespace dab
