// Weights-only binarized convolution (Section 4.3.2, Corollary 1: the forward pass I (*) W~ with
// W~ = alpha e + beta (1 - e) and full-precision activations), on the tensor cores.
//
//   y[p][co] = alpha_co * M1 + beta_co * (S - M1),   M1 = sum_{i: e_co[i] = 1} x_p[i],   S = sum_i x_p[i]
//
// M1 is a dense contraction of the patch matrix with the 0/1 filter masks (stored as 0 / -1 bytes).  It is formed exactly in integers:
// every patch row is written as 32-bit fixed point relative to its own largest magnitude
// (q_i = rint(x_i * 2^sexp), |q_i| < 2^31), q is split into its four bytes (three unsigned, the top one
// signed), and four tcgen05.mma kind::i8 products with the masks expanded to 0 / -1 bytes give four negated 32-bit
// accumulators per output in tensor memory; M1 = a3 2^24 + a2 2^16 + a1 2^8 + a0 (times 2^-sexp).  The only
// error is the rounding of x_i to q_i: at most 2^-32 of the row's largest magnitude per element.
//
// A CTA owns up to 128 output positions (the lanes of tensor memory) and 64 or 128 filters (4 accumulators each: 512 columns).
// Positions are consecutive in a strip of at most 32 output columns that runs through all images, so that a tile is full
// whatever the image size.  Patches are never formed in global memory: for each group of JS mask words (32 JS patch elements)
// the CTA stages the channels they come from in shared memory, and every thread gathers 16 elements of its row at a time,
// converts them and stores one 16-byte K chunk per byte plane in the operand layout of tc.cuh.  Both the staged channels and
// the operands are double-buffered: while the tensor cores work on one stage the threads convert the next.  (Where two CTAs share an
// SM, or a wide window leaves no room, the operands are not: see launch_wbin_conv.)
//
// Bound by shared memory: per stage of 128 elements and 128 filters the tensor cores read 128 KB of operands, the gather
// 64 KB of values (twice where lanes of a warp lie in different output rows) and writes 64 KB.  An element takes some 20
// instructions in all, the 8 or so of its conversion among them; a CTA of 128 filters halves that over one of 64.
#include <algorithm>
#include <climits>

#include "common.cuh"
#include "tc.cuh"

namespace dab {
namespace {

using namespace tc;

__device__ unsigned int g_wbin_wait_timeouts;

struct WbinArgs {
  dab_conv_desc d;
  int32_t Ho, Wo, n, words, khw;
  int32_t R, TW, strips;       // positions per tile; columns per strip; strips
  int32_t in_w, pitch;         // staged columns; words per staged row
  int32_t ch_words, max_ch;    // words per staged channel, channels per stage (both at most)
  int32_t row_slots;           // 64 or 128: rows that the threads are spread over
  uint32_t magic_khw, magic_kw;  // ceil(2^32 / d): floor(i / d) = umulhi(i, magic); 0 if d == 1
  const float* x;
  const uint32_t* pixmax;  // N x H x W: largest magnitude over the channels, as a bit pattern
  const uint32_t* wmask;
  int32_t ldw;
  const float* walpha;
  const float* wbeta;
  float* y;
};

// a / b, both positive; a 64-bit division (some 100 instructions) only where it takes one.
__device__ __forceinline__ int64_t quotient(int64_t a, int b) {
  return a >> 32 ? a / b : (int64_t)((uint32_t)a / (uint32_t)b);
}

__device__ __forceinline__ int fast_div(int i, uint32_t magic) {
  return magic ? (int)__umulhi((unsigned)i, magic) : i;
}

// Byte planes of four fixed-point values: out[p] holds byte p of q0..q3 (q0 in the lowest byte).
__device__ __forceinline__ void byte_planes(uint32_t q0, uint32_t q1, uint32_t q2, uint32_t q3, uint32_t (&out)[4]) {
  const uint32_t a = __byte_perm(q0, q1, 0x5140), b = __byte_perm(q0, q1, 0x7362);
  const uint32_t c = __byte_perm(q2, q3, 0x5140), d = __byte_perm(q2, q3, 0x7362);
  out[0] = __byte_perm(a, c, 0x5410);
  out[1] = __byte_perm(a, c, 0x7632);
  out[2] = __byte_perm(b, d, 0x5410);
  out[3] = __byte_perm(b, d, 0x7632);
}

// Place of a stage's element in its operand row: the order of expand_word_signed within a mask word.
__device__ __forceinline__ int element_of_place(int i) { return (i & ~15) + ((i & 15) >> 2) + 4 * (i & 3); }

// Sixteen elements (K chunk kc of the stage) of one row: gathered through the offset table, scaled
// by 2^sexp in two exact steps, rounded to 32-bit integers, split into byte planes and stored as one 16-byte K
// chunk per plane; the byte sums of the planes accumulate in psum.  kChecked: elements from `limit` on are 0.
// kTwoStep: the scale is beyond one fp32 factor (patches whose largest magnitude is below 2^-70).
template <uint32_t kPlane, bool kChecked, bool kTwoStep>
__device__ __forceinline__ void gather_chunk(const unsigned char* src, const int32_t* off, int kc, int limit, float fac,
                                             float fac2, unsigned char* dst0, int (&psum)[4]) {
  uint32_t pl[4][4];
#pragma unroll
  for (int g4 = 0; g4 < 4; ++g4) {
    const int4 o4 = *reinterpret_cast<const int4*>(off + kc * 16 + g4 * 4);
    const int o[4] = {o4.x, o4.y, o4.z, o4.w};
    uint32_t q[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      float v = *reinterpret_cast<const float*>(src + o[e]);
      if (kChecked && kc * 16 + element_of_place(g4 * 4 + e) >= limit) v = 0.0f;
      v = __fmul_rn(v, fac);
      if (kTwoStep) v = __fmul_rn(v, fac2);
      q[e] = (uint32_t)__float2int_rn(v);
    }
    uint32_t w4[4];
    byte_planes(q[0], q[1], q[2], q[3], w4);
#pragma unroll
    for (int p = 0; p < 4; ++p) pl[p][g4] = w4[p];
    psum[0] = (int)__dp4a(w4[0], 0x01010101u, (unsigned)psum[0]);
    psum[1] = (int)__dp4a(w4[1], 0x01010101u, (unsigned)psum[1]);
    psum[2] = (int)__dp4a(w4[2], 0x01010101u, (unsigned)psum[2]);
    psum[3] = __dp4a((int)w4[3], 0x01010101, psum[3]);
  }
  unsigned char* dst = dst0 + (uint32_t)kc * 128;
#pragma unroll
  for (int p = 0; p < 4; ++p)
    *reinterpret_cast<uint4*>(dst + p * kPlane) = make_uint4(pl[p][0], pl[p][1], pl[p][2], pl[p][3]);
}

// Bytes of shared memory for the operands.
constexpr size_t operand_bytes(int nt, int js, int buffers) { return (size_t)buffers * (4 * kLanes + nt) * js * 32; }

// The rows of input under a tile are staged one after another, those of an image together.  Row of output row `g` (counted
// over all images) in the staging area, and what a staged row holds.
struct TileRows {
  int64_t img0;
  int ho0, first, full, stride, Ho;  // rows staged for the first image (at most) and for a whole one
  __device__ __forceinline__ TileRows(const WbinArgs& a, int64_t g0) : stride(a.d.stride_h), Ho(a.Ho) {
    img0 = quotient(g0, a.Ho);
    ho0 = (int)(g0 - img0 * a.Ho);
    first = (a.Ho - 1 - ho0) * stride + a.d.kh;
    full = (a.Ho - 1) * stride + a.d.kh;
  }
  __device__ __forceinline__ int staged(int dg, int& di, int& ho) const {  // dg: output rows behind the tile's first one
    di = (ho0 + dg) / Ho;
    ho = ho0 + dg - di * Ho;
    return di == 0 ? (ho - ho0) * stride : first + (di - 1) * full + ho * stride;
  }
  __device__ __forceinline__ void source(int q, int& di, int& h) const {  // (h before the padding is taken off)
    if (q < first) { di = 0; h = ho0 * stride + q; return; }
    di = 1 + (q - first) / full;
    h = (q - first) % full;
  }
};

// THREADS 512: a CTA has the SM to itself; 256 (of 64 filters): two CTAs share it.  BUFFERS: operand stages, 1 or 2.
template <int NT, int JS, int THREADS, int BUFFERS>
__global__ void __launch_bounds__(THREADS, 512 / THREADS) wbin_conv_kernel(const WbinArgs a) {
  constexpr int KS = JS * 32, KC = JS * 2;        // patch elements and 16-byte K chunks per stage
  constexpr uint32_t SBO = KC * 128;              // bytes between groups of 8 rows
  constexpr uint32_t PLANE = kLanes * KS;         // bytes of one byte plane of the activations
  constexpr uint32_t STAGE = 4 * PLANE + NT * KS;
  constexpr int SHARE = NT / (THREADS / 128);     // filters per group of four warps in the epilogue
  static_assert(NT * JS <= THREADS, "a mask word per thread and stage");
  extern __shared__ __align__(128) unsigned char dyn_mem[];
  __shared__ __align__(8) uint64_t s_bar[2];
  __shared__ uint32_t s_tmem;
  __shared__ int s_rowsexp[kLanes];               // scale exponent of a row; INT_MIN: not in the image; INT_MAX: non-finite
  __shared__ double s_alpha[NT], s_beta[NT];
  __shared__ __align__(16) int32_t s_off[2][KS];  // byte offsets of a stage's elements in the staged channels

  const int tid = threadIdx.x, warp = (int)uniform(tid >> 5), lane = tid & 31;
  const uint32_t mem0 = (smem_u32(dyn_mem) + 127u) & ~127u;
  unsigned char* const operands = dyn_mem + (mem0 - smem_u32(dyn_mem));
  const int tile_words = a.max_ch * a.ch_words;
  float* const tiles = reinterpret_cast<float*>(operands + BUFFERS * STAGE);
  int32_t* const goff = reinterpret_cast<int32_t*>(tiles + 2 * (size_t)tile_words);  // [pixel] place in x; -1: outside
  uint32_t* const pixmax = reinterpret_cast<uint32_t*>(tiles);                        // [pixel]; until channels are staged
  int4* const rowsum = reinterpret_cast<int4*>(operands);  // [thread] byte-plane sums of q over its part of the row; at the end
  const uint32_t bar0 = smem_u32(&s_bar[0]), bar1 = smem_u32(&s_bar[1]);

  // tile of this CTA: positions f0 .. f0 + R - 1 of its strip
  const int strip = blockIdx.x % a.strips, wo0 = strip * a.TW;
  const int64_t f0 = (int64_t)(blockIdx.x / a.strips) * a.R, total = (int64_t)a.d.N * a.Ho * a.TW;
  const int rows = (int)min((int64_t)a.R, total - f0);
  const int64_t g0 = quotient(f0, a.TW);
  const int lead = (int)(f0 - g0 * a.TW);  // positions of the first output row before the tile
  const TileRows map(a, g0);
  const int w0 = wo0 * a.d.stride_w - a.d.pad_w;
  const int j0 = blockIdx.y * NT;
  const int plane_in = a.d.H * a.d.W;
  const int64_t img_stride = (int64_t)a.d.C * plane_in;
  const float* const x0 = a.x + map.img0 * img_stride;
  int pixels;  // staged words per channel
  {
    int di, ho;
    pixels = (map.staged((lead + rows - 1) / a.TW, di, ho) + a.d.kh) * a.pitch;
  }

  if (warp == 0) tmem_alloc(smem_u32(&s_tmem), 4 * NT);
  if (tid == 0) {
    mbar_init(bar0, 1);
    mbar_init(bar1, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int j = tid; j < NT; j += THREADS) {
    const bool in = j0 + j < a.d.Cout;
    s_alpha[j] = in ? (double)a.walpha[j0 + j] : 0.0;
    s_beta[j] = in ? (double)a.wbeta[j0 + j] : 0.0;
  }
  // where the staged words come from, and the per-pixel maxima (0 outside the image)
  for (int i = tid; i < pixels; i += THREADS) {
    const int q = i / a.pitch, s = i - q * a.pitch, w = w0 + s;
    int di, h;
    map.source(q, di, h);
    h -= a.d.pad_h;
    const bool in = s < a.in_w && (unsigned)h < (unsigned)a.d.H && (unsigned)w < (unsigned)a.d.W && map.img0 + di < a.d.N;
    goff[i] = in ? di * (int)img_stride + h * a.d.W + w : -1;
    pixmax[i] = in ? __ldg(a.pixmax + (map.img0 + di) * plane_in + (int64_t)h * a.d.W + w) : 0u;
  }
  __syncthreads();

  // Row = output position; its scale comes from the largest magnitude of its patch.
  const int slots = a.row_slots, groups = THREADS / slots;
  auto locate = [&](int r, int64_t& img, int& ho, int& lw) {  // returns the first staged word of the row's window
    const int dg = (lead + r) / a.TW;
    lw = lead + r - dg * a.TW;
    int di;
    const int q = map.staged(dg, di, ho);
    img = map.img0 + di;
    return q * a.pitch + lw * a.d.stride_w;
  };
  const int row = tid & (slots - 1), group = tid / slots;
  int origin = 0;
  {
    int64_t img;
    int ho, lw = 0;
    if (row < rows) origin = locate(row, img, ho, lw);
    if (tid < kLanes) {
      int sexp = INT_MIN;
      if (tid < rows && wo0 + lw < a.Wo) {  // (rows <= slots: row = tid here)
        uint32_t m = 0u;
        for (int i = 0; i < a.d.kh; ++i)
          for (int j = 0; j < a.d.kw; ++j) m = max(m, pixmax[origin + i * a.pitch + j]);
        if (m >= 0x7F800000u) sexp = INT_MAX;
        else if (m == 0u) sexp = 0;
        else sexp = 30 - ((int)(m >> 23) - 127);  // -97 .. 157 (the largest for a subnormal maximum)
      }
      s_rowsexp[tid] = sexp;
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = uniform(s_tmem);
  const int my_sexp = s_rowsexp[row];
  const bool gather = my_sexp != INT_MIN && my_sexp != INT_MAX;
  // x * 2^sexp in two exact steps: 2^sexp itself is beyond fp32 for the smallest patches
  const int sexp1 = gather ? min(my_sexp, 100) : 0, sexp2 = gather ? my_sexp - sexp1 : 0;
  const float fac = __int_as_float((sexp1 + 127) << 23), fac2 = __int_as_float((sexp2 + 127) << 23);

  const int stages = (a.words + JS - 1) / JS;
  // Asynchronous copy of the channels that stage `st` draws from into tile buffer st & 1, and the offsets of its
  // elements inside that tile.  A thread keeps to one pixel where there are few.
  const int copies = max(1, THREADS / pixels);
  const int pix0 = copies > 1 ? tid % pixels : tid, c_first = copies > 1 ? tid / pixels : 0;
  auto stage_in = [&](int st) {
    const int k0 = st * KS, k1 = min(a.n, k0 + KS);
    const int c_lo = fast_div(k0, a.magic_khw), nch = fast_div(k1 - 1, a.magic_khw) + 1 - c_lo;
    float* const tile = tiles + (st & 1) * tile_words;
    if (c_first < copies)
      for (int i = pix0; i < pixels; i += copies > 1 ? pixels : THREADS) {
        const int at = goff[i];
        const float* src = at >= 0 ? x0 + at + (int64_t)(c_lo + c_first) * plane_in : x0;
        const int64_t step = at >= 0 ? (int64_t)copies * plane_in : 0;
        uint32_t dst = smem_u32(tile + c_first * a.ch_words + i);
        for (int c = c_first; c < nch; c += copies) {
          asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(at >= 0 ? 4 : 0)
                       : "memory");  // source size 0: the word is filled with zeros
          src += step;
          dst += (uint32_t)(copies * a.ch_words) * 4;
        }
      }
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (tid < KS) {
      const int k = k0 + element_of_place(tid);
      int o = 0;  // beyond the patch length: any word of the patch (the gather replaces it by 0)
      if (k < a.n) {
        const int c = fast_div(k, a.magic_khw), rs = k - c * a.khw;
        const int r = fast_div(rs, a.magic_kw), s = rs - r * a.d.kw;
        o = (c - c_lo) * a.ch_words + r * a.pitch + s;
      }
      s_off[st & 1][tid] = 4 * o;
    }
  };
  // mask word of this thread: filter tid % NT, word tid / NT of the stage
  const int mrow = tid & (NT - 1), mword = tid / NT;
  const uint32_t* const masks = a.wmask + (int64_t)min(j0 + mrow, a.d.Cout - 1) * a.ldw;
  auto load_mask = [&](int st) {
    const int w = st * JS + mword;
    return mword < JS && w < a.words ? __ldg(masks + w) : 0u;
  };
  const uint32_t idesc_u = instr_desc(NT, false, true), idesc_s = instr_desc(NT, true, true);
  auto multiply = [&](int st) {  // (one thread) the products of stage `st`
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint64_t da = smem_desc(mem0 + st % BUFFERS * STAGE, 128, SBO), db = desc_at(da, 4 * PLANE);
    const int kw = min(JS, a.words - st * JS);
#pragma unroll
    for (int t = 0; t < JS; ++t)
      if (t < kw)
#pragma unroll
        for (int p = 0; p < 4; ++p)
          mma_i8(tmem + (uint32_t)(p * NT), desc_at(da, p * PLANE + t * 256), desc_at(db, t * 256), p == 3 ? idesc_s : idesc_u,
                 (st | t) != 0);
    mma_commit(st % BUFFERS ? bar1 : bar0);
  };

  int psum[4] = {0, 0, 0, 0};
  bool dead = false;
  uint32_t next_mask = load_mask(0);
  stage_in(0);
  for (int st = 0; st < stages; ++st) {
    const int k0 = st * KS;
    const uint32_t mask = next_mask;
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic-proxy stores of the last stage -> tensor-core reads
    __syncthreads();  // this stage's channels have arrived, the last stage's operands are complete
    if (st > 0 && warp == 0 && elect_one()) multiply(st - 1);
    if (st + 1 < stages) {
      stage_in(st + 1);
      next_mask = load_mask(st + 1);
    }
    // the tensor cores have finished reading what these buffers held before
    if (st >= BUFFERS) mbar_wait(st % BUFFERS ? bar1 : bar0, (uint32_t)(st / BUFFERS - 1) & 1u, dead, &g_wbin_wait_timeouts);
    unsigned char* const stage_a = operands + st % BUFFERS * STAGE;
    if (gather) {
      const unsigned char* const src = reinterpret_cast<const unsigned char*>(tiles + (st & 1) * tile_words + origin);
      const int32_t* const off = s_off[st & 1];
      unsigned char* const dst0 = stage_a + (uint32_t)(row >> 3) * SBO + (row & 7) * 16;
      if (k0 + KS <= a.n && sexp2 == 0) {
        for (int kc = group; kc < KC; kc += groups) gather_chunk<PLANE, false, false>(src, off, kc, 0, fac, fac2, dst0, psum);
      } else {  // a row length that is not a multiple of the stage (elements beyond it count as 0) or a two-step scale
        for (int kc = group; kc < KC && k0 + kc * 16 < a.n; kc += groups)
          gather_chunk<PLANE, true, true>(src, off, kc, a.n - k0, fac, fac2, dst0, psum);
      }
    }
    if (mword < JS)
      expand_word_signed(mask, stage_a + 4 * PLANE + (uint32_t)(mrow >> 3) * SBO + (mrow & 7) * 16 + mword * 256);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();
  if (warp == 0 && elect_one()) multiply(stages - 1);
  // the last commit covers every instruction before it
  mbar_wait_last((stages - 1) % BUFFERS ? bar1 : bar0, (uint32_t)((stages - 1) / BUFFERS) & 1u, dead, &g_wbin_wait_timeouts);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  rowsum[tid] = make_int4(psum[0], psum[1], psum[2], psum[3]);  // (a wait that ran out stores nothing to y)
  __syncthreads();

  // Epilogue: thread = row (a warp reads the 32 lanes of its quarter), an equal share of the filters per four warps.
  // The filter bytes are 0 / -1: the accumulators hold the negative sums.
  {
    const int erow = (warp & 3) * 32 + lane;
    const int sexp = s_rowsexp[erow];
    const bool valid = sexp != INT_MIN && !dead;
    const bool bad = sexp == INT_MAX;
    double Sd = 0.0, inv = 0.0;
    int64_t obase = 0;
    if (valid) {
      int64_t img;
      int ho, lw;
      locate(erow, img, ho, lw);
      obase = img * a.d.Cout * a.Ho * a.Wo + (int64_t)ho * a.Wo + wo0 + lw;
    }
    if (valid && !bad) {
      long long s4[4] = {0, 0, 0, 0};
      for (int g = 0; g < groups; ++g) {
        const int4 part = rowsum[g * slots + erow];
        s4[0] += part.x;
        s4[1] += part.y;
        s4[2] += part.z;
        s4[3] += part.w;
      }
      Sd = (double)((s4[3] << 24) + (s4[2] << 16) + (s4[1] << 8) + s4[0]);
      inv = __hiloint2double((1023 - sexp) << 20, 0);
    }
    const int64_t plane_hw = (int64_t)a.Ho * a.Wo;
    static_assert(DAB_MAX_N <= (1 << 14), "255 * 257 * n must stay below 2^31");
#pragma unroll 1
    for (int c8 = 0; c8 < SHARE / 8; ++c8) {
      const int col = (warp >> 2) * SHARE + c8 * 8;
      uint32_t v[4][8];
      const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)col;
#pragma unroll
      for (int p = 0; p < 4; ++p) tmem_load_8(taddr + (uint32_t)(p * NT), v[p]);
      tmem_load_wait();
      if (!valid) continue;
#pragma unroll
      for (int jj = 0; jj < 8; ++jj) {
        const int j = col + jj;
        if (j0 + j >= a.d.Cout) break;
        float out;
        if (bad) {
          out = __uint_as_float(0x7FC00000u);
        } else {
          const double hi = int_to_double(-((int)v[3][jj] * 256 + (int)v[2][jj]));
          const double lo = int_to_double(-((int)v[1][jj] * 256 + (int)v[0][jj]));
          const double m1 = __fma_rn(hi, 65536.0, lo), m0 = Sd - m1;  // exact: |.| < 2^45
          const double y = __dadd_rn(__dmul_rn(s_alpha[j], m1), __dmul_rn(s_beta[j], m0));
          out = (float)__dmul_rn(y, inv);
        }
        a.y[obase + (int64_t)(j0 + j) * plane_hw] = out;
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, 4 * NT);
}

// Largest magnitude over the channels of every pixel, as a bit pattern (NaN > Inf > finite): what the
// convolution kernel derives the scale of a patch from.  SHARES warps take a share of the channels of 32 pixels each: bound by
// the one read of x (with a thread per pixel too few loads are in flight where there are many channels: 35 us for 51 MB; with
// eight shares of three channels most warps have nothing to do).
constexpr int PM_WARPS = 8;
template <int SHARES>
__global__ void __launch_bounds__(32 * PM_WARPS) wbin_pixmax_kernel(const float* __restrict__ x, uint32_t* __restrict__ out,
                                                                    int C, int HW, int64_t total) {
  __shared__ uint32_t part[PM_WARPS][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, share = warp % SHARES;
  const int64_t idx = ((int64_t)blockIdx.x * (PM_WARPS / SHARES) + warp / SHARES) * 32 + lane;
  uint32_t m = 0u;
  if (idx < total) {
    const int64_t img = quotient(idx, HW), p = idx - img * HW;
    const float* src = x + img * C * (int64_t)HW + p;
#pragma unroll 8
    for (int c = share; c < C; c += SHARES) m = max(m, __float_as_uint(__ldg(src + (int64_t)c * HW)) & 0x7FFFFFFFu);
  }
  if (SHARES > 1) {
    part[warp][lane] = m;
    __syncthreads();
#pragma unroll
    for (int w = 1; w < SHARES; ++w)
      if (share == 0) m = max(m, part[warp + w][lane]);
  }
  if (share == 0 && idx < total) out[idx] = m;
}

template <int SHARES>
cudaError_t launch_pixmax(const float* x, uint32_t* out, int C, int HW, int64_t total, cudaStream_t stream) {
  const int64_t blocks = (total + 32 * PM_WARPS / SHARES - 1) / (32 * PM_WARPS / SHARES);
  if (blocks > 0x7FFFFFFF) return cudaErrorInvalidValue;
  wbin_pixmax_kernel<SHARES><<<(unsigned)blocks, 32 * PM_WARPS, 0, stream>>>(x, out, C, HW, total);
  return cudaGetLastError();
}

uint32_t magic_for(uint32_t d) { return d > 1 ? (uint32_t)((0x100000000ull + d - 1) / d) : 0u; }

constexpr size_t kSmemLimit = 227 * 1024 - 5 * 1024;  // (static shared memory aside)
constexpr size_t kSmemLimitOfTwo = 113 * 1024 - 3 * 1024;

// Sets the tile: strips of at most `tw` columns, R positions.  Returns the shared memory it takes with operands of the given size.
size_t set_tile(WbinArgs* a, int tw, int R, int nt, int js, int buffers) {
  const dab_conv_desc& d = a->d;
  a->strips = (a->Wo + tw - 1) / tw;
  a->TW = (a->Wo + a->strips - 1) / a->strips;
  const int64_t total = (int64_t)d.N * a->Ho * a->TW;
  a->R = (int)std::min<int64_t>(R, total);
  a->in_w = (a->TW - 1) * d.stride_w + d.kw;
  a->pitch = a->in_w | 1;
  // output rows a tile touches, the images they lie in, and the rows of input under them (all at most)
  const int64_t all_rows = (int64_t)d.N * a->Ho;
  const int64_t rows = std::min<int64_t>(a->R % a->TW == 0 ? a->R / a->TW : (a->R + 2 * a->TW - 2) / a->TW, all_rows);
  const int64_t images = std::min<int64_t>(1 + (rows - 1 + a->Ho - 1) / a->Ho, d.N);
  const int64_t staged = rows * d.stride_h + (d.kh > d.stride_h ? images : 1) * (d.kh - d.stride_h);  // (rows between windows are not)
  a->max_ch = std::min(d.C, (js * 32 + a->khw - 2) / a->khw + 1);
  if (staged * a->pitch > 1 << 20 || images * d.C * d.H * d.W > 0x7FFFFFFF) return SIZE_MAX;  // (32-bit places)
  a->ch_words = (int)(staged * a->pitch);
  return 128 + operand_bytes(nt, js, buffers) + sizeof(float) * (2 * (size_t)a->max_ch + 1) * a->ch_words;
}

template <int NT, int JS, int THREADS, int BUFFERS>
cudaError_t launch_tiles(const WbinArgs& a, size_t smem, cudaStream_t stream) {
  const int64_t gx = ((int64_t)a.d.N * a.Ho * a.TW + a.R - 1) / a.R * a.strips, gy = (a.d.Cout + NT - 1) / NT;
  if (gx > 0x7FFFFFFF || gy > 65535) return cudaErrorInvalidValue;
  cudaError_t e = ensure_dynamic_smem(wbin_conv_kernel<NT, JS, THREADS, BUFFERS>, smem);
  if (e != cudaSuccess) return e;
  wbin_conv_kernel<NT, JS, THREADS, BUFFERS><<<dim3((unsigned)gx, (unsigned)gy), THREADS, smem, stream>>>(a);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_wbin_conv(const dab_conv_desc& d, int32_t Ho, int32_t Wo, const float* x, const uint32_t* wmask,
                             int32_t ldw, const float* walpha, const float* wbeta, float* y, uint32_t* pixmax,
                             cudaStream_t stream) {
  WbinArgs a;
  a.pixmax = pixmax;
  a.d = d; a.Ho = Ho; a.Wo = Wo;
  a.khw = d.kh * d.kw;
  a.n = d.C * a.khw;
  a.words = (a.n + 31) / 32;
  a.x = x; a.wmask = wmask; a.ldw = ldw; a.walpha = walpha; a.wbeta = wbeta; a.y = y;
  a.magic_khw = magic_for((uint32_t)a.khw);
  a.magic_kw = magic_for((uint32_t)d.kw);
  // 128 filters per CTA share one conversion; 64 where there are no more, or where 128 leave SMs idle.  With 64 rows a tile
  // converts in half the time: for layers that do not fill the device with them either.
  const int64_t positions = (int64_t)d.N * Ho * Wo, sms = sm_count();
  int nt = d.Cout > 64 && (positions + 127) / 128 * ((d.Cout + 127) / 128) >= sms ? 128 : 64;
  const int rows = (positions + 63) / 64 * ((d.Cout + nt - 1) / nt) <= sms ? 64 : kLanes;
  // The tile: the fewest strips, then the most rows that fit.  Tiles of 64 filters beyond the first wave go to CTAs of half the
  // threads with one operand stage where 128 rows fit, two on an SM: short rows are mostly set-up, and one CTA's covers the other's.
  // Measured, 512 threads and two stages -> this: 64 x 3 x 224 x 224 (27 elements, 64 filters) 1356 -> 806 us, 64 x 32 x 112 x 112
  // (288, 32) 574 -> 392, 64 x 64 x 56 x 56 (576, 64) 198 -> 160, 64 x 64 x 28 x 28 7 x 7 (3136, 64) 170 -> 152; within the first
  // wave 196 positions of 2304 elements, 64 filters 39 -> 51.  Rows of up to 96 elements, which are
  // one stage, go there with more than 64 filters too: 3 x 2 x 141 x 141 1 x 1 (2, 177) 62 -> 45.
  // All others: two stages of 128 elements, else of 64; for 64 filters and windows that reach over two channels at most whatever the
  // stage, one of 128 instead: 16 x 2 x 80 x 80 31 x 31 104 -> 79 us, 64 x 1 x 120 x 120 64 x 64 1142 -> 770.
  struct { int nt, js, buffers, threads; } form = {0, 0, 0, 0};
  size_t smem = 0;
  auto fits = [&](int tw, int R, int js, int buffers, int threads) {
    smem = set_tile(&a, tw, R, nt, js, buffers);
    if (smem <= (threads == 512 ? kSmemLimit : kSmemLimitOfTwo)) form = {nt, js, buffers, threads};
    return form.nt != 0;
  };
  const int filters = nt;
  if ((nt == 64 || a.n <= 96) && (positions + 127) / 128 * ((d.Cout + 63) / 64) > sms) {
    nt = 64;
    for (int tw = 32; tw >= 8 && !form.nt; tw >>= 1) fits(tw, kLanes, 4, 1, 256);
    if (!form.nt) nt = filters;
  }
  for (;; nt = 64) {
    for (int tw = 32; tw >= 1 && !form.nt; tw >>= 1)
      for (int R = rows; R >= (tw > 1 ? rows / 2 : 1) && !form.nt; R -= R > 16 ? 16 : 1)
        fits(tw, R, 4, 2, 512) || (nt == 64 && a.khw >= 128 ? fits(tw, R, 4, 1, 512) : fits(tw, R, 2, 2, 512));
    if (form.nt || nt == 64) break;
  }
  if (!form.nt) return cudaErrorInvalidValue;
  a.row_slots = a.R <= 64 ? 64 : kLanes;
  // A thread per pixel where those fill the device or there is little to share.  Eight shares against it: 64 x 3 x 224 x 224 890 and
  // 806 us for the whole call, 64 x 64 x 56 x 56 167 and 160, 64 x 128 x 28 x 28 82 and 82, 64 x 256 x 14 x 14 54 and 57.
  const int HW = d.H * d.W;  // (C * H * W is below 2^31)
  const int64_t pixels = (int64_t)d.N * HW;
  cudaError_t e = d.C <= 4 || pixels > 1 << 16 ? launch_pixmax<1>(x, pixmax, d.C, HW, pixels, stream)
                                                : launch_pixmax<8>(x, pixmax, d.C, HW, pixels, stream);
  if (e != cudaSuccess) return e;
  if (form.threads == 256) return launch_tiles<64, 4, 256, 1>(a, smem, stream);
  if (form.nt == 128) return form.js == 4 ? launch_tiles<128, 4, 512, 2>(a, smem, stream) : launch_tiles<128, 2, 512, 2>(a, smem, stream);
  if (form.js == 2) return launch_tiles<64, 2, 512, 2>(a, smem, stream);
  return form.buffers == 2 ? launch_tiles<64, 4, 512, 2>(a, smem, stream) : launch_tiles<64, 4, 512, 1>(a, smem, stream);
}

cudaError_t read_wbin_wait_timeouts(unsigned int* count) {
  return cudaMemcpyFromSymbol(count, g_wbin_wait_timeouts, sizeof(unsigned int));
}

}  // namespace dab
