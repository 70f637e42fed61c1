// Patch coder that shares work between overlapping patches (Section 4.1 / Algorithm 1 per patch; Section 4.3.1
// asks for all rows of a layer to be handled as one batch).
//
// A patch is the union of kh*kw pixels (a pixel = the C channel values at one input position) and every pixel
// belongs to up to kh*kw patches, so whatever can be prepared per pixel is prepared once per tile of output positions:
//   grid       value buckets chosen for the tile: one per octave of magnitude and sign, and more where a sample of the tile
//              says that the best splits lie.  Buckets are ranges of bit patterns, so membership is exact;
//   tables     per pixel and bucket the cumulative count and the cumulative fp64 sum (from the count and the sum of the
//              mantissas: 32-bit shared-memory atomics, exact; below the grid's octaves a 64-bit fixed-point sum), and the
//              channels in bucket order.
// A patch is then searched by a warp, a lane per bucket:
//   edges      the tables of its kh*kw pixels are added: split size and prefix sum at every bucket edge, exactly;
//   prune      the objective is jointly convex in (split size, prefix sum); inside a bucket the pair stays within a
//              parallelogram, so its corners bound the objective there (bucket_bound.cuh).  Only the two or so buckets
//              whose bound reaches the best edge value can hold the maximum;
//   search     the values of those buckets (a dozen or two) are gathered from the lists and sorted, a value a lane, which
//              with the exact state below them gives the exact split size and prefix sum behind each.  Objectives closer
//              than their error are compared once more in exactly rounded form, with Algorithm 1's ">=".  Where 128 and more are left,
//              3 x 3 windows of short rows narrow them first (narrow_hull); others sort several a lane.
// The mask is a threshold compare: a thread per patch and 32 channels, values of four channels per load.
// A patch the search does not settle (too many values in its buckets, as with few distinct ones; magnitudes outside
// 2^-40..2^40, a NaN or an infinity in the tile) is marked K = kRowMark and coded by the CTA-per-patch kernel of
// patchrows.cu that follows on the stream.
#include <cmath>

#include "bucket_bound.cuh"
#include "rowcode.cuh"

namespace dab {

namespace {

constexpr int kCellBits = 4, kCells = 1 << kCellBits;          // sampled cells per octave
constexpr int kStepBits = 6, kSteps = 1 << kStepBits;          // grid steps per octave: the finest buckets
constexpr int kStepShift = 23 - kStepBits, kCellShift = 23 - kCellBits;
constexpr int kMaxBuckets = 64, kMaxOctaves = 12;
constexpr int kMaxCells = 2 * (kMaxOctaves * kCells + 1);      // both signs; the inner cell of a side: below the resolved octaves
constexpr int kMaxSteps = 2 * (kMaxOctaves * kSteps + 1);
constexpr int kTileThreads = 512, kTileWarps = kTileThreads / 32;  // two CTAs per SM at 64 registers a thread
constexpr int kSampledUnits = 512; // of four values
// A sampled value counts exp(-kSharp * (1 - D / best D)) + kPrior for the grid.  Measured on post-ReLU, N(0, 1) and network
// activations: from 3 to 30 resp. 0.03 to 0.2 the coder's time moves by less than 10 %, networks by 20 % (local optima of a patch
// differ from the tile's: broad is better there).
constexpr float kSharp = 10.0f, kPrior = 0.2f;
// Sums of at most 2048 values in 62 bits.  Values down to 2^-27 of the lowest resolved octave are exact; what smaller ones lose is
// below the rounding of an fp64 sum with any resolved value in it, and patches without one are left to the other kernel.
constexpr int kTinyBits = 51;
// From this many pixels on a thread sums a pixel's buckets one after another; below it would leave most of them idle (4200 cycles for
// 20 pixels where a warp per pixel takes 1500; at 100 pixels both take 5000, at 130 the warps 7000 to 10000).
constexpr int kSerialPixels = 80;
// Hulls of kNarrowFrom values and more are narrowed before they are sorted, in 3 x 3 windows of short rows (32 buckets).  Code that few
// patches reach is not in the instruction cache and costs some 30 cycles an instruction, which the patch's whole tile waits for, so that a
// narrowing tried in vain is dear.  64 x 56 x 56 at batch 32, us: all sorted; narrowed from 128 on; from 64 on:
//   N(0, 1)|N(0, 1)| 587, 451, 430   steps of 1/8 213, 214, 229   N(0, 1) + 4 291, 293, 324   half zeros 214, 217, 226
// 128 x 28 x 28: 219, 214, 202   101, 108, 140   163, 145, 154   108, 109, 114
// and the ResNet-18-shaped network at batch 32 4270, 3500, 3390.
// In wider windows a lane or two walk the list of a pixel alone: 32 x 48 x 27 x 27 5 x 5 steps of 1/8 107 us sorted, 166 narrowed, N(0, 1)
// 114 and 131, N(0, 1)|N(0, 1)| 247 and 227.  In longer rows a warp has three or four patches of a tile, and one that cannot be narrowed
// holds up the others: 61 x 256 x 14 x 14 N(0, 1) 117 us sorted, 124 narrowed; 32 x 256 x 13 x 13 of a network 95 and 118, though
// 32 x 384 x 13 x 13 156 and 134.
constexpr int kNarrowFrom = 128;
// One of 256 values and more that cannot be narrowed is left to the CTA-per-patch kernel in rows of up to kMarkRows values, else sorted.  A
// single marked patch costs that kernel's latency, many of them less than a sort of 16 values a lane: 64 x 56 x 56 at batch 32, values in
// steps of 1/8 N(0, 1)|N(0, 1)| 368 us marked and 475 sorted, e^(4 N(0, 1)) 667 and 779; 128 x 28 x 28 N(0, 1) 117 and 109, steps of 1/8 117 and 108.
constexpr int kMarkRows = 768;
// A bucket is kept if its bound reaches the best edge objective times this: edges and inner corners are formed in fp32 from
// sums rounded once (1e-6 relative), the place of a corner to 4e-7 of the bucket's count.
constexpr float kKeep = 0.9999f;
constexpr float kWeak = 1e-13f;             // relative difference of objectives that their rounding (4e-16) stays far below
constexpr double kCloseBand = 1.0 - 1e-11;  // objectives this close are compared in their exactly rounded form

struct TileArgs {
  dab_conv_desc d;
  int32_t Ho, Wo, n;
  int32_t TH, TW;            // output positions per tile
  int32_t in_h, in_w;        // rows and columns of input under a tile
  int32_t slots;             // pixel slots in shared memory: the most in-image pixels of a tile, and one of zeros
  int32_t quads, pitch;      // channel quadruples per pixel; words per pixel (an odd multiple of 4)
  int32_t tiles_h, tiles_w;
  int32_t buckets, octaves;  // capacity of the tables; resolved octaves
  int32_t word_pitch;        // words per assembled patch (odd)
  uint32_t tile_at;          // where the values start in shared memory
  uint32_t magic_ldp;        // ceil(2^32 / ldp)
  const float* x;
  int32_t* pK;
  float* pgamma;
  float* pdelta;
  uint32_t* pflags;  // may be null
  uint32_t* pmask;
  int32_t ldp;
};

__device__ __forceinline__ int64_t patch_count(const TileArgs& a) { return (int64_t)a.d.N * a.Ho * a.Wo; }

// The bucket grid of a tile, in shared memory.  Steps and cells ascend in value over both signs.
struct Grid {
  union {
    struct {
      double elo[kMaxBuckets];       // signed start of the bucket's octave and signed unit of the mantissas there:
      double ulp[kMaxBuckets];       // sum of a bucket = count * elo + sum of the mantissas * ulp
      uint32_t hist[kTileWarps * 32];  // sampled values per cell
      uint8_t lut[kMaxSteps + 2];    // bucket of a step
    };
    uint32_t scratch[kTileWarps][64];  // of each warp's search, once the tables are made
  };
  float edge[kMaxBuckets + 1];   // ascending; edge[B0] = 0
  float part[2][kTileWarps];     // per-warp partial sums
  uint32_t ipart[kTileWarps];
  uint32_t best;                 // largest objective of the sample (bits)
  int nb, B0;                    // buckets, first positive one
  uint32_t top;                  // largest magnitude (bits)
  int signs;                     // 1: negative values, 2: positive ones
  int base, side;                // of a step: pattern of the inner one, steps per side
};

// Step of a magnitude, counted from the inner one.
__device__ __forceinline__ int grid_step(uint32_t magnitude, int base, int side) {
  return min(max((int)(magnitude >> kStepShift) - base, 0), side - 1);
}
__device__ __forceinline__ int grid_bucket(const Grid& g, float v, int step, int side) {
  return (int)g.lut[v < 0.0f ? side - 1 - step : side + step];
}

// Sum of a pixel's values in a bucket, channel by channel.
__device__ __noinline__ double sum_by_channel(const Grid& g, const float* values, int C, int bucket) {
  double sum = 0.0;
  for (int c = 0; c < C; ++c) {
    const float v = values[c];
    if (v != 0.0f && grid_bucket(g, v, grid_step(__float_as_uint(v) & 0x7FFFFFFFu, g.base, g.side), g.side) == bucket) sum = __dadd_rn(sum, (double)v);
  }
  return sum;
}

// Inclusive prefix sum over the CTA; `total` in every thread.  part: THREADS / 32 words of shared memory.
template <int THREADS, typename T>
__device__ __forceinline__ T block_prefix(T v, T* part, T& total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const T u = __shfl_up_sync(0xFFFFFFFFu, v, o);
    if (lane >= o) v += u;
  }
  if (lane == 31) part[warp] = v;
  __syncthreads();
  T before = 0;
  total = 0;
#pragma unroll
  for (int w = 0; w < THREADS / 32; ++w) {
    if (w == warp) before = total;
    total += part[w];
  }
  return before + v;
}

// Chooses the buckets from the sampled cells (the whole CTA, two cells a thread).  Every octave of a sign present starts
// a bucket; the other buckets are spread evenly over the sampled values, those discounted whose splits fall short of
// the best sampled objective.
template <int THREADS>
__device__ __forceinline__ void choose_grid(Grid* g, int octaves, int buckets, int sampled) {
  const int tid = threadIdx.x, side = octaves * kCells + 1, steps = octaves * kSteps + 1;
  const int low = (int)(g->top >> 23) - octaves + 1;  // exponent field of the lowest resolved octave
  const int signs = g->signs;
  float k[2], x[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int c = 2 * tid + j, i = c < side ? side - 1 - c : c - side;  // cell, from the inner one
    k[j] = c < 2 * side ? (float)g->hist[c] : 0.0f;
    const float v = __uint_as_float(((uint32_t)((low << kCellBits) - 1 + i) << kCellShift) + (1u << (kCellShift - 1)));
    x[j] = c < side ? -v : v;
  }
  float m, T;
  uint32_t mass_total;
  const float cnt = block_prefix<THREADS>(k[0] + k[1], g->part[0], m);
  const float sum = block_prefix<THREADS>(k[0] * x[0] + k[1] * x[1], g->part[1], T);
  const float n = (float)sampled, z = n - m;
  auto D = [&](float s, float P) {
    const float q = T - P;
    return s > 0.0f && s < n ? __fdividef(P * P, s) + __fdividef(q * q, n - s) : 0.0f;
  };
  float d[3], s = cnt - k[0] - k[1], P = sum - k[0] * x[0] - k[1] * x[1];
  const float dz = fmaxf(D(s, P), D(s + z, P));  // (the zeros lie before cell `side`)
  d[0] = 2 * tid < side ? D(s, P) : (2 * tid == side ? dz : D(s + z, P));
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int c = 2 * tid + j;
    s += k[j];
    P += k[j] * x[j];
    d[j + 1] = c < side - 1 ? D(s, P) : (c == side - 1 ? fmaxf(D(s, P), D(s + z, P)) : D(s + z, P));
  }
  const uint32_t best_bits = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(fmaxf(d[0], fmaxf(d[1], d[2]))));
  if ((tid & 31) == 0) atomicMax(&g->best, best_bits);
  __syncthreads();
  const float best = __uint_as_float(g->best), scale = best > 0.0f ? -kSharp / best : 0.0f;
  uint32_t mass[2];  // (whole numbers: the bucket must not fall from one step to the next)
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int c = 2 * tid + j;
    const bool inner = c == side - 1 || c == side;  // (an inner cell cannot be split)
    mass[j] = inner ? 0u : (uint32_t)(k[j] * (__expf((best - fmaxf(d[j], d[j + 1])) * scale) + kPrior) * 256.0f);
  }
  uint32_t run = block_prefix<THREADS>(mass[0] + mass[1], g->ipart, mass_total) - mass[0] - mass[1];
  const int groups = (signs & 1 ? octaves + 1 : 0) + (signs & 2 ? octaves + 1 : 0), spread = buckets - groups;
  const float per = mass_total ? (float)spread / (4.0f * (float)mass_total) : 0.0f;
  static_assert(kSteps == 4 * kCells, "a cell is four steps");
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int c = 2 * tid + j;
    if (c < 2 * side && (signs & (c < side ? 1 : 2))) {
      const int i = c < side ? side - 1 - c : c - side, o = (i + kCells - 1) >> kCellBits;  // o = 0: inner, else octave + 1
      const int group = c < side ? octaves - o : o + (signs & 1 ? octaves + 1 : 0);
      if (i == 0) {
        g->lut[c < side ? steps - 1 : steps] = (uint8_t)(group + min((int)((float)(4 * run) * per), spread - 1));
      } else {
#pragma unroll
        for (int q = 0; q < kSteps / kCells; ++q) {  // ascending in value
          const int b = group + min((int)((float)(4 * run + mass[j] * q) * per), spread - 1);
          const int in_side = 1 + (i - 1) * (kSteps / kCells) + (c < side ? kSteps / kCells - 1 - q : q);
          g->lut[c < side ? steps - 1 - in_side : steps + in_side] = (uint8_t)b;
        }
      }
    }
    run += mass[j];
  }
  __syncthreads();
  // edges of the buckets: where the bucket of a step differs from that of the one before
  const int first = signs & 1 ? 0 : steps, end = signs & 2 ? 2 * steps : steps;
  const uint32_t inner = (uint32_t)((low << kStepBits) - 1);  // pattern of the inner step
  for (int t = first + tid; t < end; t += THREADS) {
    const int b = g->lut[t], before = t > first ? (int)g->lut[t - 1] : -1;
    const int i = t < steps ? steps - 1 - t : t - steps;
    if (b != before) {
      const float v = t < steps ? -__uint_as_float((inner + i + 1) << kStepShift) : (i ? __uint_as_float((inner + i) << kStepShift) : 0.0f);
      const uint32_t octave = i ? ((inner + i) << kStepShift) & 0x7F800000u : 0u;
      for (int q = before + 1; q <= b; ++q) {
        g->edge[q] = v;
        g->elo[q] = q == b && i ? (t < steps ? -(double)__uint_as_float(octave) : (double)__uint_as_float(octave)) : 0.0;
        const double unit = i ? (double)__uint_as_float(octave - (23u << 23)) : 0.0;
        g->ulp[q] = q == b ? (t < steps ? -unit : unit) : 0.0;
      }
    }
    if (t == end - 1) {
      g->nb = b + 1;
      g->edge[b + 1] = signs & 2 ? __uint_as_float((inner + i + 1) << kStepShift) : 0.0f;
      if (!(signs & 2)) g->B0 = b + 1;
    }
    if (t == steps) g->B0 = b;
  }
  if (tid == 0) { g->base = (int)inner; g->side = steps; }
  __syncthreads();
}

// KHW, the kernel's window: 9 (3 x 3, unrolled), kAnyWindow (up to 32 pixels, one per lane) or kWideWindow (up to 64, two).
constexpr int kAnyWindow = 0, kWideWindow = -1;

// The pixels of a patch's window: their slots (kh*kw of them).  3 x 3 windows keep them in registers.
template <int KHW, bool kFixed = (KHW > 0)>
struct Window {
  int slot[KHW];
  const uint16_t* map;
  const uint16_t* win;
  __device__ __forceinline__ Window(const TileArgs&, const uint16_t* m, const uint16_t* w, int at) : map(m + at), win(w) {
#pragma unroll
    for (int i = 0; i < KHW; ++i) slot[i] = map[win[i]];
  }
  __device__ __forceinline__ int operator()(int i) const { return slot[i]; }
  __device__ __forceinline__ int at(int i) const { return map[win[i]]; }  // (an index known at run time only)
  static __device__ __forceinline__ int count(const TileArgs&) { return KHW; }
};
template <int KHW>
struct Window<KHW, false> {
  const uint16_t* map;
  const uint16_t* win;
  __device__ __forceinline__ Window(const TileArgs&, const uint16_t* m, const uint16_t* w, int at) : map(m + at), win(w) {}
  __device__ __forceinline__ int operator()(int i) const { return map[win[i]]; }
  __device__ __forceinline__ int at(int i) const { return map[win[i]]; }
  static __device__ __forceinline__ int count(const TileArgs& a) { return a.d.kh * a.d.kw; }
};

// Result of a patch.  K < 0: not settled.
struct PatchCode {
  int K;
  float alpha, beta, threshold;  // the high side is v >= threshold
  bool low_side;                 // e marks the low side
};

__device__ __forceinline__ float count_to_float(int s) {  // 0 <= s < 2^23, without the conversion unit
  return __int_as_float(0x4B000000 | s) - 8388608.0f;
}

// P^2/s + (T-P)^2/(n-s) to 1e-12 relative (both terms are non-negative).
__device__ __forceinline__ double objective_near(double P, double T, int s, int n) {
  const double sd = int_to_double(s), rd = int_to_double(n - s), Q = T - P;
  double r = (double)__fdividef(1.0f, count_to_float(s)), q = (double)__fdividef(1.0f, count_to_float(n - s));
  r = r * (2.0 - sd * r);
  q = q * (2.0 - rd * q);
  return P * P * r + Q * Q * q;
}

// A split of a row as the bucket test sees it: the means of its two sides and the objective, in fp32 from sums rounded once.  A side
// without values has the bound that its first value would obey (vlo, vhi) as its mean.
struct SplitState {
  float lo, hi, d;
};
__device__ __forceinline__ SplitState split_state(int s, float P, float Q, int n, float vlo, float vhi) {
  SplitState e;
  e.lo = s > 0 ? __fdividef(P, count_to_float(s)) : vlo;
  e.hi = s < n ? __fdividef(Q, count_to_float(n - s)) : vhi;
  e.d = __fmaf_rn(e.lo, P, e.hi * Q);  // (at s = 0 and s = n T^2 / n, which no split falls short of)
  return e;
}

// Can the best split lie in a bucket?  Two tests of the splits from its lower to its upper edge, the c values between them in
// [vlo, vhi] (c: all that the two splits differ by, a run of zeros among them):
//   bound   along the chord between the edges' (s, P) the objective is convex, so at most the larger of the edges'.  A split is off
//           the chord by at most c (vhi - vlo) / 4 =: e in P, where the objective's slope is at most twice the difference of the means
//           and its curvature adds e (vhi - vlo) at most;
//   means   a value that is closer to the other side's mean would improve the objective by changing sides, so the best
//           split's threshold is the middle of its two means.  Both means grow with the split: the middle lies between those of the
//           edges, and has to be in the bucket.
// The second alone leaves a few buckets, but far ones too where the objective has several maxima.
struct BucketTest {
  float bound, mid_lo, mid_hi, gap;
  __device__ __forceinline__ BucketTest(const SplitState& L, const SplitState& U, int c, float vlo, float vhi) {
    const float w = vhi - vlo;
    bound = __fmaf_rn(0.5f * count_to_float(c) * w, U.hi - L.lo + w, fmaxf(L.d, U.d));
    mid_lo = 0.5f * (L.lo + L.hi);
    mid_hi = 0.5f * (U.lo + U.hi);
    gap = L.hi - U.lo;
  }
  // margin: error of the middles.  A split that fails by more is worse than another by 2 * gap * margin; where that is not far above the
  // rounding of the objective (weak: the gap below which it is not), the test does not count.
  __device__ __forceinline__ bool passes(float need, float margin, float weak, float vlo, float vhi) const {
    return bound >= need && ((mid_lo - margin <= vhi && mid_hi + margin >= vlo) || !(gap >= weak));
  }
};

// The values of a hull, by the lists of the pixels of a 3 x 3 window: three lanes share a pixel.
template <typename ListT>
struct HullLists {
  static constexpr int kStep = 3;
  const ListT* from;
  const float* values;
  int count, sub;
  template <typename F>
  __device__ __forceinline__ void each(F f) const {  // f(value, is there one), the whole warp together
    for (int k = sub; __any_sync(0xFFFFFFFFu, k < count); k += kStep) {
      const bool in = k < count;
      f(in ? values[from[k]] : 0.0f, in);
    }
  }
};

// A hull as the search ends it: values with lo <= hull_place(value) < hi, `size` of them.
constexpr int kHullMax32 = 511, kHullMax64 = 1023;  // values of a hull at most, with 32 buckets (where it may be narrowed) and with 64
constexpr uint32_t kPlaces = 1u << 22;              // (the sum of that many places fits 32 bits)
struct HullRange {
  float origin, scale;
  uint32_t lo, hi;
  int size;
};
__device__ __forceinline__ uint32_t hull_place(float v, float origin, float scale) {  // (grows with v)
  return min((uint32_t)__float2uint_rz(__fmul_rn(__fsub_rn(v, origin), scale)), kPlaces - 1u);
}

// Narrows a hull of kNarrowFrom values and more: they are spread over 32 buckets of equal width, a lane each, and the buckets tested by
// BucketTest, until 31 are left or little changes.  z: zeros, at the place of 0 (0: none in the hull).  s_lo, P_lo: count and sum below the hull; best:
// an objective that is reached; table: 64 words.
// (Sorted in registers, 4 to 16 values a lane by as many variants of the code, they kept the warps of an SM waiting for instructions half of
// the time: inputs of the first binarized layer of the ResNet-18-shaped network at batch 32 544 us, narrowed from 64 values on 338.)
template <typename ListT>
__device__ __noinline__ void narrow_hull(const HullLists<ListT> lists, HullRange* range, uint32_t* table, float vlo, float vhi, int s_lo, double P_lo,
                                         double T, int n, int z, float best, float margin, int lane) {
  constexpr unsigned kAll = 0xFFFFFFFFu;
  HullRange r = *range;
  r.origin = vlo;
  r.scale = __fdividef((float)kPlaces, vhi - vlo);
  r.lo = 0u;
  r.hi = kPlaces;
  const float unit = (vhi - vlo) * (1.0f / kPlaces), Tf = (float)T;
  const uint32_t zero = hull_place(0.0f, r.origin, r.scale);
  int c_below = 0;          // values of the hull below r.lo, and the sum of their places
  uint32_t q_below = 0u;
  for (int level = 0; r.size + (z > 0 ? 1 : 0) > 31; ++level) {
    const uint32_t span = r.hi - r.lo;
    const int shift = max(27 - __clz((int)(span - 1u)), 0);  // at most 32 buckets
    table[lane] = 0u;
    table[32 + lane] = 0u;
    __syncwarp();
    lists.each([&](float v, bool in) {
      const uint32_t q = hull_place(v, r.origin, r.scale);
      if (in && q >= r.lo && q < r.hi) {
        atomicAdd(table + ((q - r.lo) >> shift), 1u);
        atomicAdd(table + 32 + ((q - r.lo) >> shift), q);
      }
    });
    __syncwarp();
    const int c = (int)table[lane];
    const uint32_t qc = table[32 + lane];
    int c1 = c;
    uint32_t q1 = qc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int uc = __shfl_up_sync(kAll, c1, o);
      const uint32_t uq = __shfl_up_sync(kAll, q1, o);
      if (lane >= o) { c1 += uc; q1 += uq; }
    }
    const int c0 = c1 - c;
    const uint32_t q0 = q1 - qc;
    // places are rounded: 1.5 units off the middle of one at most
    auto sum_of = [&](int count, uint32_t places) {
      return P_lo + int_to_double(count) * ((double)vlo + 0.5 * (double)unit) + (double)places * (double)unit;
    };
    const uint32_t from = r.lo + ((uint32_t)lane << shift), to = from + (1u << shift);
    const float blo = vlo + (float)from * unit, bhi = vlo + (float)to * unit;
    const double P0 = sum_of(c_below + c0, q_below + q0), P1 = sum_of(c_below + c1, q_below + q1);
    const int s0 = s_lo + c_below + c0 + (zero < from ? z : 0), s1 = s_lo + c_below + c1 + (zero < to ? z : 0);
    const SplitState L = split_state(s0, (float)P0, s0 > 0 ? (float)(T - P0) : Tf, n, blo, bhi), U = split_state(s1, (float)P1, (float)(T - P1), n, blo, bhi);
    const BucketTest test(L, U, s1 - s0, blo, bhi);
    const float off = 1.5f * unit * count_to_float(c_below + c1);  // of a sum
    const float off_d = 2.0f * off * (fabsf(U.hi - L.lo) + bhi - blo);
    const float here = from < r.hi ? fmaxf(L.d, U.d) - off_d : 0.0f;
    best = fmaxf(best, __uint_as_float(__reduce_max_sync(kAll, __float_as_uint(fmaxf(here, 0.0f)))));
    const float m = margin + 2.0f * unit + 0.5f * off * (__fdividef(1.0f, count_to_float(max(s0, 1))) + __fdividef(1.0f, count_to_float(max(n - s1, 1))));
    const unsigned keep = __ballot_sync(kAll, from < r.hi && test.passes(best * kKeep - off_d, m, best * (kWeak / margin), blo, bhi));
    if (keep == 0u) { r.size = kHullMax32 + 1; break; }
    const int first = __ffs((int)keep) - 1, last = 31 - __clz((int)keep);
    const int upto = __shfl_sync(kAll, c1, last), below = __shfl_sync(kAll, c0, first);
    const uint32_t q_first = __shfl_sync(kAll, q0, first);
    const int before = r.size;
    c_below += below;
    q_below += q_first;
    r.size = upto - below;
    r.hi = min(r.hi, r.lo + ((uint32_t)(last + 1) << shift));
    r.lo += (uint32_t)first << shift;
    if (shift == 0 || level == 3 || (4 * r.size > 3 * before && last - first >= 8)) break;
  }
  *range = r;
}

// The parts of a hull: lane i holds the part in pixel i of the window (and in pixel i + 32 of a wide one): the pixel's slot, where
// the part begins in its list, and how many values come before it (lanes beyond the window hold the total).
template <int KHW>
struct HullParts {
  static constexpr int kPerLane = KHW == kWideWindow ? 2 : 1;
  int before[kPerLane], slot[kPerLane], begin[kPerLane];
  int parts;
  __device__ __forceinline__ int of(const int (&v)[kPerLane], int part) const {  // (any part per lane)
    int r = __shfl_sync(0xFFFFFFFFu, v[0], part & 31);
    if (kPerLane > 1) {
      const int hi = __shfl_sync(0xFFFFFFFFu, v[kPerLane - 1], part & 31);
      if (part >= 32) r = hi;
    }
    return r;
  }
};

// The best split among the `size` values of a hull (and its run of z zeros, if `zeros`): E values a lane, sorted.  s_lo, P_lo:
// count and sum below the hull.  E = 1: the values are in `gathered` already.
struct HullSplit {
  int s;             // 0: none
  double P;
  uint32_t above;    // a key that the high side reaches and the low side does not
};

template <int E, int KHW, typename ListT>
__device__ __forceinline__ HullSplit search_hull(const float* gathered, const HullParts<KHW>& h, const float* tile, int pitch,
                                                 const ListT* list, int list_pitch, int size, bool zeros, int z, int s_lo, double P_lo, double T, int n,
                                                 int lane) {
  constexpr unsigned kAll = 0xFFFFFFFFu;
  constexpr int WN = KHW > 0 ? 16 : 32 * HullParts<KHW>::kPerLane;  // at least the window's pixels
  uint32_t key[E];
#pragma unroll
  for (int j = 0; j < E; ++j) {
    const int i = j * 32 + lane;
    if (E == 1) {
      key[j] = i < size ? order_key(gathered[i]) : (zeros && i == size ? kZeroKey : kPadKey);
      continue;
    }
    int part = 0;  // the last one that starts at or before i (parts that start there before it are empty)
#pragma unroll
    for (int step = WN / 2; step >= 1; step >>= 1) {
      const int o = h.of(h.before, part + step);
      if (part + step < h.parts && i >= o) part += step;
    }
    const int o = h.of(h.before, part), slot = h.of(h.slot, part), begin = h.of(h.begin, part);
    key[j] = zeros && i == size ? kZeroKey : kPadKey;
    if (i < size) key[j] = order_key(tile[slot * pitch + (int)list[slot * list_pitch + begin + i - o]]);
  }
  group_sort<1, E>(key, lane, nullptr, 0);
  double own = 0.0, P[E];
#pragma unroll
  for (int j = 0; j < E; ++j) {
    own = __dadd_rn(own, key[j] != kPadKey ? (double)key_value(key[j]) : 0.0);
    P[j] = own;
  }
  double before = own;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double u = __shfl_up_sync(kAll, before, o);
    if (lane >= o) before = __dadd_rn(before, u);
  }
  if (E > 1) {
    before = __shfl_up_sync(kAll, before, 1);
    if (lane == 0) before = 0.0;
    before = __dadd_rn(before, P_lo);
  } else {
    P[0] = __dadd_rn(before, P_lo);
  }
  const uint32_t next_first = __shfl_down_sync(kAll, key[0], 1);
  const int first = s_lo + lane * E + 1, more = zeros ? z - 1 : 0;
  double D[E], top = -1.0;
#pragma unroll
  for (int j = 0; j < E; ++j) {
    if (E > 1) P[j] = __dadd_rn(before, P[j]);
    const int s = first + j + (key[j] >= kZeroKey ? more : 0);
    const uint32_t next = j + 1 < E ? key[j + 1 < E ? j + 1 : 0] : next_first;
    D[j] = key[j] != kPadKey && (next != key[j] || lane * E + j == 32 * E - 1) && s < n ? objective_near(P[j], T, s, n) : -1.0;
    top = fmax(top, D[j]);
  }
  const int hi = __double2hiint(top), hmax = __reduce_max_sync(kAll, hi);
  const uint32_t lmax = __reduce_max_sync(kAll, hi == hmax ? (uint32_t)__double2loint(top) : 0u);
  const double least = __hiloint2double(hmax, (int)lmax) * kCloseBand;  // (at least zero where there is a split)
  int rivals = 0;
#pragma unroll
  for (int j = 0; j < E; ++j) rivals += D[j] >= least ? 1 : 0;
  HullSplit best{0, 0.0, 0u};
  if (hmax < 0) return best;
  const unsigned holders = __ballot_sync(kAll, rivals > 0);
  const bool tie = (holders & (holders - 1)) != 0u || __any_sync(kAll, rivals > 1);
  double mine = -1.0;
#pragma unroll
  for (int j = 0; j < E; ++j) {
    if (D[j] >= least) {  // ascending: ">=" keeps the largest split of equal objectives
      const int s = first + j + (key[j] >= kZeroKey ? more : 0);
      const double exact = tie ? objective(P[j], T, s, n) : D[j];
      if (exact >= mine) { mine = exact; best.s = s; best.P = P[j]; best.above = key[j] + 1u; }
    }
  }
  unsigned who = holders;
  if (tie) {  // Algorithm 1's ">=" on the exactly rounded objective
    const int h = __double2hiint(mine), hm = __reduce_max_sync(kAll, h);
    const uint32_t lm = __reduce_max_sync(kAll, h == hm ? (uint32_t)__double2loint(mine) : 0u);
    who = __ballot_sync(kAll, h == hm && (uint32_t)__double2loint(mine) == lm);
  }
  const int src = 31 - __clz(who);
  best.s = __shfl_sync(kAll, best.s, src);
  best.P = __shfl_sync(kAll, best.P, src);
  best.above = __shfl_sync(kAll, best.above, src);
  return best;
}

// The best split among up to 32 E - 1 values in no order (the zeros as one of them, if `zeros`), E a lane: those behind each value and, if
// `above` is not 0, that before all of them, whose high side reaches the key `above`.  s_lo, P_lo: count and sum below.
template <int E>
__device__ __noinline__ HullSplit search_narrowed(const float* hull, int size, bool zeros, int z, int s_lo, double P_lo, double T, int n, uint32_t above, int lane) {
  constexpr unsigned kAll = 0xFFFFFFFFu;
  const int values = size + (zeros ? 1 : 0);
  float x[E];
  int s[E];
  double P[E];
#pragma unroll
  for (int i = 0; i < E; ++i) {
    const int at = 32 * i + lane;
    x[i] = at < size ? hull[at] : (at < values ? 0.0f : __uint_as_float(0xFF800000u));
    s[i] = s_lo;
    P[i] = 0.0;
  }
#pragma unroll 2
  for (int j = 0; j < size; ++j) {
    const float v = hull[j];
    const double vd = (double)v;
#pragma unroll
    for (int i = 0; i < E; ++i)
      if (v <= x[i]) { ++s[i]; P[i] = __dadd_rn(P[i], vd); }
  }
  double D[E], top = -1.0;
#pragma unroll
  for (int i = 0; i < E; ++i) {
    const int at = 32 * i + lane;
    if (zeros && x[i] >= 0.0f) s[i] += z;
    P[i] = __dadd_rn(P_lo, P[i]);
    D[i] = (at < values || (at == 32 * E - 1 && above != 0u)) && s[i] > 0 && s[i] < n ? objective_near(P[i], T, s[i], n) : -1.0;
    top = fmax(top, D[i]);
  }
  HullSplit best{0, 0.0, 0u};
  auto warp_max = [&](double v) {  // (at least zero, or -1 in every lane)
    const int hi = __double2hiint(v), hmax = __reduce_max_sync(kAll, hi);
    return __hiloint2double(hmax, (int)__reduce_max_sync(kAll, hi == hmax ? (uint32_t)__double2loint(v) : 0u));
  };
  top = warp_max(top);
  if (top < 0.0) return best;
  const double least = top * kCloseBand;
  int rivals = 0, pick = 0;
#pragma unroll
  for (int i = 0; i < E; ++i)
    if (D[i] >= least) { ++rivals; pick = i; }
  unsigned who = __ballot_sync(kAll, rivals > 0);
  if ((who & (who - 1u)) || __any_sync(kAll, rivals > 1)) {  // Algorithm 1's ">=" on the exactly rounded objective: the largest split of equal ones
    double exact[E], most = -1.0;
#pragma unroll
    for (int i = 0; i < E; ++i) {
      exact[i] = D[i] >= least ? objective(P[i], T, s[i], n) : -1.0;
      most = fmax(most, exact[i]);
    }
    most = warp_max(most);
    int largest = 0;
#pragma unroll
    for (int i = 0; i < E; ++i)
      if (exact[i] == most && s[i] > largest) { largest = s[i]; pick = i; }
    const int all = __reduce_max_sync(kAll, largest);
    who = __ballot_sync(kAll, largest == all);
  }
  double Pp = P[0];
  int sp = s[0];
  float xp = x[0];
#pragma unroll
  for (int i = 1; i < E; ++i)
    if (pick == i) { Pp = P[i]; sp = s[i]; xp = x[i]; }
  if (32 * pick + lane < values) above = order_key(xp) + 1u;
  const int src = 31 - __clz((int)who);
  best.s = __shfl_sync(kAll, sp, src);
  best.P = __shfl_sync(kAll, Pp, src);
  best.above = __shfl_sync(kAll, above, src);
  return best;
}

template <int E, int KHW, typename ListT>
__device__ __noinline__ HullSplit search_long_hull(const HullParts<KHW> h, const float* tile, int pitch, const ListT* list, int list_pitch,
                                                   int size, bool zeros, int z, int s_lo, double P_lo, double T, int n, int lane) {
  return search_hull<E>(nullptr, h, tile, pitch, list, list_pitch, size, zeros, z, s_lo, P_lo, T, n, lane);
}

// The best split of one patch, by a warp.  A segment is a bucket or, between the negative and the positive buckets (at
// index B0), the run of zeros.  at: the window's first pixel in `map`; hull: 64 words of
// shared memory of the warp's own.  The result is valid in all lanes.
template <int KHW, int BPL, typename ListT>
__device__ __forceinline__ PatchCode search_patch(const TileArgs& a, const Grid& g, const uint16_t* map, const uint16_t* win, int at,
                                                  const double* sums, const uint16_t* counts, const ListT* list,
                                                  const float* tile, float* hull, int lane) {
  constexpr unsigned kAll = 0xFFFFFFFFu;
  constexpr int PER_LANE = HullParts<KHW>::kPerLane;
  const int n = a.n, B0 = g.B0, slots = a.slots;
  const int wn = Window<KHW>::count(a);
  PatchCode code{kRowMark, 0.0f, 0.0f, __uint_as_float(0x7FC00000u), false};
  HullParts<KHW> hp;
  hp.parts = wn;
#pragma unroll
  for (int t = 0; t < PER_LANE; ++t) hp.slot[t] = 32 * t + lane < wn ? map[at + win[32 * t + lane]] : 0;
  // ---- count and sum at the upper edge of buckets lane, lane + 32 ----
  int cc[BPL];
  double cs[BPL];
#pragma unroll
  for (int j = 0; j < BPL; ++j) { cc[j] = 0; cs[j] = 0.0; }
  {
    const int row = lane * slots;
    auto add = [&](int slot) {
      const uint16_t* const c = counts + row + slot;
      const double* const S = sums + row + slot;
#pragma unroll
      for (int j = 0; j < BPL; ++j) {
        cc[j] += c[32 * j * slots];
        cs[j] = __dadd_rn(cs[j], S[32 * j * slots]);
      }
    };
    if (KHW > 0) {
#pragma unroll
      for (int i = 0; i < (KHW > 0 ? KHW : 0); ++i) add(__shfl_sync(kAll, hp.slot[0], i));
    } else {
#pragma unroll
      for (int t = 0; t < PER_LANE; ++t)
#pragma unroll 4
        for (int i = 0; i < min(32, wn - 32 * t); ++i) add(__shfl_sync(kAll, hp.slot[t], i));
    }
  }
  const int m = __shfl_sync(kAll, cc[BPL - 1], 31);
  const double T = __shfl_sync(kAll, cs[BPL - 1], 31);
  if (m == 0) {  // nothing but zeros
    code.K = 0;
    return code;
  }
  const int z = n - m;
  auto state_at = [&](int b, int& c, double& S) {  // count and sum of the buckets before b (the same b for the warp)
    int tc = cc[0];
    double ts = cs[0];
    if (BPL > 1 && b > 32) { tc = cc[BPL - 1]; ts = cs[BPL - 1]; }
    c = __shfl_sync(kAll, tc, (b - 1) & 31);
    S = __shfl_sync(kAll, ts, (b - 1) & 31);
    if (b <= 0) { c = 0; S = 0.0; }
  };
  // ---- objective at the edges, in fp32 from exact sums ----
  float Pf[BPL], Qf[BPL], d[BPL], best = -1.0f;
  auto edge_D = [&](int s, float P, float Q) {
    return s > 0 && s < n ? __fdividef(P * P, count_to_float(s)) + __fdividef(Q * Q, count_to_float(n - s)) : -1.0f;
  };
#pragma unroll
  for (int j = 0; j < BPL; ++j) {
    Pf[j] = (float)cs[j];
    Qf[j] = (float)(T - cs[j]);
    d[j] = edge_D(cc[j] + (32 * j + lane >= B0 ? z : 0), Pf[j], Qf[j]);
    best = fmaxf(best, d[j]);
  }
  float dz0 = -1.0f, dz1 = -1.0f;  // before and behind the run of zeros
  if (z > 0) {
    int neg = 0;
    float Pn = 0.0f, Qn = (float)T;
    if (B0 > 0) {
      const int k = BPL > 1 && B0 > 32 ? BPL - 1 : 0, from = (B0 - 1) & 31;
      neg = __shfl_sync(kAll, cc[k], from);
      Pn = __shfl_sync(kAll, Pf[k], from);
      Qn = __shfl_sync(kAll, Qf[k], from);
      dz0 = __shfl_sync(kAll, d[k], from);
    }
    dz1 = edge_D(neg + z, Pn, Qn);
    best = fmaxf(best, dz1);
  }
  best = __uint_as_float(__reduce_max_sync(kAll, __float_as_uint(fmaxf(best, 0.0f))));
  const float need = best * kKeep;
  // ---- segments whose bound reaches the best edge ----
  int seg_lo = 1 << 20, seg_hi = -1;
#pragma unroll
  for (int j = 0; j < BPL; ++j) {
    const int b = 32 * j + lane;
    int c0 = __shfl_up_sync(kAll, cc[j], 1);
    float d0 = __shfl_up_sync(kAll, d[j], 1), P0 = __shfl_up_sync(kAll, Pf[j], 1), Q0 = __shfl_up_sync(kAll, Qf[j], 1);
    if (j > 0) {
      const int k = j > 0 ? j - 1 : 0;
      const int c31 = __shfl_sync(kAll, cc[k], 31);
      const float d31 = __shfl_sync(kAll, d[k], 31), P31 = __shfl_sync(kAll, Pf[k], 31), Q31 = __shfl_sync(kAll, Qf[k], 31);
      if (lane == 0) { c0 = c31; d0 = d31; P0 = P31; Q0 = Q31; }
    } else if (lane == 0) {
      c0 = 0;
      d0 = -1.0f;
      P0 = 0.0f;
      Q0 = (float)T;
    }
    if (b == B0 && z > 0) d0 = dz1;
    double S0 = __shfl_up_sync(kAll, cs[j], 1);
    if (j > 0) {
      const double S31 = __shfl_sync(kAll, cs[j > 0 ? j - 1 : 0], 31);
      if (lane == 0) S0 = S31;
    } else if (lane == 0) {
      S0 = 0.0;
    }
    const int c = cc[j] - c0;
    float bound = fmaxf(d0, d[j]);
    if (c >= 2) {
      // the two inner corners of the region (s, P) visits inside the bucket
      const float vlo = g.edge[b], vhi = g.edge[b + 1], cf = count_to_float(c), sf = count_to_float(c0 + (b >= B0 ? z : 0));
      const float ju = fminf(fmaxf(__fdividef((float)__dsub_rn(__dsub_rn(cs[j], S0), (double)vlo * int_to_double(c)), vhi - vlo), 0.0f), cf);
      const float jl = cf - ju;
      const float nf = count_to_float(n);
      auto corner = [&](float js, float v) {
        const float s = sf + js, r = nf - s, P = P0 + js * v, Q = Q0 - js * v;
        return (s > 0.0f ? __fdividef(P * P, s) : 0.0f) + (r > 0.0f ? __fdividef(Q * Q, r) : 0.0f);
      };
      bound = fmaxf(bound, fmaxf(corner(jl, vlo), corner(ju, vhi)));
    }
    if (c > 0 && bound >= need) {
      const int seg = b + (b >= B0 ? 1 : 0);
      seg_lo = min(seg_lo, seg);
      seg_hi = max(seg_hi, seg);
    }
  }
  if (z > 0 && fmaxf(dz0, dz1) >= need) { seg_lo = min(seg_lo, B0); seg_hi = max(seg_hi, B0); }
  seg_lo = __reduce_min_sync(kAll, seg_lo);
  seg_hi = __reduce_max_sync(kAll, seg_hi);
  if (!(best > 1e-30f) || seg_hi < 0) return code;
  const int b_lo = seg_lo > B0 ? seg_lo - 1 : seg_lo, b_end = seg_hi >= B0 ? seg_hi : seg_hi + 1;  // buckets of the hull
  const bool zeros = z > 0 && seg_lo <= B0 && B0 <= seg_hi;
  int c_lo, c_end;
  double P_lo;
  state_at(b_lo, c_lo, P_lo);
  {
    const int tc = BPL > 1 && b_end > 32 ? cc[BPL - 1] : cc[0];
    c_end = __shfl_sync(kAll, tc, (b_end - 1) & 31);
  }
  const int size = c_end - c_lo, s_lo = c_lo + (seg_lo > B0 ? z : 0);
  if (size < 1 || size > (BPL == 1 ? kHullMax32 : kHullMax64) || (z == 0 && size == n)) return code;
  if (b_lo >= B0 - 1 && b_end <= B0 + 1) {  // the two buckets next to zero: does the patch have no other values?
    int below, upto;
    double unused;
    state_at(B0 - 1, below, unused);
    state_at(B0 + 1, upto, unused);
    if (upto - below == m) return code;
  }
  // ---- their values, from the lists of the window's pixels ----
  int count[PER_LANE], total = 0;
#pragma unroll
  for (int t = 0; t < PER_LANE; ++t) {
    hp.begin[t] = count[t] = 0;
    if (32 * t + lane < wn) {
      hp.begin[t] = b_lo > 0 ? counts[(b_lo - 1) * slots + hp.slot[t]] : 0;
      count[t] = (b_end > 0 ? counts[(b_end - 1) * slots + hp.slot[t]] : 0) - hp.begin[t];
    }
    int incl = count[t];
#pragma unroll
    for (int o = 1; o < (KHW > 0 ? 16 : 32); o <<= 1) {
      const int u = __shfl_up_sync(kAll, incl, o);
      if (lane >= o) incl += u;
    }
    hp.before[t] = total + incl - count[t];
    if (t + 1 < PER_LANE) total += __shfl_sync(kAll, incl, 31);
  }
  constexpr bool kNarrow = KHW == 9 && BPL == 1;
  HullSplit split;
#define DAB_HULL hp, tile, a.pitch, list, 4 * a.quads, size, zeros, z, s_lo, P_lo, T, n, lane
  if (size < 32) {  // the usual case: the pixels' lanes bring the values together in shared memory
#pragma unroll
    for (int t = 0; t < PER_LANE; ++t) {
      const ListT* const from = list + hp.slot[t] * 4 * a.quads + hp.begin[t];
      const float* const values = tile + hp.slot[t] * a.pitch;
      for (int k = 0; k < count[t]; ++k) hull[hp.before[t] + k] = values[from[k]];
    }
    __syncwarp();
    split = search_hull<1>(hull, DAB_HULL);
    __syncwarp();
  }
  else if (size < 64) split = search_long_hull<2>(DAB_HULL);
  else if (size < kNarrowFrom) split = search_long_hull<4>(DAB_HULL);
  else if (!kNarrow && size < 256) split = search_long_hull<8>(DAB_HULL);
  else if (!kNarrow && (BPL == 1 || size < 512)) split = search_long_hull<16>(DAB_HULL);
  else if (!kNarrow) split = search_long_hull<(BPL == 1 ? 16 : 32)>(DAB_HULL);
  else {  // narrowed first
    HullLists<ListT> lists;
    lists.sub = lane % lists.kStep;
    lists.count = 0;
    if (lane / lists.kStep < wn) {
      const int slot = map[at + win[lane / lists.kStep]], begin = b_lo > 0 ? counts[(b_lo - 1) * slots + slot] : 0;
      lists.count = (int)counts[(b_end - 1) * slots + slot] - begin;
      lists.from = list + slot * 4 * a.quads + begin;
      lists.values = tile + slot * a.pitch;
    }
    HullRange r;
    r.size = size;
    const float margin = 2e-6f * __uint_as_float(g.top);  // (the middles are good to 1e-6 of the larger mean)
    narrow_hull(lists, &r, reinterpret_cast<uint32_t*>(hull), g.edge[b_lo], g.edge[b_end], s_lo, P_lo, T, n, zeros ? z : 0, best, margin, lane);
    bool inside = zeros;
    int s_base = s_lo;
    uint32_t top = 0u;  // a key above all that lies below
    if (zeros) {
      const uint32_t q = hull_place(0.0f, r.origin, r.scale);
      if (q < r.lo) { s_base += z; top = kZeroKey + 1u; }
      inside = q >= r.lo && q < r.hi;
    }
    bool sorted = r.size + (inside ? 1 : 0) > 63;  // the whole hull
    if (!sorted) {
      // The lists are in the order in which threads came.  From 2^(e - 20) on, e the exponent of the hull's larger edge, values are multiples
      // of 2^(e - 43), and 511 of them stay below 2^(e + 10): their sums are exact in any order.  A hull with a smaller one is sorted.
      const float edge = fmaxf(fabsf(g.edge[b_lo]), fabsf(g.edge[b_end]));
      const float exact_from = __uint_as_float((__float_as_uint(edge) & 0x7F800000u) - (20u << 23));
      int fill = 0;
      double below = 0.0;
      bool inexact = false;
      lists.each([&](float v, bool in) {
        const uint32_t q = hull_place(v, r.origin, r.scale);
        const bool is_low = in && q < r.lo;
        in = in && q >= r.lo && q < r.hi;
        inexact = inexact || ((in || is_low) && fabsf(v) < exact_from);
        const unsigned bal = __ballot_sync(kAll, in);
        if (in) hull[fill + __popc(bal & ((1u << lane) - 1u))] = v;
        fill += __popc(bal);
        s_base += __popc(__ballot_sync(kAll, is_low));
        if (is_low) { below = __dadd_rn(below, (double)v); top = max(top, order_key(v) + 1u); }
      });
      sorted = __any_sync(kAll, inexact);
      if (!sorted) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) below = __dadd_rn(below, __shfl_xor_sync(kAll, below, o));
        top = __reduce_max_sync(kAll, top);
        __syncwarp();
        below = __dadd_rn(P_lo, below);
        split = fill < 31 ? search_narrowed<1>(hull, fill, inside, z, s_base, below, T, n, top, lane)
                          : search_narrowed<2>(hull, fill, inside, z, s_base, below, T, n, top, lane);
      }
      __syncwarp();
    }
    if (sorted) {
      if (size >= 256 && n <= kMarkRows) return code;
      split = size < 256 ? search_long_hull<8>(DAB_HULL) : search_long_hull<16>(DAB_HULL);
    }
  }
#undef DAB_HULL
  if (split.s <= 0 || split.s >= n) return code;
  // the two means side by side in the even and the odd lanes
  const bool odd = lane & 1;
  const double mean = __ddiv_rn(odd ? __dsub_rn(T, split.P) : split.P, int_to_double(odd ? n - split.s : split.s));
  const double m_lo = __shfl_sync(kAll, mean, 0), m_hi = __shfl_sync(kAll, mean, 1);
  code.low_side = fabs(m_lo) > fabs(m_hi);  // e marks the partition whose mean is larger in magnitude
  code.K = code.low_side ? split.s : n - split.s;
  code.alpha = (float)(code.low_side ? m_lo : m_hi);
  code.beta = (float)(code.low_side ? m_hi : m_lo);
  code.threshold = key_value(split.above);
  return code;
}

template <int KHW, int BPL, typename ListT>
__global__ void __launch_bounds__(kTileThreads, 2) binarize_patches_tile_kernel(const TileArgs a) {
  constexpr int THREADS = kTileThreads, WARPS = kTileWarps, BUCKETS = 32 * BPL;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int slots = a.slots, C = a.d.C, khw = a.d.kh * a.d.kw, window = a.in_h * a.in_w;
  // dead once the patches are searched; the assembled masks then take their place
  double* const sums = reinterpret_cast<double*>(smem_raw);                       // [bucket][slot] cumulative sums ...
  uint32_t* const cells = reinterpret_cast<uint32_t*>(smem_raw);                  // ... in place of (count, sum of the mantissas)
  // [2][slot] sums of what the grid does not resolve: in units of 2^-kTinyBits of its lowest octave, so that they are the same
  // whatever the order (an atomic fp64 sum rounds as the order falls)
  unsigned long long* const tiny = reinterpret_cast<unsigned long long*>(sums + (size_t)BUCKETS * slots);
  uint16_t* const counts = reinterpret_cast<uint16_t*>(tiny + 2 * slots);         // [bucket][slot] cumulative counts
  ListT* const list = reinterpret_cast<ListT*>(counts + (size_t)BUCKETS * slots);  // [slot][4 * quads] channels by bucket
  // kept
  float* const tile = reinterpret_cast<float*>(smem_raw + a.tile_at);             // [slot][pitch] values
  int* const poff = reinterpret_cast<int*>(tile + (size_t)slots * a.pitch);       // [slot] offset in a channel plane
  float* const threshold = reinterpret_cast<float*>(poff + slots);                // [patch] of the tile; NaN: empty mask
  uint32_t* const invert = reinterpret_cast<uint32_t*>(threshold + a.TH * a.TW);  // [patch] all ones: e marks the low side
  uint16_t* const map = reinterpret_cast<uint16_t*>(invert + a.TH * a.TW);        // [window] slot of a pixel under the tile
  uint16_t* const win = map + window;                                             // [kh*kw] offsets of the window
  __shared__ Grid grid;
  static_assert(kMaxCells <= kTileWarps * 32, "cells");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  int t = blockIdx.x;
  const int tx = t % a.tiles_w;
  t /= a.tiles_w;
  const int ty = t % a.tiles_h, img = t / a.tiles_h;
  const int ho0 = ty * a.TH, wo0 = tx * a.TW, th = min(a.TH, a.Ho - ho0), tw = min(a.TW, a.Wo - wo0), npatch = th * tw;
  const int h0 = ho0 * a.d.stride_h - a.d.pad_h, w0 = wo0 * a.d.stride_w - a.d.pad_w;
  // the part of the image under the tile; slot `pixels` stands for the padding
  const int r0 = max(h0, 0), r1 = min(h0 + (th - 1) * a.d.stride_h + a.d.kh, a.d.H);
  const int q0 = max(w0, 0), q1 = min(w0 + (tw - 1) * a.d.stride_w + a.d.kw, a.d.W);
  const int cols = max(q1 - q0, 0), pixels = max(r1 - r0, 0) * cols;
  const int64_t first_patch = ((int64_t)img * a.Ho + ho0) * a.Wo + wo0;
  auto patch_index = [&](int p) { return first_patch + (int64_t)(p / tw) * a.Wo + p % tw; };
  auto window_at = [&](int p) { return p / tw * a.d.stride_h * a.in_w + p % tw * a.d.stride_w; };

  // ---- tables of offsets, cleared counters ----
  for (int i = tid; i < window; i += THREADS) {
    const int h = h0 + i / a.in_w, w = w0 + i % a.in_w;
    map[i] = (uint16_t)(h >= r0 && h < r1 && w >= q0 && w < q1 ? (h - r0) * cols + w - q0 : pixels);
  }
  for (int i = tid; i < khw; i += THREADS) win[i] = (uint16_t)(i / a.d.kw * a.in_w + i % a.d.kw);
  for (int i = tid; i < pixels; i += THREADS) poff[i] = (r0 + i / cols) * a.d.W + q0 + i % cols;
  for (int i = tid; i < (BUCKETS + 2) * slots; i += THREADS) sums[i] = 0.0;
  for (int i = tid; i < kMaxCells; i += THREADS) grid.hist[i] = 0u;
  if (tid == 0) { grid.top = 0u; grid.signs = 0; grid.best = 0u; }
  for (int i = tid; i < a.pitch; i += THREADS) tile[(size_t)pixels * a.pitch + i] = 0.0f;
  __syncthreads();

  // ---- stage the values (-0.0 becomes +0.0); largest magnitude, signs ----
  const int units = pixels * a.quads;
  const uint32_t magic = pixels > 1 ? (uint32_t)((0x100000000ull + (unsigned)pixels - 1) / (unsigned)pixels) : 0u;
  {
    const int plane = a.d.H * a.d.W;
    const float* const ximg = a.x + (int64_t)img * C * plane;
    uint32_t top = 0u;
    int signs = 0;
#pragma unroll 4
    for (int u = tid; u < units; u += THREADS) {
      const int q = magic ? (int)__umulhi((unsigned)u, magic) : u, p = u - q * pixels, c = 4 * q;
      const int at = c * plane + poff[p];
      float v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = c + j < C ? __fadd_rn(__ldg(ximg + DAB_IDX(at + j * plane, (int64_t)C * plane)), 0.0f) : 0.0f;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        top = max(top, __float_as_uint(v[j]) & 0x7FFFFFFFu);
        signs |= (v[j] < 0.0f ? 1 : 0) | (v[j] > 0.0f ? 2 : 0);
      }
      *reinterpret_cast<float4*>(tile + p * a.pitch + c) = make_float4(v[0], v[1], v[2], v[3]);
    }
    top = __reduce_max_sync(0xFFFFFFFFu, top);
    signs = __reduce_or_sync(0xFFFFFFFFu, signs);
    if (lane == 0) {
      atomicMax(&grid.top, top);
      atomicOr(&grid.signs, signs);
    }
  }
  __syncthreads();
  const uint32_t top = grid.top;
  const int e = (int)(top >> 23) - 127;
  if (top != 0u && (top >= 0x7F800000u || e < -40 || e > 40)) {  // left to the CTA-per-patch kernel
    for (int p = tid; p < npatch; p += THREADS) {
      const int64_t pi = patch_index(p);
      if (DAB_IN_BOUNDS(pi, patch_count(a))) a.pK[pi] = kRowMark;
    }
    return;
  }

  if (top != 0u) {
    // ---- the grid, from about two thousand values spread over the tile ----
    {
      const int side = a.octaves * kCells + 1, base = (((int)(top >> 23) - a.octaves + 1) << kCellBits) - 1;
      const int samples = min(units, kSampledUnits), step = units / samples;
      for (int i = tid; i < samples; i += THREADS) {
        const int u = i * step, q = magic ? (int)__umulhi((unsigned)u, magic) : u, p = u - q * pixels;
        const float4 f = *reinterpret_cast<const float4*>(tile + p * a.pitch + 4 * q);
        const float v[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int c = min(max((int)((__float_as_uint(v[j]) & 0x7FFFFFFFu) >> kCellShift) - base, 0), side - 1);
          if (v[j] != 0.0f) atomicAdd(&grid.hist[v[j] < 0.0f ? side - 1 - c : side + c], 1u);
        }
      }
      __syncthreads();
      choose_grid<THREADS>(&grid, a.octaves, BUCKETS, 4 * samples);
    }
    const int nb = grid.nb, B0 = grid.B0, base = grid.base, side = grid.side;
    const bool negatives = grid.signs & 1;
    const int low = (int)(top >> 23) - 127 - a.octaves + 1;  // 2^low: what the unresolved values stay below
    const float tiny_scale = __int_as_float((127 + kTinyBits - low) << 23);
    const double tiny_unit = __hiloint2double((1023 + low - kTinyBits) << 20, 0);
    // ---- per pixel: count and sum of the mantissas per bucket ----
#pragma unroll 2
    for (int u = tid; u < units; u += THREADS) {
      const int q = magic ? (int)__umulhi((unsigned)u, magic) : u, p = u - q * pixels;
      const float4 f = *reinterpret_cast<const float4*>(tile + p * a.pitch + 4 * q);
      const float v[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (v[j] != 0.0f) {
          const uint32_t m = __float_as_uint(v[j]) & 0x7FFFFFFFu;
          const int c = grid_step(m, base, side), slot = grid_bucket(grid, v[j], c, side) * slots + p;
          atomicAdd(&cells[2 * slot], 1u);
          if (c > 0) atomicAdd(&cells[2 * slot + 1], m & 0x7FFFFFu);
          else atomicAdd(&tiny[(v[j] < 0.0f ? 0 : slots) + p], (unsigned long long)__float2ll_rn(__fmul_rn(v[j], tiny_scale)));
        }
      }
    }
    __syncthreads();
    // ---- per pixel: exclusive cumulative counts, inclusive cumulative sums ----
    if (pixels < kSerialPixels) {  // a warp each, a lane per bucket
      for (int p = warp; p <= pixels; p += WARPS) {
        int run = 0;
        double sum = 0.0;
#pragma unroll
        for (int j = 0; j < BPL; ++j) {
          const int b = 32 * j + lane;
          const uint2 cell = *reinterpret_cast<const uint2*>(cells + 2 * (b * slots + p));
          double part = __dadd_rn(__dmul_rn((double)cell.x, grid.elo[b]), __dmul_rn((double)cell.y, grid.ulp[b]));
          if (b == B0) part = __dmul_rn((double)(long long)tiny[slots + p], tiny_unit);
          if (b == B0 - 1 && negatives) part = __dmul_rn((double)(long long)tiny[p], tiny_unit);
          if (b >= nb) part = 0.0;  // (the buckets beyond nb are empty)
          int c = (int)cell.x;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const int uc = __shfl_up_sync(0xFFFFFFFFu, c, o);
            const double us = __shfl_up_sync(0xFFFFFFFFu, part, o);
            if (lane >= o) { c += uc; part = __dadd_rn(part, us); }
          }
          part = __dadd_rn(part, sum);
          counts[b * slots + p] = (uint16_t)(run + c - (int)cell.x);
          sums[b * slots + p] = part;
          run += __shfl_sync(0xFFFFFFFFu, c, 31);
          sum = __shfl_sync(0xFFFFFFFFu, part, 31);
        }
      }
    } else {  // a thread each
      for (int p = tid; p <= pixels; p += THREADS) {
        int run = 0;
        double sum = 0.0;
        const double inner_neg = __dmul_rn((double)(long long)tiny[p], tiny_unit), inner_pos = __dmul_rn((double)(long long)tiny[slots + p], tiny_unit);
#pragma unroll 4
        for (int b = 0; b < BUCKETS; ++b) {  // (the buckets beyond nb are empty)
          const uint2 cell = *reinterpret_cast<const uint2*>(cells + 2 * (b * slots + p));
          double part = __dadd_rn(__dmul_rn((double)cell.x, grid.elo[b]), __dmul_rn((double)cell.y, grid.ulp[b]));
          if (b == B0) part = inner_pos;
          if (b == B0 - 1 && negatives) part = inner_neg;
          sum = b < nb ? __dadd_rn(sum, part) : sum;
          counts[b * slots + p] = (uint16_t)run;
          run += (int)cell.x;
          sums[b * slots + p] = sum;
        }
      }
    }
    __syncthreads();
    if (sizeof(ListT) > 1 && C > 512) {
      // 32 bits hold the mantissas of 512 values: what a bucket with more of them has lost is some 2^32 units of its octave
      for (int p = tid; p < pixels; p += THREADS)
        for (int b = 0; b < nb; ++b) {  // (nb < BUCKETS)
          if (counts[(b + 1) * slots + p] - counts[b * slots + p] <= 512 || b == B0 || (b == B0 - 1 && negatives)) continue;
          const double lost = __dsub_rn(sum_by_channel(grid, tile + p * a.pitch, C, b), __dsub_rn(sums[b * slots + p], b ? sums[(b - 1) * slots + p] : 0.0));
          const double unit = __dmul_rn(4294967296.0, grid.ulp[b]);
          for (int q = b; q < BUCKETS; ++q) sums[q * slots + p] = __dadd_rn(sums[q * slots + p], __dmul_rn(rint(__ddiv_rn(lost, unit)), unit));
        }
      __syncthreads();
    }
    // ---- per pixel: channels ordered by bucket; the cursors end as inclusive cumulative counts ----
#pragma unroll 2
    for (int u = tid; u < units; u += THREADS) {
      const int q = magic ? (int)__umulhi((unsigned)u, magic) : u, p = u - q * pixels;
      const float4 f = *reinterpret_cast<const float4*>(tile + p * a.pitch + 4 * q);
      const float v[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (v[j] != 0.0f) {
          const int c = grid_step(__float_as_uint(v[j]) & 0x7FFFFFFFu, base, side);
          const int slot = grid_bucket(grid, v[j], c, side) * slots + p, shift = (slot & 1) << 4;  // 16-bit cursors, two to a word
          const uint32_t old = atomicAdd(reinterpret_cast<uint32_t*>(counts) + (slot >> 1), 1u << shift);
          list[p * 4 * a.quads + (int)((old >> shift) & 0xFFFFu)] = (ListT)(4 * q + j);
        }
      }
    }
    __syncthreads();
    // (in the buckets beyond nb the cursors never move: their cumulative counts are those of the last one)
  }

  auto store = [&](int p, const PatchCode& code) {
    threshold[p] = code.threshold;
    invert[p] = code.low_side ? 0xFFFFFFFFu : 0u;
    const int64_t pi = patch_index(p);
    if (DAB_IN_BOUNDS(pi, patch_count(a))) {
      a.pK[pi] = code.K;
      if (code.K >= 0) {
        a.pgamma[pi] = code.alpha;
        a.pdelta[pi] = code.beta;
        if (a.pflags) a.pflags[pi] = code.K > 0 ? 0u : DAB_ROW_DEGENERATE;
      }
    }
  };
  // ---- the search: a warp per patch ----
  for (int p = warp; p < npatch; p += WARPS) {
    PatchCode code{0, 0.0f, 0.0f, __uint_as_float(0x7FC00000u), false};
    if (top != 0u) code = search_patch<KHW, BPL>(a, grid, map, win, window_at(p), sums, counts, list, tile, reinterpret_cast<float*>(grid.scratch[warp]), lane);
    __syncwarp();
    if (lane == 0) store(p, code);
  }
  __syncthreads();

  // ---- masks: a thread per patch and 32 channels (kh*kw words); the words replace the tables ----
  uint32_t* const words = reinterpret_cast<uint32_t*>(smem_raw);
  const int cblocks = (a.quads + 7) >> 3, pgroups = (npatch + 31) >> 5;
  for (int u = warp; u < cblocks * pgroups; u += WARPS) {
    const int cb = u / pgroups, p = (u - cb * pgroups) * 32 + lane, pl = min(p, npatch - 1);
    const Window<KHW> w(a, map, win, window_at(pl));
    const float tv = threshold[pl];
    const uint32_t inv = invert[pl];
    const bool none = !(tv == tv);
    const float* const src = tile + cb * 32;
    uint32_t* const dst = words + pl * a.word_pitch + cb * khw;
    const int room = p < npatch ? a.word_pitch - cb * khw : 0;
    const int quads = min(8, a.quads - cb * 8);
    uint64_t acc = 0u;   // bits not yet stored
    int have = 0, k = 0;
    auto append = [&](uint32_t bits, int count) {
      acc |= (uint64_t)bits << have;
      have += count;
      if (have >= 32) {
        if (k < room) dst[k] = none ? 0u : (uint32_t)acc;
        ++k;
        acc >>= 32;
        have -= 32;
      }
    };
    // bit = [v >= tv] ^ inv = sign of v - tv, complemented unless inverted (no value is -0.0, so v = tv gives +0)
    if (KHW == 9) {
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        uint32_t b[4] = {0u, 0u, 0u, 0u};
        if (q < quads) {
#pragma unroll
          for (int i = KHW - 1; i >= 0; --i) {
            const float4 v = *reinterpret_cast<const float4*>(src + w(i) * a.pitch + 4 * q);
            b[0] = __funnelshift_l(__float_as_uint(v.x - tv), b[0], 1);
            b[1] = __funnelshift_l(__float_as_uint(v.y - tv), b[1], 1);
            b[2] = __funnelshift_l(__float_as_uint(v.z - tv), b[2], 1);
            b[3] = __funnelshift_l(__float_as_uint(v.w - tv), b[3], 1);
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) b[j] = cb * 32 + 4 * q + j < C ? (b[j] ^ ~inv) & 0x1FFu : 0u;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) append(b[j], 9);
      }
    } else {
      const int low = KHW == kWideWindow ? 32 : khw;
      for (int q = 0; q < 8; ++q) {
        uint32_t b[4] = {0u, 0u, 0u, 0u}, high[4] = {0u, 0u, 0u, 0u};  // high: pixels 32 and on of a wide window
        auto bits_of = [&](uint32_t (&to)[4], int first, int count, uint32_t all) {
#pragma unroll 5
          for (int i = first + count - 1; i >= first; --i) {
            const float4 v = *reinterpret_cast<const float4*>(src + w(i) * a.pitch + 4 * q);
            to[0] = __funnelshift_l(__float_as_uint(v.x - tv), to[0], 1);
            to[1] = __funnelshift_l(__float_as_uint(v.y - tv), to[1], 1);
            to[2] = __funnelshift_l(__float_as_uint(v.z - tv), to[2], 1);
            to[3] = __funnelshift_l(__float_as_uint(v.w - tv), to[3], 1);
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) to[j] = cb * 32 + 4 * q + j < C ? (to[j] ^ ~inv) & all : 0u;
        };
        if (q < quads) {
          bits_of(b, 0, low, low == 32 ? 0xFFFFFFFFu : (1u << low) - 1u);
          if (KHW == kWideWindow) bits_of(high, 32, khw - 32, khw == 64 ? 0xFFFFFFFFu : (1u << (khw - 32)) - 1u);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          append(b[j], low);
          if (KHW == kWideWindow) append(high[j], khw - 32);
        }
      }
    }
  }
  __syncthreads();
  // (the words of an output row of the tile are contiguous)
  const int live = (a.n + 31) >> 5, all = npatch * a.ldp;
  const uint32_t magic_tw = tw > 1 ? (uint32_t)((0x100000000ull + (unsigned)tw - 1) / (unsigned)tw) : 0u;
#pragma unroll 2
  for (int i = tid; i < all; i += THREADS) {
    const int p = (int)__umulhi((unsigned)i, a.magic_ldp), k = i - p * a.ldp;
    const int lh = magic_tw ? (int)__umulhi((unsigned)p, magic_tw) : p;
    const int64_t at = (first_patch + (int64_t)lh * a.Wo + (p - lh * tw)) * a.ldp + k;
    if (DAB_IN_BOUNDS(at, patch_count(a) * a.ldp)) a.pmask[at] = k < live ? words[p * a.word_pitch + k] : 0u;
  }
}

void set_tile(TileArgs* a, int th, int tw) {
  const dab_conv_desc& d = a->d;
  a->TH = th < a->Ho ? th : a->Ho;
  a->TW = tw < a->Wo ? tw : a->Wo;
  a->in_h = (a->TH - 1) * d.stride_h + d.kh;
  a->in_w = (a->TW - 1) * d.stride_w + d.kw;
  a->tiles_h = (a->Ho + a->TH - 1) / a->TH;
  a->tiles_w = (a->Wo + a->TW - 1) / a->TW;
  a->slots = (a->in_h < d.H ? a->in_h : d.H) * (a->in_w < d.W ? a->in_w : d.W) + 1;
  a->slots |= 1;  // odd: the buckets of a pixel in different banks
}

template <typename ListT>
size_t tile_bytes(TileArgs* t) {
  TileArgs& a = *t;
  const size_t slots = a.slots, khw = (size_t)a.d.kh * a.d.kw, patches = (size_t)a.TH * a.TW;
  size_t tables = slots * (10 * (size_t)a.buckets + 16 + 4 * (size_t)a.quads * sizeof(ListT));
  const size_t words = sizeof(uint32_t) * patches * a.word_pitch;  // the assembled masks replace the tables
  if (words > tables) tables = words;
  a.tile_at = (uint32_t)((tables + 15) & ~(size_t)15);
  return a.tile_at + sizeof(float) * slots * a.pitch + 4 * slots + 8 * patches + 2 * ((size_t)a.in_h * a.in_w + khw);
}

constexpr size_t kSmemPerSm = 228 * 1024, kSmemCtaMax = 227 * 1024, kTileStatic = sizeof(Grid) + 64;

// The tile whose estimated time over the whole layer is least, in cycles.  From phase timings on 64 x 56 x 56 (7 x 14 tiles,
// two CTAs per SM): per tile a fixed part, 4.3 per staged value and 6200 per round of 16 patches (a warp each); a CTA alone
// on its SM takes 0.65 of that.  The model met the measured times of 30 tile shapes on four layers within 10 %.
// Returned is what the chosen tiles take with all that is left out there because every tile has it (tables of offsets, the grid,
// masks): 25000 cycles, 2.7 per staged value and 8100 per round for a CTA of a pair, 20000, 1.5 and 6000 for one alone.
template <typename ListT>
double choose_tile(TileArgs* a, size_t* smem_out, double* cost_out) {
  double best = 0.0, whole = 0.0;
  int bh = 0, bw = 0;
  const int khw = a->d.kh * a->d.kw, sms = sm_count();
  const double round_scale = (a->buckets > 32 ? 1.3 : 1.0) * (0.6 + 0.4 * khw / 9.0);
  // (extents that a number of tiles needs: a smaller one adds tiles or nothing)
  for (int nh = (a->Ho + 15) / 16, th = 17; th > 1; ++nh) {
    if ((a->Ho + nh - 1) / nh == th) continue;
    th = (a->Ho + nh - 1) / nh;
    for (int nw = (a->Wo + 31) / 32, tw = 33; tw > 1; ++nw) {
      if ((a->Wo + nw - 1) / nw == tw) continue;
      tw = (a->Wo + nw - 1) / nw;
      if (th * tw > 256) continue;
      TileArgs t = *a;
      set_tile(&t, th, tw);
      const size_t smem = tile_bytes<ListT>(&t);
      if (smem + kTileStatic > kSmemCtaMax || t.slots > 32767) continue;
      const bool pair = 2 * (smem + kTileStatic + 1024) <= kSmemPerSm;
      const int64_t tiles = (int64_t)t.tiles_h * t.tiles_w * t.d.N, resident = (int64_t)sms * (pair ? 2 : 1);
      const double waves = (double)((tiles + resident - 1) / resident);
      const int rounds = (t.TH * t.TW + kTileWarps - 1) / kTileWarps;
      const double values = (double)t.slots * 4 * t.quads, searches = rounds * round_scale;
      const bool paired = pair && tiles > sms;
      const double cost = waves * (8000.0 + 4.3 * values + 6200.0 * searches) * (paired ? 1.0 : 0.65);
      if (best == 0.0 || cost < best) {
        best = cost; bh = th; bw = tw;
        whole = waves * (paired ? 25000.0 + 2.7 * values + 8100.0 * searches : 20000.0 + 1.5 * values + 6000.0 * searches);
      }
    }
  }
  *cost_out = best;
  if (best == 0.0) return 0.0;
  set_tile(a, bh, bw);
  *smem_out = tile_bytes<ListT>(a);
  return (int64_t)a->tiles_h * a->tiles_w * a->d.N <= 0x7FFFFFFF ? whole : 0.0;
}

// budget: cycles that the tiles may take.
template <int KHW, int BPL, typename ListT>
cudaError_t launch_tile(TileArgs& a, double budget, cudaStream_t stream, bool* applicable) {
  a.buckets = 32 * BPL;
  a.octaves = BPL == 1 ? 8 : 12;
  size_t smem = 0;
  double cost;
  const double cycles = choose_tile<ListT>(&a, &smem, &cost);
  if (cycles == 0.0 || budget < cycles) return cudaSuccess;
  auto kern = binarize_patches_tile_kernel<KHW, BPL, ListT>;
  cudaError_t e = ensure_dynamic_smem(kern, smem);
  if (e != cudaSuccess) return e;
  *applicable = true;
  kern<<<(unsigned)(a.tiles_h * a.tiles_w * a.d.N), kTileThreads, smem, stream>>>(a);
  return cudaGetLastError();
}

// 32 buckets for short rows, 64 from 1536 values on.  (Post-ReLU rows of 1152 take 13 % longer with 64, N(0, 1) ones 9 % less;
// of 2304: 8 % longer and 15 % less.)  With a stride a tile stages many values for its patches, and tables of half the size may let
// two tiles share an SM, or make them larger: 64 x 48 x 56 x 56 7 x 7 stride 2 post-ReLU 798 -> 467 us, N(0, 1) 753 -> 683.  Not for a
// small gain, since N(0, 1) rows lose: 64 x 256 x 28 x 28 3 x 3 stride 2 (estimated gain 1.13) 213 -> 170, 207 -> 233.
template <int KHW, typename ListT>
cudaError_t launch_tile_buckets(TileArgs& a, bool always, cudaStream_t stream, bool* applicable) {
  // A layer of few patches is done sooner by a CTA per patch: about 15000 cycles and 5 + 0.012 n per patch, where this kernel
  // has 8000 to 35000 on top of its tiles (the kernel for marked patches, code that is not in the cache, longer hulls in longer
  // rows).  Measured, a CTA per patch and this, post-ReLU; N(0, 1): 2 x 64 x 28 x 28, 1568 patches of 576, 21 and 23 us; 21 and 28;
  // 4 x 128 x 28 x 28, 3136 of 1152, 45 and 34; 46 and 48; 24 x 128 x 28 x 28 with stride 2, 4704 of 1152, 61 and 50; 62 and 60;
  // 8 x 256 x 14 x 14, 1568 of 2304, 39 and 32; 38 and 44; 2 x 32 x 27 x 27 5 x 5, 1458 of 800, 23 and 26; 25 and 32;
  // 32 x 256 x 14 x 14 with stride 2, 1568 of 2304, 38 and 45; 38 and 46.
  const double by_patch = 15000.0 + (5.0 + 0.012 * a.n) * (double)a.d.N * a.Ho * a.Wo;
  const double set_up = (a.n < 1300 ? 5000.0 + 10.0 * a.n : 15000.0 + 2.4 * a.n) + (a.d.kh * a.d.kw > 9 ? 8000.0 : 0.0) +
                        (a.n >= 1536 && a.d.stride_h * a.d.stride_w > 1 ? 10000.0 : 0.0);
  const double budget = always ? 1e30 : by_patch - set_up;
  // Less than choose_tile estimates for any tile: the smallest calls are spared its trying all of them (1.6 us of 25 on the host for
  // 64 x 32 x 32 at batch 1).
  if (budget < 20000.0 + 6000.0 * (0.6 + 0.4 * a.d.kh * a.d.kw / 9.0)) return cudaSuccess;
  bool longer = a.n >= 1536;
  if (longer && a.d.stride_h * a.d.stride_w > 1) {
    double cost[2];
    for (int k = 0; k < 2; ++k) {
      TileArgs t = a;
      size_t smem;
      t.buckets = 32 << k;
      choose_tile<ListT>(&t, &smem, &cost[k]);
    }
    longer = cost[0] == 0.0 || (cost[1] > 0.0 && cost[1] <= (KHW == 9 ? 1.25 : 1.15) * cost[0]);
  }
  return longer ? launch_tile<KHW, 2, ListT>(a, budget, stream, applicable) : launch_tile<KHW, 1, ListT>(a, budget, stream, applicable);
}

}  // namespace

// Patches of 257..8192 values (up to 2048 channels, windows of up to 64 pixels) through the tile coder and the kernel that codes what it marked.
// *applicable = false (nothing launched) when the geometry has no tile that fits shared memory or, unless `always`, when a CTA
// per patch is expected to be faster.
cudaError_t launch_binarize_patches_tile(const dab_conv_desc& d, int32_t Ho, int32_t Wo, const float* x, int32_t* pK,
                                         float* pgamma, float* pdelta, uint32_t* pmask, int32_t ldp, uint32_t* pflags,
                                         bool always, cudaStream_t stream, bool* applicable) {
  TileArgs a;
  a.d = d; a.Ho = Ho; a.Wo = Wo; a.n = d.C * d.kh * d.kw;
  a.x = x; a.pK = pK; a.pgamma = pgamma; a.pdelta = pdelta; a.pflags = pflags; a.pmask = pmask; a.ldp = ldp;
  *applicable = false;
  if (a.n <= 256 || a.n > 8192 || d.C > 2048 || d.kh * d.kw > 64 || (int64_t)d.C * d.H * d.W > 0x7FFFFFFF) return cudaSuccess;
  a.quads = (d.C + 3) / 4;
  a.pitch = 4 * (a.quads + 1 - (a.quads & 1));  // an odd number of quadruples: neighbouring pixels in different banks
  a.word_pitch = ldp | 1;
  a.magic_ldp = (uint32_t)((0x100000000ull + (uint64_t)ldp - 1) / (uint64_t)ldp);
  cudaError_t e;
  if (d.kh == 3 && d.kw == 3)
    e = d.C <= 256 ? launch_tile_buckets<9, uint8_t>(a, always, stream, applicable) : launch_tile_buckets<9, uint16_t>(a, always, stream, applicable);
  else if (d.kh * d.kw <= 32) e = launch_tile_buckets<kAnyWindow, uint16_t>(a, always, stream, applicable);
  else e = launch_tile_buckets<kWideWindow, uint16_t>(a, always, stream, applicable);
  if (e != cudaSuccess || !*applicable) return e;
  return launch_binarize_patches_bucket(d, Ho, Wo, x, pK, pgamma, pdelta, pmask, ldp, pflags, /*marked_only=*/true, stream);
}

}  // namespace dab
