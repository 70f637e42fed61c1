// Bucket-pruned search for the best split of one row (Section 4.1 / Algorithm 1), a CTA of T threads per row: rows of a
// matrix (binarize.cu), patches of layers with too few of them for the tile coder, and the patches that coder marks.
//
//   1. the row's values are staged in shared memory; the largest magnitude fixes the bucket grid: NB buckets on either
//      side of zero, 2^LOG2M of equal width in each of the top NB / 2^LOG2M octaves of magnitude.  A bucket is a range of
//      bit patterns, so membership is exact;
//   2. per bucket the count and the sum of the low bits of the patterns, by 32-bit shared-memory atomics.  Within a
//      bucket value = edge + low bits * ulp, so count and low sum give the bucket's sum of values exactly.  (What lies
//      below the resolved octaves is summed in fp64 by the threads themselves.);
//   3. a scan over the buckets gives split size and prefix sum at every bucket edge exactly; each bucket's splits are
//      bounded through the convexity of the objective (bucket_bound.cuh) and the buckets that can hold the maximum (the
//      hull, a few dozen values) are gathered, sorted and searched by the exact evaluator of rowcode.cuh;
//   4. the mask is a threshold compare over the staged values.
// Rows the search does not settle (a hull above the cap, as with few distinct values; a magnitude outside
// 2^-40..2^40) have the distinct values of their hull counted; where those are many, the row is sorted in place by the whole CTA and
// every split is evaluated.  Sorted before: 512 rows of 4608 values -1, 0, 1 152 -> 29 us, 512 of 16384 values 0, 1 650 -> 109 us.
//
// Bound by instruction issue (61 % of the slots, ALU pipe 49 %) and the barriers between the passes; 100 warp
// instructions per 32 values in rows of 4608.  It replaced a sorting network over the whole row with up to 32 warps per row, and a
// one-warp histogram for large matrices.  Measured, before -> this: 4096 x 9216 N(0, 1) 4.27 -> 0.128 ms (1.2 TB/s of
// values read), 8192 x 4608 Laplace 1.05 -> 0.22 ms, 4096 x 2304 0.22 -> 0.066 ms, 512 x 4608 0.114 -> 0.023 ms.
#pragma once

#include "bucket_bound.cuh"
#include "rowcode.cuh"

namespace dab {

// Shape of the coder by row length: T threads, PB of the 2 NB buckets each, 2^LOG2M per octave (12 octaves, 16 for the
// longest rows).  A bucket's low sum takes 23 - LOG2M bits per value: it stays below 2^32 for kMaxCount values.
template <int T> struct BucketShape;
template <> struct BucketShape<32> { static constexpr int kMaxN = 512, LOG2M = 3, PB = 6, kHull = 256, kMaxCount = 4096; };
template <> struct BucketShape<64> { static constexpr int kMaxN = 1024, LOG2M = 3, PB = 3, kHull = 256, kMaxCount = 4096; };
template <> struct BucketShape<128> { static constexpr int kMaxN = 4096, LOG2M = 4, PB = 3, kHull = 512, kMaxCount = 8192; };
template <> struct BucketShape<256> { static constexpr int kMaxN = DAB_MAX_N, LOG2M = 4, PB = 2, kHull = 1024, kMaxCount = 8192; };

// A warp per row where there are rows for some 20 warps on every SM: it has no barriers to wait at.  Measured, two warps and one:
// 512 rows of 300 values 7.8 and 9.8 us, 2048 11.6 and 11.7, 4096 21.3 and 16.9, 16384 74 and 57; 4096 of 512 20.7 and 18.1.
inline bool many_short_rows(int64_t rows, int n) { return n <= BucketShape<32>::kMaxN && rows >= (int64_t)20 * sm_count(); }

template <int T>
struct __align__(16) BlockShared {  // (a multiple of 16 bytes: the staged values behind it are read 16 bytes at a time)
  static constexpr int W = T / 32;
  double wsum[W], wtiny[W][2];
  double P_below, P_upto;
  long long wbestD[W];
  double wbestP[W];
  int wcnt[W], wtinyc[W][2];
  uint32_t wmax[W];
  float wbest[W];
  int wlo[W], whi[W], wbestS[W];
  uint32_t wbestT[W];
  int c_below, c_upto, fill, overflow;
  uint32_t hull_first, hull_last;  // keys; 0: the segments that can hold the best split are not known
  RowResult result;
};

// Words of shared memory behind the staged values: (count, low sum) per bucket, later the hull.
template <int T>
__host__ __device__ constexpr int bucket_words() { return 2 * BucketShape<T>::PB * T; }

template <int T>
inline size_t block_row_bytes(int n) {
  return sizeof(BlockShared<T>) + sizeof(uint32_t) * bucket_words<T>() + sizeof(float) * (size_t)((n + 31) & ~31);
}

// The hull, one warp: sort and exact evaluation.
template <int E>
__device__ __noinline__ RowResult bucket_sort_select(const uint32_t* keys, int m, int z, int n, int lane, const SplitBase base) {
  uint32_t r[E];
#pragma unroll
  for (int j = 0; j < E; ++j) {
    const int idx = j * 32 + lane;
    r[j] = idx < m ? keys[idx] : kPadKey;
  }
  group_sort<1, E>(r, lane, nullptr, 0);
  return group_select<1, E, false, true>(r, m, z, n, lane, nullptr, 0, nullptr, base);
}

// Every split of the row, by the whole CTA: the n staged values become keys, are sorted in place (bitonic network of
// upward compare-exchanges, partners beyond n left out) and evaluated exactly.  bs->result is valid for all threads.
template <int T>
__device__ __noinline__ void block_sort_code(uint32_t* keys, int n, BlockShared<T>* bs) {
  constexpr int W = T / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  __syncthreads();  // another warp may still read its sample of the values (block_distinct_code)
  for (int i = tid; i < n; i += T) keys[i] = order_key(__uint_as_float(keys[i]));
  int half = 1;  // half of the padded length
  while (2 * half < n) half <<= 1;
  for (int k = 2; k <= 2 * half; k <<= 1) {
    __syncthreads();
    const int kh = k >> 1;
    for (int idx = tid; idx < half; idx += T) {  // mirror stage
      const int o = idx & (kh - 1), lo = (idx - o) * 2 + o, hi = (idx - o) * 2 + k - 1 - o;
      if (hi < n) {
        const uint32_t a = keys[lo], b = keys[hi];
        if (a > b) { keys[lo] = b; keys[hi] = a; }
      }
    }
    for (int st = k >> 2; st >= 1; st >>= 1) {
      __syncthreads();
      for (int idx = tid; idx < half; idx += T) {
        const int o = idx & (st - 1), lo = (idx - o) * 2 + o, hi = lo + st;
        if (hi < n) {
          const uint32_t a = keys[lo], b = keys[hi];
          if (a > b) { keys[lo] = b; keys[hi] = a; }
        }
      }
    }
  }
  __syncthreads();
  const int per = (n + T - 1) / T, q0 = min(tid * per, n), q1 = min(q0 + per, n);
  double local = 0.0;
  for (int q = q0; q < q1; ++q) local = __dadd_rn(local, (double)key_value(keys[q]));
  double incl = local;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double u = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= o) incl = __dadd_rn(incl, u);
  }
  if (lane == 31) bs->wsum[warp] = incl;
  __syncthreads();
  double before = 0.0, total = 0.0;
#pragma unroll
  for (int w = 0; w < W; ++w) {
    if (w < warp) before = __dadd_rn(before, bs->wsum[w]);
    total = __dadd_rn(total, bs->wsum[w]);
  }
  double P = __dadd_rn(before, __dsub_rn(incl, local)), bD = -1.0, bP = 0.0;
  int bS = 0;
  uint32_t bT = 0;
  for (int q = q0; q < q1; ++q) {
    const uint32_t kc = keys[q];
    P = __dadd_rn(P, (double)key_value(kc));
    if (q + 1 < n && keys[q + 1] != kc) {
      const double D = objective(P, total, q + 1, n);
      if (D >= bD) { bD = D; bP = P; bS = q + 1; bT = keys[q + 1]; }
    }
  }
  long long d = __double_as_longlong(bD);  // D >= 0, or -1 for none: the bits order like integers
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const long long od = __shfl_xor_sync(0xFFFFFFFFu, d, o);
    const int os = __shfl_xor_sync(0xFFFFFFFFu, bS, o);
    const double oP = __shfl_xor_sync(0xFFFFFFFFu, bP, o);
    const uint32_t oT = __shfl_xor_sync(0xFFFFFFFFu, bT, o);
    if (od > d || (od == d && os > bS)) { d = od; bS = os; bP = oP; bT = oT; }
  }
  if (lane == 0) { bs->wbestD[warp] = d; bs->wbestS[warp] = bS; bs->wbestP[warp] = bP; bs->wbestT[warp] = bT; }
  __syncthreads();
  if (tid == 0) {
    int w = 0;
    for (int i = 1; i < W; ++i)
      if (bs->wbestD[i] > bs->wbestD[w] || (bs->wbestD[i] == bs->wbestD[w] && bs->wbestS[i] > bs->wbestS[w])) w = i;
    bs->result = bs->wbestS[w] ? finish_row(bs->wbestP[w], bs->wbestS[w], bs->wbestT[w], total, n)
                               : trivial_row(false, key_value(keys[0]));
  }
  __syncthreads();
}

__device__ __forceinline__ int hash_slot(uint32_t key, int slots) { return (int)__umulhi(key * 2654435761u, (uint32_t)slots); }

// The best of the splits between the `distinct` values of a hash table (keys, counts; list: the keys in no order), one warp.
// s_below, P_below: count and sum of the row below them; total: of the row, unless they are all of it (whole).  False: one value only.
template <int E>
__device__ __forceinline__ bool search_distinct(const uint32_t* keys, const uint32_t* counts, int slots, const uint32_t* list, int distinct,
                                                int s_below, double P_below, double total, bool whole, int n, int lane, RowResult* result) {
  constexpr unsigned kAll = 0xFFFFFFFFu;
  uint32_t key[E];
#pragma unroll
  for (int j = 0; j < E; ++j) key[j] = j * 32 + lane < distinct ? list[j * 32 + lane] : kPadKey;
  group_sort<1, E>(key, lane, nullptr, 0);
  int c[E], csum = 0;
  double S[E], ssum = 0.0;
#pragma unroll
  for (int j = 0; j < E; ++j) {
    int count = 0;
    if (key[j] != kPadKey) {
      int h = hash_slot(key[j], slots);
      while (keys[h] != key[j]) h = h + 1 == slots ? 0 : h + 1;  // (it is there)
      count = (int)counts[h];
      ssum = __dadd_rn(ssum, __dmul_rn((double)count, (double)key_value(key[j])));
    }
    csum += count;
    c[j] = csum;
    S[j] = ssum;
  }
  int cincl = csum;
  double sincl = ssum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(kAll, cincl, o);
    const double w = __shfl_up_sync(kAll, sincl, o);
    if (lane >= o) { cincl += u; sincl = __dadd_rn(sincl, w); }
  }
  double before = __shfl_up_sync(kAll, sincl, 1);
  if (lane == 0) before = 0.0;
  if (whole) total = __shfl_sync(kAll, sincl, 31);
  const uint32_t next_first = __shfl_down_sync(kAll, key[0], 1);
  double bD = -1.0, bP = 0.0;
  int bS = 0;
  uint32_t bT = 0u;
#pragma unroll
  for (int j = 0; j < E; ++j) {
    const uint32_t next = j + 1 < E ? key[j + 1 < E ? j + 1 : 0] : (lane == 31 ? kPadKey : next_first);
    if (key[j] == kPadKey || next == kPadKey) continue;
    const int split = s_below + cincl - csum + c[j];
    const double P = __dadd_rn(P_below, __dadd_rn(before, S[j])), D = objective(P, total, split, n);
    if (D >= bD) { bD = D; bP = P; bS = split; bT = next; }
  }
  long long d = __double_as_longlong(bD);  // D >= 0, or -1 for none: the bits order like integers
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const long long od = __shfl_xor_sync(kAll, d, o);
    const int os = __shfl_xor_sync(kAll, bS, o);
    const double oP = __shfl_xor_sync(kAll, bP, o);
    const uint32_t oT = __shfl_xor_sync(kAll, bT, o);
    if (od > d || (od == d && os > bS)) { d = od; bS = os; bP = oP; bT = oT; }
  }
  if (lane == 0) {
    if (bS) *result = finish_row(bP, bS, bT, total, n);
    else if (whole) *result = trivial_row(false, key_value(key[0]));
  }
  return bS > 0 || whole;
}

// Rows of few distinct values: those of the staged values whose keys lie in [first, last], and the zeros if `zeros`, are counted in a
// hash table, its keys sorted by one warp, and the splits between them evaluated exactly.  False, in every thread: too many
// distinct values, or a single one that is not the whole row.  Otherwise bs->result is valid for all threads.
template <int T>
__device__ __noinline__ bool block_distinct_code(const float* vals, int n, uint32_t* table, uint32_t first, uint32_t last, bool zeros,
                                                 int s_below, double P_below, double total, bool whole, BlockShared<T>* bs) {
  constexpr int CAP = bucket_words<T>() / 4, SLOTS = (bucket_words<T>() - CAP) / 2;  // 96, 192 and 256 distinct values
  constexpr unsigned kAll = 0xFFFFFFFFu;
  uint32_t* const keys = table;
  uint32_t* const counts = table + SLOTS;
  uint32_t* const list = table + 2 * SLOTS;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  {  // a sample of 32, the same in every warp: hardly a value twice among it, and there are too many of them
    const uint32_t key = order_key(vals[(int)((int64_t)n * lane >> 5)]);
    const bool in = key != kZeroKey && key >= first && key <= last;
    const unsigned peers = __match_any_sync(kAll, in ? key : kPadKey);
    const int count = __popc(__ballot_sync(kAll, in)), distinct = __popc(__ballot_sync(kAll, in && (peers & ((1u << lane) - 1u)) == 0u));
    if (count >= 4 && 4 * distinct > 3 * count) return false;
  }
  for (int i = tid; i < SLOTS; i += T) { keys[i] = kPadKey; counts[i] = 0u; }
  if (tid == 0) bs->fill = bs->overflow = 0;
  __syncthreads();
  for (int base = warp * 32; base < n; base += T) {
    const int i = base + lane;
    const uint32_t key = i < n ? order_key(vals[i]) : kPadKey;
    const bool in = i < n && (key == kZeroKey ? zeros : key >= first && key <= last);
    if (!__any_sync(kAll, in)) continue;
    if (__any_sync(kAll, *static_cast<volatile int*>(&bs->overflow))) break;
    const unsigned peers = __match_any_sync(kAll, in ? key : kPadKey);
    if (in && (peers & ((1u << lane) - 1u)) == 0u) {  // one lane per value
      int h = hash_slot(key, SLOTS);
      for (int probe = 0;; ++probe, h = h + 1 == SLOTS ? 0 : h + 1) {
        uint32_t old = probe < SLOTS ? atomicCAS(keys + h, kPadKey, key) : key;
        if (old == kPadKey) {
          const int at = atomicAdd(&bs->fill, 1);
          if (at < CAP) list[at] = key;
          old = key;
        }
        if (old == key) break;
      }
      atomicAdd(counts + h, (uint32_t)__popc(peers));
      if (*static_cast<volatile int*>(&bs->fill) > CAP) bs->overflow = 1;  // (before the table is full: CAP + T / 32 values at most)
    }
  }
  __syncthreads();
  if (bs->overflow || bs->fill > CAP) return false;
  if (warp == 0) {
    const int distinct = bs->fill;
    const bool ok = distinct <= 32 ? search_distinct<1>(keys, counts, SLOTS, list, distinct, s_below, P_below, total, whole, n, lane, &bs->result)
                                   : search_distinct<8>(keys, counts, SLOTS, list, distinct, s_below, P_below, total, whole, n, lane, &bs->result);
    if (lane == 0 && !ok) bs->overflow = 1;
  }
  __syncthreads();
  return !bs->overflow;
}

__device__ __forceinline__ uint32_t magnitude_bits(float v) { return __float_as_uint(v) & 0x7FFFFFFFu; }

// Where a coded row goes.
struct RowOut {
  int32_t* K;
  float* alpha;
  float* beta;
  uint32_t* flags;  // may be null
  uint32_t* mask;
  int32_t ld;
  int64_t rows;
};

// A row of values in global memory, as block_code_row takes it.  stage<T>: the CTA copies the row to `vals`, padded with
// zeros (which no pass counts) to `quads` quadruples, and each thread returns the largest magnitude bits it saw; restage<T>:
// the same values once more; finish: called by every thread when the row's code is known, with the row still staged.
struct MatrixRow {
  const float* v;
  int n;
  bool aligned;  // 16-byte loads reach every value
  __device__ __forceinline__ MatrixRow(const float* row, int n_) : v(row), n(n_), aligned((n_ & 3) == 0 && (reinterpret_cast<uintptr_t>(row) & 15) == 0) {}
  template <int T>
  __device__ __forceinline__ uint32_t stage(float* vals, int quads, BlockShared<T>*) const {
    uint32_t top = 0u;
    if (aligned) {
#pragma unroll 4
      for (int q = threadIdx.x; q < quads; q += T) {
        const float4 x = 4 * q < n ? __ldg(reinterpret_cast<const float4*>(v + DAB_IDX(4 * q, n - 3))) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        *reinterpret_cast<float4*>(vals + 4 * q) = x;
        top = max(max(top, max(magnitude_bits(x.x), magnitude_bits(x.y))), max(magnitude_bits(x.z), magnitude_bits(x.w)));
      }
    } else {
#pragma unroll 8
      for (int i = threadIdx.x; i < 4 * quads; i += T) {
        const float x = i < n ? __ldg(v + DAB_IDX(i, n)) : 0.0f;
        vals[i] = x;
        top = max(top, magnitude_bits(x));
      }
    }
    return top;
  }
  template <int T>
  __device__ __forceinline__ void restage(float* vals, int quads) const { stage<T>(vals, quads, nullptr); }
  template <int T>
  __device__ __forceinline__ void finish(const float*, const RowResult&) const {}
};

// Codes row `row`.  smem: block_row_bytes<T>(n) bytes.  All threads of the CTA call it; the shared memory is free again
// when it has returned in all threads (a barrier is the caller's).
template <int T, typename Source>
__device__ __forceinline__ void block_code_row(const Source& source, int n, unsigned char* smem, const RowOut& out, int64_t row) {
  constexpr int W = T / 32, PB = BucketShape<T>::PB, NB = PB * T / 2, SHIFT = 23 - BucketShape<T>::LOG2M;
  BlockShared<T>* const bs = reinterpret_cast<BlockShared<T>*>(smem);
  uint32_t* const hist = reinterpret_cast<uint32_t*>(bs + 1);  // [2 NB] counts, then [2 NB] low sums
  float* const vals = reinterpret_cast<float*>(hist + bucket_words<T>());
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  // ---- stage the row; largest magnitude ----
#pragma unroll
  for (int j = 0; j < 2 * PB; ++j) hist[j * T + tid] = 0u;
  if (tid == 0) { bs->fill = bs->overflow = 0; bs->hull_last = 0u; }
  const int words = (n + 31) >> 5, quads = 8 * words;
  uint32_t top = source.template stage<T>(vals, quads, bs);
  top = __reduce_max_sync(0xFFFFFFFFu, top);
  if (lane == 0) bs->wmax[warp] = top;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < W; ++w) top = max(top, bs->wmax[w]);

  RowResult res;
  const int e = (int)(top >> 23) - 127;
  if (top >= 0x7F800000u || top == 0u) {
    res = trivial_row(top != 0u, 0.0f);
  } else {
    bool retry = e < -40 || e > 40;
    const int base = (int)(top >> SHIFT) - (NB - 1);
    int m_sub = 0, z_in = 0, s_below = 0;
    double T_row = 0.0;
    if (!retry) {
      // ---- count and low sum per bucket ----
      double tiny[2] = {0.0, 0.0};
      int tinyc[2] = {0, 0};
      auto count = [&](float v) {  // whether v lies below the resolved octaves
        const uint32_t bits = magnitude_bits(v);
        const int b = (int)(bits >> SHIFT) - base;
        if (b > 0) {
          uint32_t* const slot = hist + NB + (b ^ (__float_as_int(v) >> 31));  // NB + b, or NB - 1 - b for a negative value
          atomicAdd(slot, 1u);
          atomicAdd(slot + 2 * NB, bits & ((1u << SHIFT) - 1u));
        }
        return b <= 0 && bits != 0u;
      };
      auto count_tiny = [&](float v, bool in) {
        const bool negative = v < 0.0f;
        tiny[0] = __dadd_rn(tiny[0], in && negative ? (double)v : 0.0);
        tiny[1] = __dadd_rn(tiny[1], in && !negative ? (double)v : 0.0);
        tinyc[0] += in && negative;
        tinyc[1] += in && !negative;
      };
#pragma unroll 2
      for (int q = tid; q < quads; q += T) {
        const float4 v = *reinterpret_cast<const float4*>(vals + 4 * q);
        const bool t0 = count(v.x), t1 = count(v.y), t2 = count(v.z), t3 = count(v.w);
        if (t0 || t1 || t2 || t3) {  // rare
          count_tiny(v.x, t0);
          count_tiny(v.y, t1);
          count_tiny(v.z, t2);
          count_tiny(v.w, t3);
        }
      }
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        const int c = __reduce_add_sync(0xFFFFFFFFu, tinyc[s]);
        double t = tiny[s];
        if (c)  // the same for all lanes
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) t = __dadd_rn(t, __shfl_xor_sync(0xFFFFFFFFu, t, o));
        if (lane == 0) { bs->wtinyc[warp][s] = c; bs->wtiny[warp][s] = t; }
      }
      __syncthreads();
      // ---- scan: this thread's buckets are tid * PB + j ----
      int cc[PB];       // counts, then inclusive cumulative counts
      double cs[PB];    // sums, likewise
      int csum = 0;
      double ssum = 0.0;
#pragma unroll
      for (int j = 0; j < PB; ++j) {
        const int b = tid * PB + j, i = b < NB ? NB - 1 - b : b - NB;
        int c = (int)hist[b];
        const uint32_t lo = (uint32_t)(i + base) << SHIFT;
        const double ulp = (double)__uint_as_float((lo & 0x7F800000u) - (23u << 23));
        double s = __dadd_rn(__dmul_rn((double)c, (double)__uint_as_float(lo)), __dmul_rn((double)hist[2 * NB + b], ulp));
        if (b < NB) s = -s;
        if (i == 0) {
          c = 0;
          s = 0.0;
#pragma unroll
          for (int w = 0; w < W; ++w) {
            c += bs->wtinyc[w][b < NB ? 0 : 1];
            s = __dadd_rn(s, bs->wtiny[w][b < NB ? 0 : 1]);
          }
        }
        if (BucketShape<T>::kMaxN > BucketShape<T>::kMaxCount && c > BucketShape<T>::kMaxCount && i > 0) bs->overflow = 1;
        csum += c;
        ssum = __dadd_rn(ssum, s);
        cc[j] = csum;
        cs[j] = ssum;
      }
      int cincl = csum;
      double sincl = ssum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xFFFFFFFFu, cincl, o);
        const double w = __shfl_up_sync(0xFFFFFFFFu, sincl, o);
        if (lane >= o) { cincl += u; sincl = __dadd_rn(sincl, w); }
      }
      if (lane == 31) { bs->wcnt[warp] = cincl; bs->wsum[warp] = sincl; }
      double sbefore = __shfl_up_sync(0xFFFFFFFFu, sincl, 1);
      int cbefore = __shfl_up_sync(0xFFFFFFFFu, cincl, 1);
      if (lane == 0) { cbefore = 0; sbefore = 0.0; }
      __syncthreads();
      int m = 0, neg = 0, cw = 0;
      double Pneg = 0.0, sw = 0.0;
#pragma unroll
      for (int w = 0; w < W; ++w) {
        if (w == warp) { cw = m; sw = T_row; }
        m += bs->wcnt[w];
        T_row = __dadd_rn(T_row, bs->wsum[w]);
        if (w == W / 2 - 1) { neg = m; Pneg = T_row; }  // the first half of the threads holds the negative buckets
      }
      if (W == 1) {
        neg = __shfl_sync(0xFFFFFFFFu, cincl, 15);
        Pneg = __shfl_sync(0xFFFFFFFFu, sincl, 15);
      }
      cbefore += cw;
      sbefore = __dadd_rn(sw, sbefore);
      const int z = n - m;
      const double nd = (double)n;
      // ---- objective at the edges, bound inside each bucket ----
      const bool positive = tid >= T / 2;
      const int zoff = positive ? z : 0;  // the zeros precede the positive buckets
      const float dz0 = z > 0 && neg > 0 ? objective_bound((double)neg, Pneg, T_row, nd) : -1.0f;
      const float dz1 = z > 0 && neg + z < n ? objective_bound((double)(neg + z), Pneg, T_row, nd) : -1.0f;
      float best = fmaxf(dz0, dz1), bound[PB];
      {
        const int s0 = cbefore + zoff;
        float d0 = s0 > 0 && s0 < n ? objective_bound((double)s0, sbefore, T_row, nd) : -1.0f;
        best = fmaxf(best, d0);
        int pc = cbefore;
        double ps = sbefore;
#pragma unroll
        for (int j = 0; j < PB; ++j) {
          const int b = tid * PB + j;
          cc[j] += cbefore;
          cs[j] = __dadd_rn(cs[j], sbefore);
          const int c = cc[j] - pc, s1 = cc[j] + zoff;
          float d1 = d0, dk = -1.0f;
          if (c > 0) d1 = s1 > 0 && s1 < n ? objective_bound((double)s1, cs[j], T_row, nd) : -1.0f;
          if (c >= 2) {
            const int i = positive ? b - NB : NB - 1 - b;
            dk = bucket_corner_bound<SHIFT>(i, i + base, !positive, pc + zoff, c, ps, __dsub_rn(cs[j], ps), T_row, nd);
          }
          best = fmaxf(best, d1);
          bound[j] = c > 0 ? fmaxf(fmaxf(d0, d1), dk) : -2.0f;
          d0 = d1;
          pc = cc[j];
          ps = cs[j];
        }
      }
      const uint32_t wb = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(fmaxf(best, 0.0f)));
      if (lane == 0) bs->wbest[warp] = __uint_as_float(wb);
      __syncthreads();
      best = 0.0f;
#pragma unroll
      for (int w = 0; w < W; ++w) best = fmaxf(best, bs->wbest[w]);
      // ---- hull, in segments: buckets below NB keep their index, the zeros are NB, the rest + 1 ----
      const float need = best * prune_margin;
      int seg_lo = 1 << 20, seg_hi = -1;
#pragma unroll
      for (int j = 0; j < PB; ++j) {
        if (bound[j] >= need) {
          const int seg = tid * PB + j + (positive ? 1 : 0);
          seg_lo = min(seg_lo, seg);
          seg_hi = max(seg_hi, seg);
        }
      }
      if (z > 0 && fmaxf(dz0, dz1) >= need) { seg_lo = min(seg_lo, NB); seg_hi = max(seg_hi, NB); }
      seg_lo = __reduce_min_sync(0xFFFFFFFFu, seg_lo);
      seg_hi = __reduce_max_sync(0xFFFFFFFFu, seg_hi);
      if (lane == 0) { bs->wlo[warp] = seg_lo; bs->whi[warp] = seg_hi; }
      __syncthreads();
#pragma unroll
      for (int w = 0; w < W; ++w) { seg_lo = min(seg_lo, bs->wlo[w]); seg_hi = max(seg_hi, bs->whi[w]); }
      const int b_lo = seg_lo > NB ? seg_lo - 1 : seg_lo, b_hi = seg_hi >= NB ? seg_hi - 1 : seg_hi;
      retry = bs->overflow || !(best > 1e-30f) || seg_hi < 0 || b_lo > b_hi || b_lo < 0 || b_hi >= 2 * NB;
      if (!retry) {
        z_in = (z > 0 && seg_lo <= NB && NB <= seg_hi) ? z : 0;
        {
          int pc = cbefore;
          double ps = sbefore;
#pragma unroll
          for (int j = 0; j < PB; ++j) {
            if (tid * PB + j == b_lo) { bs->c_below = pc; bs->P_below = ps; }
            if (tid * PB + j == b_hi) { bs->c_upto = cc[j]; bs->P_upto = cs[j]; }
            pc = cc[j];
            ps = cs[j];
          }
        }
        // ---- gather the hull: values from the smallest of bucket b_lo to the largest of bucket b_hi, zeros left out ----
        const uint32_t first = bucket_first_key<SHIFT>(b_lo, NB, base), last = bucket_last_key<SHIFT>(b_hi, NB, base);
        if (tid == 0) { bs->hull_first = first; bs->hull_last = last; }
        const float vfirst = key_value(first), vlast = key_value(last);
        const unsigned lt = (1u << lane) - 1u;
#pragma unroll 2
        for (int q0 = warp * 32; q0 < quads; q0 += T) {
          const int q = q0 + lane;
          const float4 v = q < quads ? *reinterpret_cast<const float4*>(vals + 4 * q) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
          const float x[4] = {v.x, v.y, v.z, v.w};
          bool in[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) in[j] = x[j] >= vfirst && x[j] <= vlast && x[j] != 0.0f;
          if (__any_sync(0xFFFFFFFFu, in[0] || in[1] || in[2] || in[3])) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const unsigned bal = __ballot_sync(0xFFFFFFFFu, in[j]);
              if (bal) {
                int at = 0;
                if (lane == 0) at = atomicAdd(&bs->fill, __popc(bal));
                at = __shfl_sync(0xFFFFFFFFu, at, 0) + __popc(bal & lt);
                if (in[j] && at < BucketShape<T>::kHull) hist[at] = order_key(x[j]);
              }
            }
          }
        }
        __syncthreads();
        m_sub = bs->c_upto - bs->c_below;
        s_below = bs->c_below + (seg_lo > NB ? z : 0);
        // (a constant row is one bucket; a count that differs cannot happen)
        retry = m_sub < 1 || m_sub > BucketShape<T>::kHull || m_sub != bs->fill || (z == 0 && m_sub == n);
      }
    }
    if (!retry) {
      if (warp == 0) {
        const SplitBase sb{s_below, bs->P_below, __dsub_rn(T_row, bs->P_upto)};
        RowResult r;
        if (m_sub <= 32) r = bucket_sort_select<1>(hist, m_sub, z_in, n, lane, sb);
        else if (m_sub <= 64) r = bucket_sort_select<2>(hist, m_sub, z_in, n, lane, sb);
        else if (m_sub <= 128) r = bucket_sort_select<4>(hist, m_sub, z_in, n, lane, sb);
        else if (m_sub <= 256) r = bucket_sort_select<8>(hist, m_sub, z_in, n, lane, sb);
        else if (m_sub <= 512) r = bucket_sort_select<16>(hist, m_sub, z_in, n, lane, sb);
        else r = bucket_sort_select<32>(hist, m_sub, z_in, n, lane, sb);
        if (lane == 0) bs->result = r;
      }
      __syncthreads();
      retry = bs->result.tkey == kPadKey;  // a split at the hull's outer edge won: not certified
    }
    if (retry) {
      const uint32_t first = bs->hull_first, last = bs->hull_last;
      const bool hull = last != 0u;
      const double P_below = hull ? bs->P_below : 0.0;
      __syncthreads();
      if (!block_distinct_code<T>(vals, n, hist, hull ? first : 0u, hull ? last : kPadKey, !hull || z_in > 0, s_below, P_below, T_row,
                                  !hull || m_sub + z_in == n, bs)) {
        block_sort_code<T>(reinterpret_cast<uint32_t*>(vals), n, bs);
        source.template restage<T>(vals, quads);  // for the mask
        __syncthreads();
      }
    }
    res = bs->result;
  }

  // ---- outputs ----
  if (tid == 0 && DAB_IN_BOUNDS(row, out.rows)) {
    out.K[row] = res.K;
    out.alpha[row] = res.alpha;
    out.beta[row] = res.beta;
    if (out.flags) out.flags[row] = res.flags;
  }
  uint32_t* const mrow = out.mask + row * (int64_t)out.ld;
  const int per = (words + W - 1) / W, wend = min(words, (warp + 1) * per);
  const bool flip = res.mode == 1, none = res.mode == 2;
  const float tv = key_value(res.tkey);
  const uint32_t last = n & 31 ? (1u << (n & 31)) - 1u : 0xFFFFFFFFu;  // the bits of the last word that exist
  for (int wb = warp * per; wb < wend; wb += 32) {  // this warp's words, 32 at a time: word wb + j ends up in lane j
    const int cnt = min(32, wend - wb);
    uint32_t mine = 0u;
#pragma unroll 4
    for (int j = 0; j < cnt; ++j) {
      const uint32_t word = __ballot_sync(0xFFFFFFFFu, vals[(wb + j) * 32 + lane] >= tv);
      if (lane == j) mine = word;
    }
    if (flip) mine = ~mine;
    if (wb + lane == words - 1) mine &= last;
    if (lane < cnt && DAB_IN_BOUNDS(row * out.ld + wb + lane, out.rows * out.ld)) mrow[wb + lane] = none ? 0u : mine;
  }
  for (int w = words + tid; w < out.ld; w += T)
    if (DAB_IN_BOUNDS(row * out.ld + w, out.rows * out.ld)) mrow[w] = 0u;
  source.template finish<T>(vals, res);
}

}  // namespace dab
