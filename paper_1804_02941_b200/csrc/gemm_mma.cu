// Tensor-core form of the AND-popcount contraction (Section 4.2: the four population counts of a pair of
// coded rows).  popc(e AND f) over a row of n bits is the dot product of the two rows written as 0/1 bytes,
// so each CTA expands mask words to bytes in shared memory and lets the fifth-generation tensor cores
// (tcgen05.mma, kind::i8, 32-bit integer accumulators in tensor memory) form a 128 x NT block of exact integer
// counts.  The bytes are single bits left where they stand in the mask word, mirrored on one side, so that an AND
// makes four of them and every product of two set bits is 128.  The four-term rescale then runs on the counts as they are read
// back from tensor memory, with the same arithmetic as the population-count kernel.
//
// Shared-memory operand layout (K-major, no swizzle): 8 rows x 16 bytes form one contiguous 128-byte core
// matrix; core matrices of consecutive 16-byte K chunks follow each other (leading byte offset 128) and
// groups of 8 rows are one whole stage row apart (stride byte offset = K chunks per stage x 128).  One mask
// word is 32 K bytes = two K chunks = the K extent of one kind::i8 instruction.
#include <algorithm>

#include "contraction.cuh"
#include "tc.cuh"

namespace dab {
namespace {

using namespace tc;

__device__ unsigned int g_mma_wait_timeouts;

constexpr int MMA_M = tc::kLanes;  // activation rows per CTA = lanes of tensor memory
constexpr int MMA_NMAX = 256;      // weight rows per CTA = columns of tensor memory

// One operand of the contraction: packed rows with their popcounts and the two reconstruction values
// (gamma, delta on the activation side; alpha, beta on the weight side).
struct Side {
  const uint32_t* mask;
  int32_t ld;
  const int32_t* K;
  const float* v1;  // value of the set bits
  const float* v0;  // value of the clear bits
  int64_t rows;
  bool weights;
  __device__ __forceinline__ RescaleSide rescaled(int64_t row, int n) const {
    const double a = (double)v1[DAB_IDX(row, rows)], b = (double)v0[DAB_IDX(row, rows)];
    const int k = K[DAB_IDX(row, rows)];
    return weights ? rescale_weight(a, b, k, n) : rescale_activation(a, b, k);
  }
  __device__ __forceinline__ bool gathered(int64_t row) const { return gathers(v1[DAB_IDX(row, rows)], v0[DAB_IDX(row, rows)]); }
};

// What the epilogue needs of one column-side row: its part of the rescale and of the output offset.
struct __align__(16) ColumnParams {
  RescaleSide r;
  int64_t off;
};

// Where activation row i and weight row j meet in the output: act_offset(i) + j * col_stride.
__device__ __forceinline__ int64_t act_offset(const GemmArgs& g, int64_t i) {
  return (i / g.map.inner) * g.map.outer_stride + (i % g.map.inner) * g.map.row_stride;
}

// Outputs of one lane-side row and up to 32 columns from column `first` (counted over the whole matrix) on.  v: their counts.
// gathered: every one of these rows and the lane's own gathers().
template <bool kLanesAreActivations, bool kPost>
__device__ __forceinline__ void store_columns(const GemmArgs& g, uint32_t (&v)[32], int left, const ColumnParams* col, int64_t first,
                                              int64_t gl, const RescaleSide& lane_side, int64_t off, bool gathered) {
  // this row's counts: element (gl, column) when the lanes are activation rows, (column, gl) otherwise
  const int64_t pblock = kLanesAreActivations ? gl * g.ldp + first : first * g.ldp + gl;
  const int64_t pstep = kLanesAreActivations ? 1 : g.ldp;
#pragma unroll
  for (int jj = 0; jj < 32; ++jj) v[jj] >>= kBitProductLog;
  if (!gathered) {  // rare: the counts wait in the outputs' own places for a loop that is not unrolled
#pragma unroll
    for (int jj = 0; jj < 32; ++jj) {
      if (jj >= left) break;
      const int64_t to = off + col[jj].off;
      if (DAB_IN_BOUNDS(to, g.c_extent)) g.C[to] = __int_as_float((int)v[jj]);
    }
    const int count = min(left, 32);
#pragma unroll 1
    for (int jj = 0; jj < count; ++jj) {
      const int64_t to = off + col[jj].off, at = first + jj;
      if (!DAB_IN_BOUNDS(to, g.c_extent)) continue;
      const int p11 = __float_as_int(g.C[to]);
      const float y = kLanesAreActivations ? rescale_any(g, p11, gl, at) : rescale_any(g, p11, at, gl);
      g.C[to] = kPost ? apply_post(g.post, y, (int)at, to, g.c_extent) : y;
      if (g.p11 && DAB_IN_BOUNDS(pblock + jj * pstep, (g.M - 1) * g.ldp + g.N)) g.p11[pblock + jj * pstep] = p11;
    }
    return;
  }
  if (!kPost && left >= 32 && !g.p11) {  // the usual case
    float* const row = g.C + off;
#pragma unroll
    for (int jj = 0; jj < 32; ++jj) {
      const ColumnParams cp = col[jj];
      const float y = kLanesAreActivations ? rescale((int)v[jj], cp.r, lane_side) : rescale((int)v[jj], lane_side, cp.r);
      if (DAB_IN_BOUNDS(off + cp.off, g.c_extent)) row[cp.off] = y;
    }
    return;
  }
#pragma unroll
  for (int jj = 0; jj < 32; ++jj) {
    if (jj >= left) break;
    const ColumnParams cp = col[jj];
    const float y = kLanesAreActivations ? rescale((int)v[jj], cp.r, lane_side) : rescale((int)v[jj], lane_side, cp.r);
    if (!kPost && DAB_IN_BOUNDS(off + cp.off, g.c_extent)) g.C[off + cp.off] = y;
    if (g.p11 && DAB_IN_BOUNDS(pblock + jj * pstep, (g.M - 1) * g.ldp + g.N)) g.p11[pblock + jj * pstep] = (int)v[jj];
    if (kPost) v[jj] = __float_as_uint(y);
  }
  if (kPost) {  // the layers behind a convolution, one after another over the 32 columns
    const int64_t step = g.map.col_stride, at = off + first * step;
    // Bound by the stores and the tensor to add.  The kind of a layer is looked at once for 32 columns, and columns beyond the last repeat
    // it, so that no branch stands between the loads: 16 are in flight.  One element at a time, with its kind: 32 x 64 x 56 x 56 -> 64 with
    // a normalisation layer and ReLU behind it 32 us, this 23; with a shortcut to add as well 79 and 30; 128 x 28 x 28 57 and 21.
    // In the form for 65 to 128 filters and rows below 32 words 128 bytes a thread are spilled, and it is ahead all the same: 16 x 64 x 56 x 56
    // -> 128, coder included, 141 and 129, 16 x 96 x 56 x 56 -> 96 with a shortcut 193 and 163.
    // Ordinary loads of the tensor to add: this thread may have stored it, in a kPostStore of the same chain.
    for (int k = 0; k < g.post.count; ++k) {
      const PostOp o = g.post.op[k];
      if (o.kind == kPostAffine) {
#pragma unroll
        for (int jj = 0; jj < 32; ++jj) v[jj] = __float_as_uint(post_affine(o, __uint_as_float(v[jj]), (int)first + min(jj, left - 1)));
      } else if (o.kind == kPostRelu) {
#pragma unroll
        for (int jj = 0; jj < 32; ++jj) v[jj] = __uint_as_float(v[jj]) > 0.0f ? v[jj] : 0u;
      } else if (o.kind == kPostAdd) {
        int64_t to = at;
#pragma unroll
        for (int j0 = 0; j0 < 32; j0 += 16) {
          float other[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            other[j] = o.a[DAB_IDX(to, g.c_extent)];
            if (j0 + j < left - 1) to += step;
          }
#pragma unroll
          for (int j = 0; j < 16; ++j) v[j0 + j] = __float_as_uint(__fadd_rn(__uint_as_float(v[j0 + j]), other[j]));
        }
      } else {
        int64_t to = at;
#pragma unroll
        for (int jj = 0; jj < 32; ++jj, to += step) {
          if (jj >= left) break;
          if (DAB_IN_BOUNDS(to, g.c_extent)) o.to[to] = __uint_as_float(v[jj]);
        }
      }
    }
    int64_t to = at;
#pragma unroll
    for (int jj = 0; jj < 32; ++jj, to += step) {
      if (jj >= left) break;
      if (DAB_IN_BOUNDS(to, g.c_extent)) g.C[to] = __uint_as_float(v[jj]);
    }
  }
}

template <bool kLanesAreActivations>
__device__ __forceinline__ void both_sides(const GemmArgs& g, Side& L, Side& S) {
  const Side act{g.A, g.lda, g.KA, g.gamma, g.delta, g.M, false}, wgt{g.B, g.ldb, g.KB, g.alpha, g.beta, g.N, true};
  L = kLanesAreActivations ? act : wgt;  // lane side
  S = kLanesAreActivations ? wgt : act;  // column side
}

template <bool kLanesAreActivations>
__device__ __forceinline__ ColumnParams column_params(const GemmArgs& g, const Side& S, int64_t j) {
  return {S.rescaled(j, g.n), kLanesAreActivations ? j * g.map.col_stride : act_offset(g, j)};
}

// The pieces one thread expands per stage: unit u covers row (u>>3)/KQ*8 + (u&7), 16-byte piece (u>>3)%KQ.
// Eight consecutive lanes hold the eight rows of one core matrix, so their 16-byte stores are one
// contiguous 128 bytes; their loads read KQ x 16 contiguous bytes per row.
//
// One CTA forms one 128 x NT tile over the whole row length, 4*KQ mask words per stage.  There is a single
// stage: a CTA alternates between expanding and waiting for the tensor cores, and the overlap comes from the
// several CTAs resident on an SM (expansion, the fp64 rescale and the tensor pipe use different units), which
// measured faster than two stages with fewer resident CTAs.
//
// kLanesAreActivations: the rows that ride the 128 lanes of tensor memory (and the threads of the epilogue)
// are activation rows, the columns weight rows: coalesced stores when the output is contiguous along the
// activation rows (NCHW).  Otherwise the roles are exchanged: coalesced for a row-major M x N output.
template <int THREADS, int KQ, int MIN_CTAS, int NT_MAX, bool kLanesAreActivations, bool kPost>
__global__ void __launch_bounds__(THREADS, MIN_CTAS) binary_gemm_mma_kernel(const GemmArgs g, const int tile_cols) {
  constexpr int KC = 8 * KQ;            // 16-byte K chunks per stage (two per mask word)
  constexpr uint32_t SBO = KC * 128;    // bytes between groups of 8 rows
  constexpr int kMaxUnits = ((MMA_M + NT_MAX) * KQ + THREADS - 1) / THREADS;  // NT <= NT_MAX in this shape
  extern __shared__ __align__(128) unsigned char dyn_mem[];  // [lane-side stage][column-side stage][ColumnParams]
  __shared__ __align__(8) uint64_t s_bar;
  __shared__ uint32_t s_tmem;

  Side L, S;
  both_sides<kLanesAreActivations>(g, L, S);

  const int tid = threadIdx.x, warp = (int)uniform(tid >> 5), lane = tid & 31;
  const int64_t i0 = (int64_t)blockIdx.x * MMA_M;
  const int64_t j0 = (int64_t)blockIdx.y * tile_cols;        // tile_cols: 64, 128 or 256 column-side rows per CTA
  const int nrows = (int)min((int64_t)tile_cols, S.rows - j0);  // column-side rows of this tile
  const int NT = (nrows + 15) & ~15;                            // instruction N
  uint32_t tmem_cols = 32;
  while ((int)tmem_cols < NT) tmem_cols <<= 1;

  const uint32_t a_bytes = MMA_M * KC * 16;
  const int ncap = (int)min((int64_t)tile_cols, (S.rows + 15) & ~(int64_t)15);  // widest tile of this launch
  const uint32_t mem0 = (smem_u32(dyn_mem) + 127u) & ~127u;
  unsigned char* const stage = dyn_mem + (mem0 - smem_u32(dyn_mem));
  ColumnParams* const s_col = reinterpret_cast<ColumnParams*>(stage + a_bytes + (uint32_t)ncap * KC * 16);
  const uint32_t bar = smem_u32(&s_bar);

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                 "r"(tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    mbar_init(bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  bool gathered = true;
  for (int j = tid; j < nrows; j += THREADS) {
    s_col[j] = column_params<kLanesAreActivations>(g, S, j0 + j);
    gathered = gathered && S.gathered(j0 + j);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  gathered = __syncthreads_and(gathered);  // of the tile's columns
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = uniform(s_tmem);
  const uint32_t idesc = instr_desc(NT);

  // units of this thread: lane-side pieces first, then column-side pieces
  const int l_units = MMA_M * KQ, units = l_units + NT * KQ;
  const int chunks = (g.words + 4 * KQ - 1) / (4 * KQ);
  const int real_words = (g.n + 31) >> 5;  // words beyond these hold no bits
  uint4 q[kMaxUnits];

  auto fetch = [&](int c) {  // the 16-byte pieces of chunk c, zero beyond the operands
    const int w0 = c * 4 * KQ;
#pragma unroll
    for (int t = 0; t < kMaxUnits; ++t) {
      const int u = tid + t * THREADS;
      q[t] = make_uint4(0, 0, 0, 0);
      if (u >= units) continue;
      const bool isL = u < l_units;
      const int v = isL ? u : u - l_units;
      const int row = ((v >> 3) / KQ) * 8 + (v & 7), piece = (v >> 3) % KQ;
      const int w = w0 + 4 * piece;
      if (w >= g.words) continue;
      if (isL) {
        if (i0 + row < L.rows)
          q[t] = *reinterpret_cast<const uint4*>(L.mask + DAB_IDX((i0 + row) * (int64_t)L.ld + w, L.rows * L.ld - 3));
      } else {
        if (row < nrows)
          q[t] = *reinterpret_cast<const uint4*>(S.mask + DAB_IDX((j0 + row) * (int64_t)S.ld + w, S.rows * S.ld - 3));
      }
    }
  };

  bool dead = false;
  uint32_t parity = 0;
  fetch(0);
  for (int c = 0; c < chunks; ++c) {
    if (c > 0) {  // the instructions that read the stage for the previous chunk have completed
      mbar_wait(bar, parity, dead, &g_mma_wait_timeouts);
      parity ^= 1;
    }
#pragma unroll
    for (int t = 0; t < kMaxUnits; ++t) {
      const int u = tid + t * THREADS;
      if (u >= units) continue;
      const bool isL = u < l_units;
      const int v = isL ? u : u - l_units;
      const int group = (v >> 3) / KQ, piece = (v >> 3) % KQ;
      if (c * 4 * KQ + 4 * piece >= g.words) continue;  // no instruction reads this part of the stage
      unsigned char* dst =
          stage + (isL ? 0u : a_bytes) + (uint32_t)group * SBO + (uint32_t)(8 * piece) * 128 + (v & 7) * 16;
      const uint32_t w[4] = {q[t].x, q[t].y, q[t].z, q[t].w};
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        if (isL) expand_word_bits<false>(w[m], dst + 256 * m);
        else expand_word_bits<true>(w[m], dst + 256 * m);
      }
    }
    if (c + 1 < chunks) fetch(c + 1);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic-proxy stores -> tensor-core reads
    __syncthreads();
    if (warp == 0 && elect_one()) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint64_t da = smem_desc(mem0, 128, SBO), db = smem_desc(mem0 + a_bytes, 128, SBO);
      const int kw = min(4 * KQ, real_words - c * 4 * KQ);
#pragma unroll
      for (int t = 0; t < 4 * KQ; ++t)  // one mask word = 32 K bytes = two K chunks per instruction
        if (t < kw) mma_i8(tmem, desc_at(da, t * 256), desc_at(db, t * 256), idesc, (c | t) != 0);
      mma_commit(bar);
    }
  }
  mbar_wait_last(bar, parity, dead, &g_mma_wait_timeouts);  // the last commit covers every instruction issued before it
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

  // Epilogue: thread = lane-side row (a warp reads the 32 lanes of its quarter), 32 columns at a time.
  {
    const int64_t gl = i0 + (warp & 3) * 32 + lane;
    const bool valid = gl < L.rows && !dead;
    RescaleSide lane_side{0.0, 0.0, 0.0};
    int64_t off = 0;
    if (valid) {
      lane_side = L.rescaled(gl, g.n);
      gathered = gathered && L.gathered(gl);
      off = kLanesAreActivations ? act_offset(g, gl) : gl * g.map.col_stride;
    }
    for (int cb = warp >> 2; cb * 32 < NT; cb += THREADS / 128) {
      uint32_t v[32];
      tmem_load_32(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(cb * 32), v);
      if (valid) store_columns<kLanesAreActivations, kPost>(g, v, nrows - cb * 32, s_col + cb * 32, j0 + cb * 32, gl, lane_side, off, gathered);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols) : "memory");
}

// The form for long rows: 128 x 128 outputs per CTA, two CTAs per SM.  The lane side never passes through shared memory: every
// thread writes four words of its row, expanded, into tensor memory, from where the tensor cores take their first operand.
// What is left there is the column side, written and read once: in the kernel above 24 KB pass through shared memory per 32 bits
// of 128 x 256 outputs, 192 cycles, where the products take 128; here it is 16 KB, 128 cycles.  Two stages of eight words, one
// barrier each, on which the workers only arrive: a warp of its own issues the products.  Bound by the load and shared-memory
// pipe (0.79 busy; tensor cores 0.46): a warp's load of 16 bytes per row takes it 32 cycles.  8192 x 8192 x 4608 bits: 346 us in
// the kernel above, 278 here (287 with a worker issuing; 369 with stages of four words and loads of 8 bytes; 310 with
// the words staged in shared memory by 16-byte asynchronous copies, 418 by bulk copies of 64 bytes per row).
constexpr int WIDE_WORKERS = 256, WIDE_THREADS = WIDE_WORKERS + 32, WIDE_COLS = 128, WIDE_WORDS = 8, WIDE_BUFFERS = 2;
constexpr uint32_t WIDE_SBO = 2 * WIDE_WORDS * 128, WIDE_STAGE = WIDE_COLS * WIDE_WORDS * 32;  // bytes
constexpr uint32_t WIDE_ACOLS = WIDE_WORDS * 8;            // columns of a lane-side stage: 4 bytes each; behind the accumulator
constexpr uint32_t WIDE_TMEM = WIDE_COLS + WIDE_BUFFERS * WIDE_ACOLS;
static_assert(WIDE_TMEM == 256, "two CTAs share the 512 columns");
constexpr size_t WIDE_BYTES = WIDE_BUFFERS * WIDE_STAGE + WIDE_COLS * sizeof(ColumnParams) + 128;

template <bool kLanesAreActivations, bool kPost>
__global__ void __launch_bounds__(WIDE_THREADS, 2) binary_gemm_wide_kernel(const GemmArgs g) {
  extern __shared__ __align__(128) unsigned char dyn_mem[];  // [two column-side stages][ColumnParams]
  __shared__ __align__(8) uint64_t s_bar[WIDE_BUFFERS];
  __shared__ uint32_t s_tmem;
  Side L, S;
  both_sides<kLanesAreActivations>(g, L, S);
  const int tid = threadIdx.x, warp = (int)uniform(tid >> 5), lane = tid & 31;
  const int64_t i0 = (int64_t)blockIdx.x * MMA_M, j0 = (int64_t)blockIdx.y * WIDE_COLS;
  const int nrows = (int)min((int64_t)WIDE_COLS, S.rows - j0);
  const uint32_t mem0 = (smem_u32(dyn_mem) + 127u) & ~127u;
  unsigned char* const stages = dyn_mem + (mem0 - smem_u32(dyn_mem));
  ColumnParams* const s_col = reinterpret_cast<ColumnParams*>(stages + WIDE_BUFFERS * WIDE_STAGE);
  const uint32_t bars = smem_u32(s_bar);

  if (warp == 0) tmem_alloc(smem_u32(&s_tmem), WIDE_TMEM);
  if (tid == 0) {
    for (int b = 0; b < WIDE_BUFFERS; ++b) mbar_init(bars + 8 * b, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  bool gathered = true;
  for (int j = tid; j < nrows; j += WIDE_THREADS) {
    s_col[j] = column_params<kLanesAreActivations>(g, S, j0 + j);
    gathered = gathered && S.gathered(j0 + j);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  gathered = __syncthreads_and(gathered);  // of the tile's columns
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = uniform(s_tmem);
  const uint32_t idesc = instr_desc((nrows + 15) & ~15);

  // lane side: thread = row (a warp reaches the 32 lanes of its quarter) and half of the stage's words
  const int quarter = warp & 3, half = warp >> 2;
  const int64_t gl = i0 + quarter * 32 + lane;
  const bool row_in = gl < L.rows;
  const int64_t row_at = (row_in ? gl : 0) * (int64_t)L.ld + 4 * half;
  const uint32_t lanes = (uint32_t)(quarter * 32) << 16;
  // column side: thread = row and two words; eight neighbouring threads write 128 contiguous bytes
  const int crow = (tid >> 4) * 8 + (tid & 7), piece = (tid >> 3) & 1;
  const bool col_in = crow < nrows;
  const int64_t col_at = (j0 + (col_in ? crow : 0)) * (int64_t)S.ld + 4 * piece;
  const int chunks = (g.words + WIDE_WORDS - 1) / WIDE_WORDS, real_words = (g.n + 31) >> 5;

  uint4 qa, qb;
  auto fetch = [&](int c) {
    const int w = c * WIDE_WORDS;
    qa = row_in && w + 4 * half < g.words ? __ldg(reinterpret_cast<const uint4*>(L.mask + DAB_IDX(row_at + w, L.rows * L.ld - 3))) : make_uint4(0, 0, 0, 0);
    qb = col_in && w + 4 * piece < g.words ? __ldg(reinterpret_cast<const uint4*>(S.mask + DAB_IDX(col_at + w, S.rows * S.ld - 3))) : make_uint4(0, 0, 0, 0);
  };
  bool dead = false;
  if (warp == WIDE_WORKERS / 32) {  // the last warp issues the products
    const uint64_t b_desc = smem_desc(mem0, 128, WIDE_SBO);
    for (int c = 0; c < chunks; ++c) {
      const uint32_t buffer = c % WIDE_BUFFERS;
      bar_sync(1 + buffer, WIDE_THREADS);
      if (elect_one()) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint64_t db = desc_at(b_desc, buffer * WIDE_STAGE);
        const uint32_t a_col = tmem + WIDE_COLS + buffer * WIDE_ACOLS;
        const int kw = min(WIDE_WORDS, real_words - c * WIDE_WORDS);
#pragma unroll
        for (int t = 0; t < WIDE_WORDS; ++t)
          if (t < kw) mma_i8_tmem(tmem, a_col + 8 * t, desc_at(db, t * 256), idesc, (c | t) != 0);
        mma_commit(bars + 8 * buffer);
      }
      __syncwarp();
    }
  } else {
    fetch(0);
    for (int c = 0; c < chunks; ++c) {
      const uint32_t buffer = c % WIDE_BUFFERS, bar = bars + 8 * buffer;
      // the products that read this buffer last are done
      if (c >= WIDE_BUFFERS) mbar_wait(bar, (uint32_t)(c / WIDE_BUFFERS - 1) & 1u, dead, &g_mma_wait_timeouts);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      uint32_t e[32];
      expand_bits(qa.x, e);
      expand_bits(qa.y, e + 8);
      expand_bits(qa.z, e + 16);
      expand_bits(qa.w, e + 24);
      tmem_store_32(tmem + lanes + WIDE_COLS + buffer * WIDE_ACOLS + half * 32, e);
      unsigned char* const dst = stages + buffer * WIDE_STAGE + (uint32_t)(crow >> 3) * WIDE_SBO + (uint32_t)(8 * piece) * 128 + (crow & 7) * 16;
      expand_word_bits<true>(qb.x, dst);
      expand_word_bits<true>(qb.y, dst + 256);
      expand_word_bits<true>(qb.z, dst + 512);
      expand_word_bits<true>(qb.w, dst + 768);
      if (c + 1 < chunks) fetch(c + 1);
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic-proxy stores -> tensor-core reads
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      stage_handover(1 + buffer, WIDE_THREADS, dead);  // (the buffer's next use waits for the products, which wait for this barrier)
    }
  }
  // the last commit covers every instruction issued before it
  mbar_wait_last(bars + 8 * ((chunks - 1) % WIDE_BUFFERS), (uint32_t)((chunks - 1) / WIDE_BUFFERS) & 1u, dead, &g_mma_wait_timeouts);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  {
    const bool valid = row_in && !dead && warp < WIDE_WORKERS / 32;
    RescaleSide lane_side{0.0, 0.0, 0.0};
    int64_t off = 0;
    if (valid) {
      lane_side = L.rescaled(gl, g.n);
      gathered = gathered && L.gathered(gl);
      off = kLanesAreActivations ? act_offset(g, gl) : gl * g.map.col_stride;
    }
#pragma unroll 1
    for (int cb = 2 * half; cb < 2 * half + 2 && cb * 32 < nrows && warp < WIDE_WORKERS / 32; ++cb) {
      uint32_t v[32];
      tmem_load_32(tmem + lanes + cb * 32, v);
      if (valid) store_columns<kLanesAreActivations, kPost>(g, v, nrows - cb * 32, s_col + cb * 32, j0 + cb * 32, gl, lane_side, off, gathered);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, WIDE_TMEM);
}

inline size_t dynamic_bytes(int kq, int ncap) {
  return (size_t)(MMA_M + ncap) * (8 * kq) * 16 + (size_t)ncap * sizeof(ColumnParams) + 128;
}

template <int THREADS, int KQ, int MIN_CTAS, int NT_MAX, bool kLanesAreActivations, bool kPost>
cudaError_t launch_shape(const GemmArgs& args, dim3 grid, int tile_cols, int ncap, cudaStream_t stream) {
  auto kernel = binary_gemm_mma_kernel<THREADS, KQ, MIN_CTAS, NT_MAX, kLanesAreActivations, kPost>;
  cudaError_t e = ensure_dynamic_smem(kernel, dynamic_bytes(KQ, NT_MAX));
  if (e != cudaSuccess) return e;
  kernel<<<grid, THREADS, dynamic_bytes(KQ, ncap), stream>>>(args, tile_cols);
  return cudaGetLastError();
}

template <bool kLanesAreActivations, bool kPost>
cudaError_t launch_side(const GemmArgs& args, cudaStream_t stream) {
  const int64_t lane_rows = kLanesAreActivations ? args.M : args.N, col_rows = kLanesAreActivations ? args.N : args.M;
  // Column tile: the full 256 columns of an accumulator unless that leaves most SMs without a CTA.
  const int64_t wide_x = (lane_rows + MMA_M - 1) / MMA_M, wide_y = (col_rows + WIDE_COLS - 1) / WIDE_COLS;
  // Rows of 32 words or more, tiles for every SM: measured, the other form against this one, 256 images of 128 x 28 x 28 (36 words)
  // 60 and 56 us, 256 x 14 x 14 (72) 47 and 37, 512 x 7 x 7 (144) 47 and 35; but 64 x 56 x 56 (18) 95 and 136, where the store
  // of the outputs is most of it and narrow tiles keep more CTAs in flight.
  if (args.words >= 32 && col_rows > 64 && wide_x * wide_y >= sm_count() && wide_x <= 0x7FFFFFFF && wide_y <= 65535) {
    auto kernel = binary_gemm_wide_kernel<kLanesAreActivations, kPost>;
    cudaError_t e = ensure_dynamic_smem(kernel, WIDE_BYTES);
    if (e != cudaSuccess) return e;
    kernel<<<dim3((unsigned)wide_x, (unsigned)wide_y), WIDE_THREADS, WIDE_BYTES, stream>>>(args);
    return cudaGetLastError();
  }
  const int64_t gx = (lane_rows + MMA_M - 1) / MMA_M;
  int tile_cols = MMA_NMAX;
  while (tile_cols > 64 && gx * ((col_rows + tile_cols - 1) / tile_cols) < 2 * sm_count()) tile_cols >>= 1;
  const int64_t gy = (col_rows + tile_cols - 1) / tile_cols;
  if (gx > 0x7FFFFFFF || gy > 65535) return cudaErrorInvalidValue;
  const dim3 grid((unsigned)gx, (unsigned)gy);
  const int ncap = (int)std::min<int64_t>(tile_cols, (col_rows + 15) & ~(int64_t)15);
  // CTA shape by tile width, from timings of the four layer shapes of the ResNet-18-like stack: narrow tiles
  // run best as many small CTAs (six of 128 threads per SM), wider ones as fewer CTAs of 256 threads with
  // longer stages (two per SM at the full 256 columns, where shared memory is the limit).
  if (ncap <= 64) return launch_shape<128, 1, 6, 64, kLanesAreActivations, kPost>(args, grid, tile_cols, ncap, stream);
  if (ncap <= 128 && args.words >= 64)  // long rows: eight words per stage halve the dependent stage rounds
    return launch_shape<256, 2, 3, 128, kLanesAreActivations, kPost>(args, grid, tile_cols, ncap, stream);
  if (ncap <= 128) return launch_shape<256, 1, 4, 128, kLanesAreActivations, kPost>(args, grid, tile_cols, ncap, stream);
  return launch_shape<256, 2, 2, MMA_NMAX, kLanesAreActivations, kPost>(args, grid, tile_cols, ncap, stream);
}

}  // namespace

cudaError_t launch_gemm_mma(const GemmArgs& args, bool lanes_along_rows, cudaStream_t stream) {
  if (args.words < 1 || args.M < 1 || args.N < 1) return cudaErrorInvalidValue;
  if (!lanes_along_rows) return launch_side<false, false>(args, stream);
  return args.post.count > 0 ? launch_side<true, true>(args, stream) : launch_side<true, false>(args, stream);
}

cudaError_t read_mma_wait_timeouts(unsigned int* count) {
  return cudaMemcpyFromSymbol(count, g_mma_wait_timeouts, sizeof(unsigned int));
}

}  // namespace dab
