// dab_binary_gemm: AND-popcount contraction of packed rows with the four-term rescale fused in.
// Integer work (AND, carry-save adders, POPC, IADD); the only large byte stream is the output store.
//
// A launch of few tiles splits the row length over the CTAs of a cluster: each counts its share of the words, then
// finishes its share of the tile's outputs from the counts of all of them (distributed shared memory).  Bound by the chain
// of slices and by POPC (16 a clock and SM): 1 x 512 outputs of 392 words took 65 us on 8 CTAs of 64 x 64 outputs and
// 7 on 64 of 16 x 64; the five such layers of a sketch classified alone 132 us, now 55.
#include <cooperative_groups.h>

#include <algorithm>

#include "contraction.cuh"

namespace dab {

constexpr int BN = 64;           // tile of outputs: 16 TM x 64
constexpr int BK = 48;           // words per staged slice (a multiple of 3 for the carry-save groups and of 4)
constexpr int TN = 4;            // outputs per thread: TM x 4
constexpr int GEMM_THREADS = 256;
constexpr int kMaxSplit = 8;     // CTAs per cluster

// Population counts issue at a quarter of the rate of logic operations, so three AND-ed words are first
// compressed by a carry-save adder (two 3-input logic operations) into a sum word and a carry word:
// popc(x0) + popc(x1) + popc(x2) = popc(sum) + 2 popc(carry).  Two counts instead of three.
__device__ __forceinline__ void csa(uint32_t x0, uint32_t x1, uint32_t x2, uint32_t& sum, uint32_t& carry) {
  asm("lop3.b32 %0, %1, %2, %3, 0x96;" : "=r"(sum) : "r"(x0), "r"(x1), "r"(x2));    // x0 ^ x1 ^ x2
  asm("lop3.b32 %0, %1, %2, %3, 0xE8;" : "=r"(carry) : "r"(x0), "r"(x1), "r"(x2));  // majority
}

// kLanesAlongRows: consecutive threads own consecutive activation rows i (coalesced when the output is
// contiguous along i, as in NCHW); otherwise consecutive threads own consecutive weight columns j.
template <bool kLanesAlongRows, int TM, bool kSplit>
__global__ void __launch_bounds__(GEMM_THREADS) binary_gemm_kernel(const GemmArgs g, const int share) {
  constexpr int BM = 16 * TM, ALD = BM + 4, BLD = BN + 4;  // padded smem rows, keep 16-byte alignment
  __shared__ __align__(16) uint32_t operands[BK * (ALD + BLD)];
  uint32_t (*const As)[ALD] = reinterpret_cast<uint32_t (*)[ALD]>(operands);
  uint32_t (*const Bs)[BLD] = reinterpret_cast<uint32_t (*)[BLD]>(operands + BK * ALD);

  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  const int a_t = kLanesAlongRows ? tx : ty;  // which group of TM activation rows
  const int b_t = kLanesAlongRows ? ty : tx;  // which group of TN weight rows
  const int64_t i0 = (int64_t)blockIdx.x * BM;
  const int64_t j0 = (int64_t)blockIdx.y * BN;

  int ones[TM][TN], twos[TM][TN];  // p11 = ones + 2 * twos
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) ones[i][j] = twos[i][j] = 0;

  // words of this CTA: all of them, or a cluster member's share (a multiple of 4)
  const int k_begin = kSplit ? (int)blockIdx.z * share : 0, k_end = kSplit ? min(g.words, k_begin + share) : g.words;
  for (int k0 = k_begin; k0 < k_end; k0 += BK) {
    // stage BK words of the rows of each operand, transposed; words beyond the share become 0
#pragma unroll
    for (int rep = 0; rep < ((BM + BN) * BK / 4 + GEMM_THREADS - 1) / GEMM_THREADS; ++rep) {
      const int t = tid + rep * GEMM_THREADS;
      if (t >= (BM + BN) * BK / 4) break;
      const int r = t / (BK / 4), q = (t % (BK / 4)) * 4;
      uint4 v = make_uint4(0, 0, 0, 0);
      if (r < BM) {
        if (k0 + q < k_end && i0 + r < g.M)
          v = *reinterpret_cast<const uint4*>(g.A + DAB_IDX((i0 + r) * (int64_t)g.lda + k0 + q, g.M * g.lda - 3));
        As[q + 0][r] = v.x; As[q + 1][r] = v.y; As[q + 2][r] = v.z; As[q + 3][r] = v.w;
      } else {
        if (k0 + q < k_end && j0 + r - BM < g.N)
          v = *reinterpret_cast<const uint4*>(g.B + DAB_IDX((j0 + r - BM) * (int64_t)g.ldb + k0 + q, g.N * g.ldb - 3));
        Bs[q + 0][r - BM] = v.x; Bs[q + 1][r - BM] = v.y; Bs[q + 2][r - BM] = v.z; Bs[q + 3][r - BM] = v.w;
      }
    }
    __syncthreads();
    const int kw = min(BK, k_end - k0);
    const int groups = (kw + 2) / 3;  // the slice is zero-filled up to BK, a multiple of 3
#pragma unroll 1
    for (int gq = 0; gq < groups; ++gq) {
      const int w = gq * 3;
      uint32_t av[3][TM], bv[3][TN];
#pragma unroll
      for (int t = 0; t < 3; ++t) {
        if (TM == 4) {
          const uint4 a = *reinterpret_cast<const uint4*>(&As[w + t][a_t * TM]);
          av[t][0] = a.x; av[t][TM > 1 ? 1 : 0] = a.y; av[t][TM > 2 ? 2 : 0] = a.z; av[t][TM > 3 ? 3 : 0] = a.w;
        } else {
#pragma unroll
          for (int i = 0; i < TM; ++i) av[t][i] = As[w + t][a_t * TM + i];
        }
        const uint4 b = *reinterpret_cast<const uint4*>(&Bs[w + t][b_t * TN]);
        bv[t][0] = b.x; bv[t][1] = b.y; bv[t][2] = b.z; bv[t][3] = b.w;
      }
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) {
          uint32_t sum, carry;
          csa(av[0][i] & bv[0][j], av[1][i] & bv[1][j], av[2][i] & bv[2][j], sum, carry);
          ones[i][j] += __popc(sum);
          twos[i][j] += __popc(carry);
        }
    }
    __syncthreads();
  }

  auto weight = [&](int64_t gj) {
    return rescale_weight((double)g.alpha[DAB_IDX(gj, g.N)], (double)g.beta[DAB_IDX(gj, g.N)], g.KB[DAB_IDX(gj, g.N)], g.n);
  };
  auto activation = [&](int64_t gi) {
    return rescale_activation((double)g.gamma[DAB_IDX(gi, g.M)], (double)g.delta[DAB_IDX(gi, g.M)], g.KA[DAB_IDX(gi, g.M)]);
  };
  auto weight_gathers = [&](int64_t gj) { return gathers(g.alpha[DAB_IDX(gj, g.N)], g.beta[DAB_IDX(gj, g.N)]); };
  auto activation_gathers = [&](int64_t gi) { return gathers(g.gamma[DAB_IDX(gi, g.M)], g.delta[DAB_IDX(gi, g.M)]); };
  if (kSplit) {
    // The counts meet in shared memory, [column][row] or [row][column] as the lanes of the stores run; a member finishes
    // every splits-th line of the tile.
    constexpr int LINE = kLanesAlongRows ? BM : BN, LINES = kLanesAlongRows ? BN : BM, PITCH = LINE + 1;
    static_assert(LINES * PITCH <= BK * (ALD + BLD), "the counts fit the operands' place");
    int* const counts = reinterpret_cast<int*>(operands);
    cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        const int ii = a_t * TM + i, jj = b_t * TN + j;
        counts[kLanesAlongRows ? jj * PITCH + ii : ii * PITCH + jj] = ones[i][j] + 2 * twos[i][j];
      }
    cluster.sync();
    const int splits = (int)gridDim.z, rank = (int)cluster.block_rank();
    const int* member[kMaxSplit];
#pragma unroll
    for (int z = 0; z < kMaxSplit; ++z) member[z] = cluster.map_shared_rank(counts, z < splits ? z : 0);
    bool gathered = true;
    auto finish = [&](auto each_pair) {
      for (int t = tid; t < LINE * LINES / splits; t += GEMM_THREADS) {
        const int line = t / LINE * splits + rank, at = t % LINE;
        int p11 = 0;
#pragma unroll
        for (int z = 0; z < kMaxSplit; ++z)
          if (z < splits) p11 += member[z][line * PITCH + at];
        const int64_t gi = i0 + (kLanesAlongRows ? at : line), gj = j0 + (kLanesAlongRows ? line : at);
        if (gi >= g.M || gj >= g.N) continue;
        const int64_t to = (gi / g.map.inner) * g.map.outer_stride + (gi % g.map.inner) * g.map.row_stride + gj * g.map.col_stride;
        const float y = decltype(each_pair)::value ? rescale_any(g, p11, gi, gj) : rescale(p11, weight(gj), activation(gi));
        if (!decltype(each_pair)::value) gathered = gathered && weight_gathers(gj) && activation_gathers(gi);
        if (DAB_IN_BOUNDS(to, g.c_extent)) g.C[to] = apply_post(g.post, y, (int)gj, to, g.c_extent);
        if (g.p11 && DAB_IN_BOUNDS(gi * g.ldp + gj, (g.M - 1) * g.ldp + g.N)) g.p11[gi * g.ldp + gj] = p11;
      }
    };
    finish(std::false_type());
    if (!gathered) finish(std::true_type());
    cluster.sync();  // a member's counts are read until here
    return;
  }

  RescaleSide side[TN];
  bool gathered = true;
#pragma unroll
  for (int j = 0; j < TN; ++j) {
    const int64_t gj = j0 + b_t * TN + j;
    side[j] = gj < g.N ? weight(gj) : RescaleSide{0.0, 0.0, 0.0};
    gathered = gathered && (gj >= g.N || weight_gathers(gj));
  }
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    int64_t gi = i0 + a_t * TM + i;
    if (gi >= g.M) continue;
    const RescaleSide act = activation(gi);
    gathered = gathered && activation_gathers(gi);
    int64_t base = (gi / g.map.inner) * g.map.outer_stride + (gi % g.map.inner) * g.map.row_stride;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      int64_t gj = j0 + b_t * TN + j;
      if (gj >= g.N) continue;
      int p11 = ones[i][j] + 2 * twos[i][j];
      if (DAB_IN_BOUNDS(base + gj * g.map.col_stride, g.c_extent))
        g.C[base + gj * g.map.col_stride] =
            apply_post(g.post, rescale(p11, side[j], act), (int)gj, base + gj * g.map.col_stride, g.c_extent);
      if (g.p11 && DAB_IN_BOUNDS(gi * g.ldp + gj, (g.M - 1) * g.ldp + g.N)) g.p11[gi * g.ldp + gj] = p11;
    }
  }
  if (!gathered) {  // rare: the counts wait in the outputs' own places for a loop that is not unrolled
    auto place = [&](int64_t gi, int64_t gj) {
      return (gi / g.map.inner) * g.map.outer_stride + (gi % g.map.inner) * g.map.row_stride + gj * g.map.col_stride;
    };
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        const int64_t gi = i0 + a_t * TM + i, gj = j0 + b_t * TN + j;
        if (gi < g.M && gj < g.N && DAB_IN_BOUNDS(place(gi, gj), g.c_extent)) g.C[place(gi, gj)] = __int_as_float(ones[i][j] + 2 * twos[i][j]);
      }
#pragma unroll 1
    for (int t = 0; t < TM * TN; ++t) {
      const int64_t gi = i0 + a_t * TM + t / TN, gj = j0 + b_t * TN + t % TN;
      if (gi >= g.M || gj >= g.N) continue;
      const int64_t to = place(gi, gj);
      if (DAB_IN_BOUNDS(to, g.c_extent))
        g.C[to] = apply_post(g.post, rescale_any(g, __float_as_int(g.C[to]), gi, gj), (int)gj, to, g.c_extent);
    }
  }
}

namespace {

template <bool kLanesAlongRows, int TM>
cudaError_t launch_rows(const GemmArgs& args, cudaStream_t stream) {
  const dim3 grid((unsigned)((args.M + 16 * TM - 1) / (16 * TM)), (unsigned)((args.N + BN - 1) / BN));
  if (grid.y > 65535) return cudaErrorInvalidValue;
  // Split up to eight ways while the CTAs fit the SMs once and a member has six words.  The cluster and its two barriers cost 3 us,
  // so two ways pay only for long rows.  Measured, whole and split: 225 x 256 of 72 words 14.5 and 7.9 us (eight ways), of 36 words
  // 9.4 and 7.3 (four), 10.4 (two); 32 x 4096 of 128 words 21.9 and 12.7 (two), 17.5 (eight, four waves of CTAs).
  const int64_t tiles = (int64_t)grid.x * grid.y;
  int splits = 1;
  while (splits < kMaxSplit && tiles * 2 * splits <= sm_count() && args.words >= 12 * splits) splits *= 2;
  if (splits == 2 && args.words < 96) splits = 1;
  if (splits == 1) {
    binary_gemm_kernel<kLanesAlongRows, TM, false><<<grid, GEMM_THREADS, 0, stream>>>(args, args.words);
    return cudaGetLastError();
  }
  const int share = ((args.words + splits - 1) / splits + 3) & ~3;
  cudaLaunchConfig_t config = {};
  config.gridDim = dim3(grid.x, grid.y, (unsigned)splits);
  config.blockDim = dim3(GEMM_THREADS);
  config.stream = stream;
  cudaLaunchAttribute cluster[1];
  cluster[0].id = cudaLaunchAttributeClusterDimension;
  cluster[0].val.clusterDim.x = 1;
  cluster[0].val.clusterDim.y = 1;
  cluster[0].val.clusterDim.z = (unsigned)splits;
  config.attrs = cluster;
  config.numAttrs = 1;
  return cudaLaunchKernelEx(&config, binary_gemm_kernel<kLanesAlongRows, TM, true>, args, share);
}

}  // namespace

// 16 activation rows per tile where there are no more (a tile counts all its rows, also those beyond M), else 64.
cudaError_t launch_gemm(const GemmArgs& args, bool lanes_along_rows, cudaStream_t stream) {
  if (args.M <= 16) return lanes_along_rows ? launch_rows<true, 1>(args, stream) : launch_rows<false, 1>(args, stream);
  return lanes_along_rows ? launch_rows<true, 4>(args, stream) : launch_rows<false, 4>(args, stream);
}

}  // namespace dab
