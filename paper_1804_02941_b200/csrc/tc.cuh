// Inline-PTX helpers shared by the tensor-core kernels: shared-memory and instruction descriptors of
// tcgen05.mma kind::i8, bounded mbarrier waits, tensor-memory loads and the expansion of mask bits to bytes.
//
// Shared-memory operand layout used throughout (K-major, no swizzle): 8 rows x 16 bytes form one contiguous
// 128-byte core matrix; core matrices of consecutive 16-byte K chunks follow each other (leading byte offset
// 128) and groups of 8 rows are one whole stage row apart (stride byte offset = K chunks per stage x 128).
// One kind::i8 instruction covers 32 K bytes = two K chunks.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace dab {
namespace tc {

constexpr int kLanes = 128;                      // rows of an accumulator = lanes of tensor memory
constexpr long long kWaitCycles = 4000000000ll;  // about two seconds; a wait that long has failed

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor: address, leading and stride byte offsets in 16-byte units, descriptor
// version 1 in bits [46,48), no swizzle (layout type 0 in bits [61,64)).
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo_bytes >> 4) << 16) |
         ((uint64_t)(sbo_bytes >> 4) << 32) | (1ull << 46);
}

// The descriptor of the same operand `bytes` (a multiple of 16) further on.
__device__ __forceinline__ uint64_t desc_at(uint64_t desc, uint32_t bytes) { return desc + (bytes >> 4); }

// Named barriers: `threads` threads in all, of which some only arrive.
__device__ __forceinline__ void bar_arrive(int id, int threads) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory"); }
__device__ __forceinline__ void bar_sync(int id, int threads) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory"); }

// Instruction descriptor of kind::i8: D format S32 (2 at bit 4), A format at bit 7 and B format at bit 10
// (0: unsigned 8-bit, 1: signed 8-bit), both K-major (0 at bits 15 and 16), N / 8 at bit 17, M / 16 at bit 24.
__device__ __forceinline__ uint32_t instr_desc(int nt, bool a_signed = false, bool b_signed = false) {
  return (2u << 4) | ((a_signed ? 1u : 0u) << 7) | ((b_signed ? 1u : 0u) << 10) | ((uint32_t)(nt >> 3) << 17) |
         ((uint32_t)(kLanes >> 4) << 24);
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

// Bounded wait for the phase with the given parity.  Returns false after `limit` cycles and counts the failure
// in *failures (device global); the caller then stops waiting on anything (dead stays set) but keeps its
// control flow, so that every thread still reaches every barrier and the CTA ends.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, bool& dead, unsigned int* failures,
                                          long long limit = kWaitCycles) {
  if (dead) return false;
  const long long t0 = clock64();
  for (;;) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
    if (clock64() - t0 > limit) {
      dead = true;
      atomicAdd(failures, 1u);
      return false;
    }
  }
}

// The wait for the last commit before tensor memory is given back: with a limit of its own, also after an earlier wait ran out.
__device__ __forceinline__ void mbar_wait_last(uint32_t bar, uint32_t parity, bool& dead, unsigned int* failures,
                                               long long limit = kWaitCycles) {
  bool late = false;
  mbar_wait(bar, parity, late, failures, limit);
  dead = dead || late;
}

// A producer warp hands a stage to the warp that issues the products (which takes it with bar_sync).  It does not block: the wait
// for the buffer's next use keeps the two in step.  A producer whose waits no longer hold (dead) waits here instead: running
// ahead, it would arrive twice in one phase, and the issuing warp would wait for arrivals that have been spent.
__device__ __forceinline__ void stage_handover(int id, int threads, bool dead) {
  if (__any_sync(0xFFFFFFFFu, dead)) bar_sync(id, threads);
  else bar_arrive(id, threads);
}

// The operands of an instruction live in uniform registers.  Issued under a branch on the thread, with operands the compiler
// cannot tell are the warp's, one took 175 cycles to issue, whatever it multiplied (128 x 128 x 32: 64 cycles of tensor-core
// time).  So: a warp's number and the tensor-memory address go through uniform(), the loops over instructions are unrolled,
// and elect_one() picks the thread inside a branch that the whole warp takes.
__device__ __forceinline__ void mma_i8(uint32_t tmem_d, uint64_t desc_a, uint64_t desc_b, uint32_t idesc,
                                       uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}"
      :
      : "r"(tmem_d), "l"(desc_a), "l"(desc_b), "r"(idesc), "r"(accumulate)
      : "memory");
}

// The same with the first operand in tensor memory: row i in lane i, four consecutive K bytes per column.
__device__ __forceinline__ void mma_i8_tmem(uint32_t tmem_d, uint32_t tmem_a, uint64_t desc_b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::i8 [%0], [%1], %2, %3, p;\n\t}"
      :
      : "r"(tmem_d), "r"(tmem_a), "l"(desc_b), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ uint32_t uniform(uint32_t v) { return __shfl_sync(0xFFFFFFFFu, v, 0); }

// True in one thread of the (converged) warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t e;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.b32 %0, 1, 0, p;\n\t}" : "=r"(e));
  return e != 0u;
}

// Arrives on the barrier once every tcgen05.mma issued by this thread so far has completed.
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tmem_alloc(uint32_t slot_smem_addr, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot_smem_addr), "r"(cols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t tmem, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols) : "memory");
}

__device__ __forceinline__ void tmem_load_32(uint32_t taddr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
        "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
        "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// 32 consecutive columns of this warp's 32 lanes (no wait: follow with tcgen05.wait::st).
__device__ __forceinline__ void tmem_store_32(uint32_t taddr, const uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%32], "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31};"
      :
      : "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
        "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]),
        "r"(v[16]), "r"(v[17]), "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]),
        "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]), "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31]), "r"(taddr)
      : "memory");
}

// Eight consecutive columns of this warp's 32 lanes (no wait: follow with tmem_load_wait).
__device__ __forceinline__ void tmem_load_8(uint32_t taddr, uint32_t (&v)[8]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
      : "r"(taddr)
      : "memory");
}

__device__ __forceinline__ void tmem_load_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Four mask bits -> four bytes of 0 / -1 with one byte permutation: the selector's nibbles are bits s, s+4, s+8
// and s+12 of the word shifted right by s (their lowest bit picks byte 0x00 or 0xFF of the source; the other
// selector bits pick among copies of the same two bytes, and sign replication of 0x00 / 0xFF changes nothing).
__device__ __forceinline__ uint32_t select4(uint32_t selector) {
  uint32_t d;
  asm("prmt.b32 %0, %1, %1, %2;" : "=r"(d) : "r"(0xFF00FF00u), "r"(selector));
  return d;
}

// One mask word of one row -> two 16-byte K chunks of 0 / -1 bytes (signed 8-bit
// operands).  Within a word's 32 bytes the bits appear in the order 0 4 8 12, 1 5 9 13, 2 6 10 14, 3 7 11 15, then the
// same for the upper half.
__device__ __forceinline__ void expand_word_signed(uint32_t w, unsigned char* dst) {
  uint4 lo, hi;
  lo.x = select4(w);
  lo.y = select4(w >> 1);
  lo.z = select4(w >> 2);
  lo.w = select4(w >> 3);
  hi.x = select4(w >> 16);
  hi.y = select4(w >> 17);
  hi.z = select4(w >> 18);
  hi.w = select4(w >> 19);
  *reinterpret_cast<uint4*>(dst) = lo;
  *reinterpret_cast<uint4*>(dst + 128) = hi;
}

// Mask words as unsigned bytes for the contraction of two such rows.  Register j of a word holds its bits j, j + 8, j + 16 and
// j + 24, one per byte and where they stand: 2^j or 0.  The other side's are mirrored, 2^(7-j) or 0, so that every product of two set
// bits is 128: the integer dot product of the rows is kBitProduct * popc(e AND f), and an AND per four bits is all it takes.
constexpr int kBitProductLog = 7;
__device__ __forceinline__ void expand_bits(uint32_t w, uint32_t* out) {
#pragma unroll
  for (int j = 0; j < 8; ++j) out[j] = w & (0x01010101u << j);
}
__device__ __forceinline__ void expand_bits_mirrored(uint32_t w, uint32_t* out) {
  const uint32_t m = __byte_perm(__brev(w), 0u, 0x0123);  // the bits of every byte in reverse order
#pragma unroll
  for (int j = 0; j < 8; ++j) out[j] = m & (0x80808080u >> j);
}

// A mask word of one row -> its two 16-byte K chunks, 128 bytes apart.
template <bool kMirrored>
__device__ __forceinline__ void expand_word_bits(uint32_t w, unsigned char* dst) {
  uint32_t b[8];
  if (kMirrored) expand_bits_mirrored(w, b);
  else expand_bits(w, b);
  *reinterpret_cast<uint4*>(dst) = make_uint4(b[0], b[1], b[2], b[3]);
  *reinterpret_cast<uint4*>(dst + 128) = make_uint4(b[4], b[5], b[6], b[7]);
}

}  // namespace tc
}  // namespace dab
