// PTX building blocks of the tcgen05 kernels (sm_103a): mbarriers, TMA tile loads, shared-memory
// and instruction descriptors, MMA issue and commit, TMEM loads; and the host-side encoding of
// a BF16 [rows][kp] tensor map with 128-byte swizzle.  Shared by the fused bound kernel and the
// convolution GEMMs.
#pragma once

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include <string>

#include "bcrown_internal.cuh"

namespace bcrown {
namespace tc {

constexpr int KBLK = 64;  // bf16 per K block (128 bytes, one swizzle row)

__device__ __forceinline__ uint32_t su32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
  asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(su32(b)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
  asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(su32(b)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(su32(b)), "r"(parity)
      : "memory");
  return ok != 0;
}
// As mbar_try, but a thread whose phase is not complete yet is suspended (for at most about
// `ns` nanoseconds) until it completes, instead of returning at once: waiting threads then
// leave the issue slots and the shared-memory pipe to the warps doing work.
__device__ __forceinline__ bool mbar_try_sleep(uint64_t* b, uint32_t parity, uint32_t ns) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(su32(b)), "r"(parity), "r"(ns)
      : "memory");
  return ok != 0;
}
// Wait by a whole warp whose lanes all poll.  Their answers are combined, so that they leave the wait
// together and take the same branch, also where the time (about 2 s) runs out for some of them only: what
// follows elects a lane among all 32, or keeps the warp at one place of a ring, where a lane left
// behind would wait for a parity that has passed.  The phase stays complete while the warp waits for it, so
// a lane that has seen it sees it again.  aborted(): whether another warp gave up; give_up(): records it.
__device__ __forceinline__ bool mbar_try_together(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "vote.sync.all.pred q, p, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(ok)
      : "r"(su32(b)), "r"(parity)
      : "memory");
  return ok != 0;
}
template <class Aborted, class GiveUp>
__device__ __forceinline__ bool mbar_wait_together(uint64_t* b, uint32_t parity, Aborted aborted, GiveUp give_up) {
  if (mbar_try_together(b, parity)) return true;
  const long long t0 = clock64();
  while (true) {
    if (__all_sync(0xffffffffu, mbar_try_sleep(b, parity, 20000u))) return true;
    const bool late = clock64() - t0 > 4000000000LL;
    if (__any_sync(0xffffffffu, late || aborted())) {
      if (late) give_up();
      return false;
    }
  }
}
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          su32(dst)),
      "l"((uint64_t)map), "r"(x), "r"(y), "r"(su32(bar))
      : "memory");
}
__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                            uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];" ::
          "r"(su32(dst)),
      "l"((uint64_t)map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(su32(bar))
      : "memory");
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// Shared-memory matrix descriptor, K-major, 128-byte swizzle, 8-row groups 1024 B apart.
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)1 << 16;                 // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;       // stride byte offset
  d |= (uint64_t)1 << 46;                 // descriptor version
  d |= (uint64_t)2 << 61;                 // SWIZZLE_128B
  return d;
}
// Instruction descriptor: BF16 x BF16 -> FP32, both K-major, M = 128, N = n.
__host__ __device__ constexpr uint32_t idesc_bf16(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}
// One 64-wide K block: four MMAs of K = 16.  Descriptors of consecutive 16-element K steps
// differ by 32 bytes in the start address (field unit 16 bytes: +2); `acc` = 0 starts the
// accumulator with the first MMA.
__device__ __forceinline__ void umma_kblock(uint32_t dtmem, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.eq.b32 q, 0, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %5, %6, %3, q;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %7, %8, %3, q;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %9, %10, %3, q;\n\t}" ::"r"(dtmem),
      "l"(ad), "l"(bd), "r"(idesc), "r"(acc), "l"(ad + 2), "l"(bd + 2), "l"(ad + 4), "l"(bd + 4), "l"(ad + 6),
      "l"(bd + 6)
      : "memory");
}
// Low word of sdesc (the high word is a constant).
__device__ __forceinline__ uint32_t sdesc_lo(uint32_t saddr) { return ((saddr >> 4) & 0x3FFFu) | (1u << 16); }
// A K pair -- the K block at (alo, blo) and, with `two`, the one ASTEP / BSTEP 16-byte units on -- and
// the commit to `bar`, for a whole converged warp: elect.sync picks the lane, the instructions are
// predicated (no one-lane branch), and the descriptors are built from 32-bit words.  This matters
// to a warp whose own instructions are what an MMA waits for: measured per MMA of 128 x N x 16,
// issued back to back, 39 cycles (48 at N = 64, the tensor core's own time) against 47 from a
// one-lane branch and 67 under a predicate computed from the lane index.
template <uint32_t ASTEP, uint32_t BSTEP>
__device__ __forceinline__ void umma_kpair(uint32_t dtmem, uint32_t alo, uint32_t blo, uint32_t idesc, uint32_t acc,
                                           uint32_t two, uint32_t bar) {
  constexpr uint32_t hi = (1024u >> 4) | (1u << 14) | (2u << 29);
#define BC_UMMA(P, OFF_A, OFF_B, ACC)                                                                  \
  "add.u32 x, %1, " OFF_A ";\n\tadd.u32 y, %2, " OFF_B ";\n\tmov.b64 a, {x, %6};\n\tmov.b64 b, {y, %6};\n\t" \
  "@" P " tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, " ACC ";\n\t"
  asm volatile(
      "{\n\t.reg .pred l, m, p, q;\n\t.reg .b64 a, b;\n\t.reg .b32 x, y, d;\n\telect.sync d|l, 0xffffffff;\n\t"
      "setp.ne.and.b32 m, %5, 0, l;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.eq.b32 q, 0, 0;\n\t"
      BC_UMMA("l", "0", "0", "p") BC_UMMA("l", "2", "2", "q") BC_UMMA("l", "4", "4", "q") BC_UMMA("l", "6", "6", "q")
      BC_UMMA("m", "%8", "%9", "q") BC_UMMA("m", "%10", "%11", "q") BC_UMMA("m", "%12", "%13", "q")
      BC_UMMA("m", "%14", "%15", "q")
      "@l tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%7];\n\t}" ::"r"(dtmem),
      "r"(alo), "r"(blo), "r"(idesc), "r"(acc), "r"(two), "n"(hi), "r"(bar), "n"(ASTEP), "n"(BSTEP),
      "n"(ASTEP + 2), "n"(BSTEP + 2), "n"(ASTEP + 4), "n"(BSTEP + 4), "n"(ASTEP + 6), "n"(BSTEP + 6)
      : "memory");
#undef BC_UMMA
}
// One K block and the commit to `bar` for a converged warp, as above.  HI_A: high word of the A
// descriptor, STEP_A: its advance per K step of 16 (16-byte units).
template <uint32_t HI_A, uint32_t STEP_A>
__device__ __forceinline__ void umma_kblock_warp(uint32_t dtmem, uint32_t alo, uint32_t blo, uint32_t idesc,
                                                 uint32_t acc, uint32_t bar) {
  constexpr uint32_t hi = (1024u >> 4) | (1u << 14) | (2u << 29);
#define BC_UMMA1(OFF_A, OFF_B, ACC)                                                                    \
  "add.u32 x, %1, " OFF_A ";\n\tadd.u32 y, %2, " OFF_B ";\n\tmov.b64 a, {x, %5};\n\tmov.b64 b, {y, %6};\n\t" \
  "@l tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, " ACC ";\n\t"
  asm volatile(
      "{\n\t.reg .pred l, p, q;\n\t.reg .b64 a, b;\n\t.reg .b32 x, y, d;\n\telect.sync d|l, 0xffffffff;\n\t"
      "setp.ne.b32 p, %4, 0;\n\tsetp.eq.b32 q, 0, 0;\n\t"
      BC_UMMA1("0", "0", "p") BC_UMMA1("%8", "2", "q") BC_UMMA1("%9", "4", "q") BC_UMMA1("%10", "6", "q")
      "@l tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%7];\n\t}" ::"r"(dtmem),
      "r"(alo), "r"(blo), "r"(idesc), "r"(acc), "n"(HI_A), "n"(hi), "r"(bar), "n"(STEP_A), "n"(2 * STEP_A),
      "n"(3 * STEP_A)
      : "memory");
#undef BC_UMMA1
}
constexpr uint32_t SDESC_HI = (1024u >> 4) | (1u << 14) | (2u << 29);         // sdesc's high word
// High and low word of a K-major descriptor without swizzle: 8-row x 16-byte core matrices of 128 contiguous
// bytes, `sbo` bytes apart along M and `lbo` bytes apart along K.
__host__ __device__ constexpr uint32_t SDESC_PLAIN_HI(uint32_t sbo) { return (sbo >> 4) | (1u << 14); }
__device__ __forceinline__ uint32_t sdesc_plain_lo(uint32_t saddr, uint32_t lbo) {
  return ((saddr >> 4) & 0x3FFFu) | ((lbo >> 4) << 16);
}
// A commit by one lane of a converged warp.
__device__ __forceinline__ void umma_commit_warp(uint32_t bar) {
  asm volatile(
      "{\n\t.reg .pred l;\n\t.reg .b32 d;\n\telect.sync d|l, 0xffffffff;\n\t"
      "@l tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar)
      : "memory");
}
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(su32(bar))
               : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&v)[8]) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}
// Split form of tmem_ld8: the load, then the wait.  The wait names the registers as in-out
// operands, so no use of them can be scheduled before it.
__device__ __forceinline__ void tmem_ld8_issue(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void tmem_wait8(uint32_t (&r)[8]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7])
               :
               : "memory");
}

// The same for 4 columns.
__device__ __forceinline__ void tmem_ld4_issue(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void tmem_wait4(uint32_t (&r)[4]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]) : : "memory");
}
template <int N>
__device__ __forceinline__ void tmem_ld_issue(uint32_t taddr, uint32_t (&r)[N]) {
  static_assert(N == 4 || N == 8, "columns per load");
  if constexpr (N == 8) tmem_ld8_issue(taddr, r);
  else tmem_ld4_issue(taddr, r);
}
template <int N>
__device__ __forceinline__ void tmem_wait(uint32_t (&r)[N]) {
  if constexpr (N == 8) tmem_wait8(r);
  else tmem_wait4(r);
}

// Tensor map of a BF16 [rows][kp] matrix (kp a multiple of 64): boxes of 64 x box_rows, 128-byte
// swizzle (the K-major layout sdesc describes).
inline int encode_map(CUtensorMap* m, void* base, int rows, int kp, int box_rows) {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        !p)
      return fail(BCROWN_ERR_CUDA, "cuTensorMapEncodeTiled not available");
    fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
  }
  cuuint64_t dims[2] = {(cuuint64_t)kp, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)kp * 2};
  cuuint32_t box[2] = {(cuuint32_t)KBLK, (cuuint32_t)box_rows};
  cuuint32_t es[2] = {1, 1};
  CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(BCROWN_ERR_CUDA, "cuTensorMapEncodeTiled failed: " + std::to_string((int)r));
  return BCROWN_OK;
}

// Tensor map of a BF16 tensor of `rank` dimensions (innermost first: dims[0] elements of 2 bytes,
// strides[d - 1] bytes between consecutive indices of dimension d), boxes of box[0..rank), with
// the 128-byte swizzle (box[0] = 64: one 128-byte row per index of the outer dimensions).
// Coordinates outside the tensor read as zero.  estride (optional): the traversal step of each
// dimension; a box then holds ceil(box[d] / estride[d]) elements of dimension d, every
// estride[d]-th from its start coordinate.  swizzle = false: no swizzle (a box of 16-byte rows
// lands as consecutive 16-byte rows).
inline int encode_map_nd(CUtensorMap* m, void* base, int rank, const cuuint64_t* dims, const cuuint64_t* strides,
                         const cuuint32_t* box, const cuuint32_t* estride = nullptr, bool swizzle = true) {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        !p)
      return fail(BCROWN_ERR_CUDA, "cuTensorMapEncodeTiled not available");
    fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
  }
  cuuint32_t es[5] = {1, 1, 1, 1, 1};
  if (estride)
    for (int d = 0; d < rank; ++d) es[d] = estride[d];
  CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, base, dims, strides, box, es,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(BCROWN_ERR_CUDA, "cuTensorMapEncodeTiled failed: " + std::to_string((int)r));
  return BCROWN_OK;
}

}  // namespace tc
}  // namespace bcrown
