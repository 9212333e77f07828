// Blackwell (sm_103a) tensor-core building blocks written as inline PTX:
// tcgen05.alloc/dealloc (tensor memory), tcgen05.mma kind::f16 with BF16
// operands and an FP32 accumulator in tensor memory, tcgen05.commit to an
// mbarrier, tcgen05.ld of the accumulator, and the shared-memory operand
// layout these MMAs read.
//
// Operand layout ("SW128 block"): a [R x 64] BF16 matrix block (R rows, 64
// elements of K per row, R a multiple of 8) occupies R * 128 bytes of shared
// memory, 1024-byte aligned.  Row r starts at r * 128; the 16-byte chunk c
// (elements 8c..8c+7) of row r sits at chunk position c ^ (r % 8).  This is
// the 128-byte swizzle of the UMMA descriptor (layout type 2) with K-major
// rows; the stride between 8-row groups is 1024 bytes.  Longer K is a
// sequence of such blocks.
#pragma once
#include <cstdint>
#include <cuda_bf16.h>

namespace lbmgnn {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Byte offset of element (r, k) (0 <= k < 64) inside an SW128 block.
__host__ __device__ __forceinline__ uint32_t sw128_off(uint32_t r, uint32_t k) {
  return r * 128u + ((((k >> 3) ^ (r & 7u)) & 7u) << 4) + (k & 7u) * 2u;
}

// Shared-memory matrix descriptor: start address, leading byte offset 16,
// stride byte offset 1024 (8 rows x 128 B), descriptor version 1, 128-byte
// swizzle.  `addr` is a shared-space byte address.
__device__ __forceinline__ uint64_t sw128_desc(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)(16u >> 4) << 16;
  d |= (uint64_t)(1024u >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// Instruction descriptor of tcgen05.mma kind::f16: BF16 A and B (both
// K-major), FP32 accumulator, M x N tile.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}

// ---- tensor memory -------------------------------------------------------
// Allocate `ncols` columns (power of two >= 32); executed by one full warp.
// The address is written to the shared-memory word `slot`.
__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                   smem_u32(slot)),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// Make generic-proxy shared-memory writes visible to the tensor core.
__device__ __forceinline__ void fence_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// ---- mbarrier ----------------------------------------------------------------
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
               : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// The same test with a suspend-time hint: a thread whose phase is not yet
// complete may sleep up to `ns` nanoseconds and is woken when it completes,
// so a wait costs one instruction instead of a polling loop.  CLUSTER: the
// phase completes with writes of other CTAs of the cluster (st.async), which
// an acquire at the default scope, the CTA's, does not cover.
template <bool CLUSTER = false>
__device__ __forceinline__ bool mbar_try_wait_sleep(uint64_t* bar, uint32_t parity, uint32_t ns) {
  uint32_t ok;
  if constexpr (CLUSTER) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity), "r"(ns)
        : "memory");
  } else {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity), "r"(ns)
        : "memory");
  }
  return ok != 0;
}
// Bounded wait: gives up after ~`max_cycles` SM cycles and returns false.
// Each try may sleep up to 0.1 ms (woken at once by the phase's completion);
// the clock is read only when a try comes back empty.
template <bool CLUSTER = false>
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity,
                                          long long max_cycles = 4000000000LL) {
  if (mbar_try_wait_sleep<CLUSTER>(bar, parity, 100000u)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait_sleep<CLUSTER>(bar, parity, 100000u)) {
    if (clock64() - t0 > max_cycles) return false;
  }
  return true;
}

// ---- MMA -------------------------------------------------------------------------
// D[tmem] (+)= A * B^T with A: M x 16 and B: N x 16 slices given by descriptors.
__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc,
                                          uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// D[tmem] (+)= A * B^T with the A slice (M = 128 rows x 16 K, BF16) read from
// tensor memory: lane r holds row r, K packed two per 32-bit column (element
// 2c in the low half of column c), 8 columns per K step starting at tmem_a.
__device__ __forceinline__ void umma_bf16_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc,
                                             uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(tmem_d),
      "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrive on `bar` when all previously issued MMAs of this thread completed.
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(bar))
      : "memory");
}

// D (M=128 rows) = sum over kb < nkb of A_kb * B_kb^T, where A_kb and B_kb are
// SW128 blocks of 128 and N rows at a_addr + kb*a_stride, b_addr + kb*b_stride
// (shared-space byte addresses).  Issued by a single thread.
// `nks` (<= 4) is the number of 16-wide K steps used in each block.
__device__ __forceinline__ void umma_128xN(uint32_t tmem_d, uint32_t a_addr, uint32_t a_stride,
                                           uint32_t b_addr, uint32_t b_stride, int nkb, int N,
                                           bool accumulate, int nks = 4) {
  const uint32_t id = idesc_bf16(128, N);
  for (int kb = 0; kb < nkb; ++kb) {
    for (int ks = 0; ks < nks; ++ks) {
      const uint64_t ad = sw128_desc(a_addr + kb * a_stride + ks * 32);
      const uint64_t bd = sw128_desc(b_addr + kb * b_stride + ks * 32);
      umma_bf16(tmem_d, ad, bd, id, (accumulate || kb > 0 || ks > 0) ? 1u : 0u);
    }
  }
}

// ---- operands read across their rows (MN-major) ------------------------------------
// The same SW128 blocks serve as an operand whose K runs down the rows: a block
// of R rows x 64 values is then K = R (rows) by 64 values of M or N, so a tile
// stored [node][feature] is also the transposed operand of a contraction over
// nodes, without a transposed copy.  Rows stay 128 bytes apart, 8-row groups
// 1024; `blk` is the distance of the next block of 64 M (or N) values.  16 K
// steps are 2048 bytes.
__device__ __forceinline__ uint64_t sw128_desc_mn(uint32_t addr, uint32_t blk) {
  return (sw128_desc(addr) & ~((uint64_t)0x3FFF << 16)) | (uint64_t)((blk & 0x3FFFFu) >> 4) << 16;
}
constexpr uint32_t A_MN = 1u << 15, B_MN = 1u << 16;  // instruction descriptor bits

// D (M x N) (+)= A^T B over `nks` K steps, A and B both MN-major.
__device__ __forceinline__ void umma_tt(uint32_t tmem_d, uint32_t a_addr, uint32_t a_blk,
                                        uint32_t b_addr, uint32_t b_blk, int N, int nks,
                                        bool accumulate) {
  const uint32_t id = idesc_bf16(128, N) | A_MN | B_MN;
  for (int ks = 0; ks < nks; ++ks)
    umma_bf16(tmem_d, sw128_desc_mn(a_addr + ks * 2048, a_blk),
              sw128_desc_mn(b_addr + ks * 2048, b_blk), id, (accumulate || ks > 0) ? 1u : 0u);
}
// The same with B K-major: SW128 blocks of N rows x 64 K at b_addr + kb * b_stride.
__device__ __forceinline__ void umma_tn(uint32_t tmem_d, uint32_t a_addr, uint32_t a_blk,
                                        uint32_t b_addr, uint32_t b_stride, int N, int nks,
                                        bool accumulate) {
  const uint32_t id = idesc_bf16(128, N) | A_MN;
  for (int ks = 0; ks < nks; ++ks)
    umma_bf16(tmem_d, sw128_desc_mn(a_addr + ks * 2048, a_blk),
              sw128_desc(b_addr + (ks >> 2) * b_stride + (ks & 3) * 32), id,
              (accumulate || ks > 0) ? 1u : 0u);
}
// And with A K-major (blocks of 128 rows x 64 K) and B MN-major.
__device__ __forceinline__ void umma_nt(uint32_t tmem_d, uint32_t a_addr, uint32_t a_stride,
                                        uint32_t b_addr, uint32_t b_blk, int N, int nks,
                                        bool accumulate) {
  const uint32_t id = idesc_bf16(128, N) | B_MN;
  for (int ks = 0; ks < nks; ++ks)
    umma_bf16(tmem_d, sw128_desc(a_addr + (ks >> 2) * a_stride + (ks & 3) * 32),
              sw128_desc_mn(b_addr + ks * 2048, b_blk), id, (accumulate || ks > 0) ? 1u : 0u);
}

// D (M = 128) = A * B^T over `nks` K steps of 16, A from tensor memory at
// tmem_a (8 columns per step), B from one SW128 block of N rows at b_addr.
__device__ __forceinline__ void umma_128xN_ts(uint32_t tmem_d, uint32_t tmem_a, uint32_t b_addr,
                                              int N, int nks) {
  const uint32_t id = idesc_bf16(128, N);
  for (int ks = 0; ks < nks; ++ks)
    umma_bf16_ts(tmem_d, tmem_a + 8u * ks, sw128_desc(b_addr + ks * 32), id, ks > 0 ? 1u : 0u);
}

// ---- tensor memory stores ---------------------------------------------------------
// 16 / 32 consecutive 32-bit columns of the calling thread's lane; the
// stores are complete for later tensor-core reads after tmem_st_wait()
// and a thread barrier with the tcgen05 fences.
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&w)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
      "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]),
      "r"(w[8]), "r"(w[9]), "r"(w[10]), "r"(w[11]), "r"(w[12]), "r"(w[13]), "r"(w[14]),
      "r"(w[15])
      : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&w)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
      "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]),
      "r"(w[8]), "r"(w[9]), "r"(w[10]), "r"(w[11]), "r"(w[12]), "r"(w[13]), "r"(w[14]),
      "r"(w[15]), "r"(w[16]), "r"(w[17]), "r"(w[18]), "r"(w[19]), "r"(w[20]), "r"(w[21]),
      "r"(w[22]), "r"(w[23]), "r"(w[24]), "r"(w[25]), "r"(w[26]), "r"(w[27]), "r"(w[28]),
      "r"(w[29]), "r"(w[30]), "r"(w[31])
      : "memory");
}
__device__ __forceinline__ void tmem_st_wait() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// ---- tensor memory loads ---------------------------------------------------------
// 32 consecutive FP32 columns of the calling thread's lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
        "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
        "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
        "=r"(r[31])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
// tmem_ld32 without the wait: the registers are valid after tmem_ld_wait().
__device__ __forceinline__ void tmem_ld32_async(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
        "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
        "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
        "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
// 16 consecutive FP32 columns of the calling thread's lane.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
        "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

}  // namespace lbmgnn
