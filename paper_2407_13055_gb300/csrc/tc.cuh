// Blackwell tensor-core (tcgen05), tensor-memory, bulk-copy and mbarrier
// primitives as inline PTX, and the exact integer arithmetic that runs the
// BConv matrix product (Eq. 2; Sec. 4.2 treats BConv as a matrix product)
// on the fp16 tensor pipe.
//
// Exactness. A centered residue y (|y| < 2^30) is written as four balanced
// signed bytes, y = sum_a d_a 2^(8a) with d_a in [-128, 128); the byte
// weights are folded into the matrix, m'_(k,a) = [m_k 2^(8a)]_p centered, and
// each m' is split the same way into four bytes e_(k,a,b) ("planes" b). Every
// byte is an exact fp16 value and every product d e (|d e| <= 2^14) an exact
// fp32 value, and plane b's sum over the K sources and 4 digits,
// P_b = sum_(k,a) d_(k,a) e_(k,a,b), stays below 2^20 in magnitude for
// K <= 16 (448 2^7 per source), so the fp32 accumulation is exact in any order.
// Then sum_b P_b 2^(8b) = sum_k y_k m_k modulo p; reduced, it is the residue
// that the CUDA-core lazy sum gives.
#pragma once
#include <cuda_fp16.h>

#include <cstdint>

#include "arith.cuh"

namespace ckks {
namespace tc {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor (tcgen05), no swizzling: the operand is a
// grid of core matrices of 8 rows x 16 bytes (128 contiguous bytes each);
// lbo = byte distance between core matrices adjacent along K, sbo = between
// core matrices adjacent along M (or N). Bits 46-48 hold the fixed value 1.
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo & 0x3FFFFu) >> 4) << 16;
  d |= (uint64_t)((sbo & 0x3FFFFu) >> 4) << 32;
  d |= 1ull << 46;
  return d;
}

// Instruction descriptor of tcgen05.mma.kind::f16: A and B fp16, D fp32,
// both operands K-major, M x N tile (M = 128: N a multiple of 16 up to 256).
__host__ __device__ constexpr uint32_t idesc_f16(int m, int n) {
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

// D[tmem] (+)= A[tmem] * B^T, executed by a whole converged warp and issued by
// one elected lane; completion is tracked with commit(). A: one tensor-memory
// lane per row, two consecutive K elements per 32-bit column. The election
// sits in the instruction's predicate: under a branch on the lane the operands
// cannot be uniform registers, and an issue took 119 cycles instead of 8
// (32 products of N = 16: 3946 against 408 cycles to their completion).
template <bool ACCUMULATE>
__device__ __forceinline__ void mma_f16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t idesc) {
  asm volatile(
      "{\n.reg .pred p, q;\nelect.sync _|q, 0xffffffff;\nsetp.ne.b32 p, %4, 0;\n"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b), "r"(idesc), "n"(ACCUMULATE ? 1 : 0)
      : "memory");
}

// The mbarrier at mbar receives one arrival when every tcgen05.mma issued so
// far by the elected lane of this (whole, converged) warp has completed.
__device__ __forceinline__ void commit(uint32_t mbar) {
  asm volatile(
      "{\n.reg .pred q;\nelect.sync _|q, 0xffffffff;\n"
      "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(mbar)
      : "memory");
}

// Tensor-memory allocation: executed by one whole warp; the base address is
// written to shared memory at slot. ncols is a power of two >= 32.
__device__ __forceinline__ void tmem_alloc(uint32_t slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Four consecutive 32-bit columns of this thread's TMEM lane (the warp reads
// the 32 lanes of its quadrant, warp id mod 4); taddr carries the quadrant's
// first lane in its upper half. And two columns written.
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t& a, uint32_t& b, uint32_t& c, uint32_t& d) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(a), "=r"(b), "=r"(c), "=r"(d)
               : "r"(taddr)
               : "memory");
}
// Waits for this thread's loads; the registers pass through the statement so
// that nothing reads them before it.
__device__ __forceinline__ void tmem_wait_ld32(uint32_t (&f)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(f[0]), "+r"(f[1]), "+r"(f[2]), "+r"(f[3]), "+r"(f[4]), "+r"(f[5]), "+r"(f[6]), "+r"(f[7]),
                 "+r"(f[8]), "+r"(f[9]), "+r"(f[10]), "+r"(f[11]), "+r"(f[12]), "+r"(f[13]), "+r"(f[14]), "+r"(f[15]),
                 "+r"(f[16]), "+r"(f[17]), "+r"(f[18]), "+r"(f[19]), "+r"(f[20]), "+r"(f[21]), "+r"(f[22]),
                 "+r"(f[23]), "+r"(f[24]), "+r"(f[25]), "+r"(f[26]), "+r"(f[27])
               :
               : "memory");
  asm volatile("" : "+r"(f[28]), "+r"(f[29]), "+r"(f[30]), "+r"(f[31])::"memory");
}
__device__ __forceinline__ void tmem_st2(uint32_t taddr, uint32_t a, uint32_t b) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1,%2};" ::"r"(taddr), "r"(a), "r"(b) : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void mbar_init(uint32_t mbar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mbar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_init_fence() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

// Non-blocking test / potentially blocking try of the phase with the given
// parity.
__device__ __forceinline__ bool mbar_test(uint32_t mbar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(mbar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_try(uint32_t mbar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(mbar), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait: true once the phase completed, false after `limit` SM clock
// cycles without completion. Limits below kPollLimit cycles poll with the
// non-blocking test only (a blocking try may sleep past such a limit), so a
// limit of a few cycles expires whenever the phase is still pending at the
// call; longer limits let the hardware suspend the waiting warp.
constexpr long long kPollLimit = 1024;
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity, long long limit) {
  if (mbar_test(mbar, parity)) return true;
  const long long t0 = clock64();
  if (limit < kPollLimit) {
    while (clock64() - t0 <= limit)
      if (mbar_test(mbar, parity)) return true;
    return false;
  }
  while (clock64() - t0 <= limit)
    if (mbar_try(mbar, parity)) return true;
  return false;
}

__device__ __forceinline__ void mbar_arrive(uint32_t mbar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar) : "memory");
}

// One arrival that also expects `bytes` of transaction (bulk-copy) data.
__device__ __forceinline__ void mbar_expect_tx(uint32_t mbar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"(bytes) : "memory");
}

// Bulk copy global -> shared of `bytes` (a multiple of 16; both addresses
// 16-byte aligned) that completes on mbar's transaction count. The source is
// this GPU's own memory; the destination is this CTA's shared memory.
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t mbar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
      "l"(src), "r"(bytes), "r"(mbar)
      : "memory");
}

// Status word bits written by bounded waits that expired (read back by the
// host as CKKS_ETIMEOUT).
constexpr uint32_t kStatusTimeout = 1u;
// Set by the range checks of the checked launch mode (a residue >= its prime).
constexpr uint32_t kStatusRange = 2u;

__device__ __forceinline__ void report_timeout(uint32_t* status) {
  if (status) atomicOr(status, kStatusTimeout);
}

// Four balanced signed-byte digits of a centered residue y (|y| < 2^30) as two
// fp16 pairs, in order d0 d1 | d2 d3, from z = y + 0x80808080: byte a of z is
// d_a + 128 (d3 in [-64, 64]). Each byte u becomes the fp16 1024 + u by placing
// 0x64 above it; subtracting 1152 then leaves u - 128 exactly.
__device__ __forceinline__ uint2 digits_f16(uint32_t z) {
  uint32_t lo = __byte_perm(z, 0x64646464u, 0x4140);
  uint32_t hi = __byte_perm(z, 0x64646464u, 0x4342);
  const __half2 off = __halves2half2(__ushort_as_half((unsigned short)0x6480), __ushort_as_half((unsigned short)0x6480));
  __half2 a = __hsub2(*reinterpret_cast<__half2*>(&lo), off);
  __half2 b = __hsub2(*reinterpret_cast<__half2*>(&hi), off);
  return make_uint2(*reinterpret_cast<uint32_t*>(&a), *reinterpret_cast<uint32_t*>(&b));
}

}  // namespace tc
}  // namespace ckks
