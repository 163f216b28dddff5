// Blackwell (sm_103a) tensor-core building blocks in inline PTX: tensor-memory
// allocation, tcgen05.mma with A in tensor memory or shared memory and B in
// shared memory, completion through mbarriers, tensor-memory loads and stores,
// and bulk (TMA) copies between global and shared memory.
//
// Conventions used by the kernels built on these:
//  * A shared-memory operand is stored K-major without swizzling, in 8-row x
//    16-byte core matrices: element (r, k) of an R x K 16-bit matrix sits at
//    byte (r / 8) * SBO + (k / 8) * 128 + (r % 8) * 16 + (k % 8) * 2, with
//    SBO = (K / 8) * 128 (an 8-row group keeps all its K chunks together).
//  * A tensor-memory A operand (M = 128 rows) keeps row m in lane m and two
//    16-bit values per 32-bit column, k = 2c in the low half and 2c + 1 in the
//    high half of column c.
//  * The FP32 accumulator D of an M = 128 product keeps row m in lane m and
//    column n in column n.
//  * Every wait polls a bounded number of times and reports failure instead of
//    hanging; callers turn that into an error flag.
#pragma once

#include <cstdint>

namespace dgx {
namespace tc {

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Shared-memory matrix descriptor (no swizzle, K-major): start address,
// leading byte offset (between K-adjacent core matrices), stride byte offset
// (between 8-row groups), descriptor version 1.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= uint64_t((saddr & 0x3FFFFu) >> 4);
  d |= uint64_t((lbo >> 4) & 0x3FFFu) << 16;
  d |= uint64_t((sbo >> 4) & 0x3FFFu) << 32;
  d |= uint64_t(1) << 46;
  return d;
}

// Instruction descriptor of kind::f16 with FP32 accumulation, both operands
// K-major: FP16 (bf16 = false) or BF16 inputs, shape M x N.
__host__ __device__ constexpr uint32_t idesc_f16(int M, int N, bool bf16) {
  return (1u << 4) | ((bf16 ? 1u : 0u) << 7) | ((bf16 ? 1u : 0u) << 10) | (uint32_t(N >> 3) << 17) |
         (uint32_t(M >> 4) << 24);
}

__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t ncols) {  // one full warp
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_addr(slot)),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {  // the allocating warp
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(taddr), "r"(ncols) : "memory");
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }
// generic-proxy shared-memory writes -> visible to the async proxy (MMA operand reads, bulk stores)
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

// D (tensor memory) [+]= A (tensor memory) x B (shared memory)^T
__device__ __forceinline__ void mma_ts(uint32_t d, uint32_t a, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d),
      "r"(a), "l"(bdesc), "r"(idesc), "r"(acc)
      : "memory");
}
// D (tensor memory) [+]= A (shared memory) x B (shared memory)^T
__device__ __forceinline__ void mma_ss(uint32_t d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc)
      : "memory");
}
// the mbarrier receives one arrival once every earlier MMA of this thread has completed
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                   smem_addr(bar))
               : "memory");
}

__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_addr(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_init_fence() {
  asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_addr(b)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t globaltimer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %globaltimer;\n" : "=l"(t));
  return t;
}
// Warp-collective wait for the phase of parity `parity` to complete, bounded
// in time (default one second, far beyond any tile's work): false if it gave
// up. The votes keep the warp converged for the aligned instructions after it.
constexpr uint64_t kWaitLimitNs = 1000000000ull;
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, uint64_t limit_ns = kWaitLimitNs) {
  if (__all_sync(0xffffffffu, mbar_try(b, parity))) return true;  // most waits: no clock is read
  const uint64_t t0 = globaltimer_ns();
  for (;;) {
    if (__all_sync(0xffffffffu, mbar_try(b, parity))) return true;
    if (__any_sync(0xffffffffu, globaltimer_ns() - t0 > limit_ns)) return false;
  }
}
// A wait that gave up sets the block's abort flag, and every later wait then
// returns at once: all warps run to the end of their loops (their named
// barriers stay matched) and the block ends.
__device__ __forceinline__ bool aborted(volatile int* flag) { return __any_sync(0xffffffffu, *flag != 0); }
// (False if it gave up, here or before.)
__device__ __forceinline__ bool wait_or_abort(uint64_t* b, uint32_t parity, volatile int* abort_flag) {
  if (aborted(abort_flag)) return false;
  if (mbar_wait(b, parity)) return true;
  *abort_flag = 1;
  return false;
}
// Before a block ends: its last copies and products have to be done also when a wait
// gave up, or they would reach memory that is another block's by then (bounded too).
__device__ __forceinline__ void wait_done(uint64_t* b, uint32_t parity, volatile int* abort_flag) {
  if (!mbar_wait(b, parity)) *abort_flag = 1;
}
__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
  asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.shared::cta.b64 st, [%0];\n}\n" ::"r"(smem_addr(b)) : "memory");
}
__device__ __forceinline__ void bar_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(threads) : "memory");
}
// arm the barrier for `bytes` of bulk-copy traffic (one arrival)
__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
  asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}\n" ::"r"(
                   smem_addr(b)),
               "r"(bytes)
               : "memory");
}
// bulk copy global -> shared (16-byte aligned addresses, size a multiple of 16),
// completion counted on the mbarrier
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
          smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}

// tensor-memory loads / stores of the calling warp's 32 lanes (lane base =
// 32 * (warp % 4) in bits 16..31 of the address), consecutive 32-bit columns
__device__ __forceinline__ void tmem_ld8(uint32_t a, uint32_t (&v)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(a)
               : "memory");
}
__device__ __forceinline__ void tmem_ld4(uint32_t a, uint32_t (&v)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
               : "r"(a)
               : "memory");
}
__device__ __forceinline__ void tmem_ld1(uint32_t a, uint32_t& v) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];\n" : "=r"(v) : "r"(a) : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void tmem_st8(uint32_t a, const uint32_t (&v)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};\n" ::"r"(a), "r"(v[0]),
               "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory"); }

// x * 2^e for |e| <= 252 (two exact power-of-two factors)
__device__ __forceinline__ float ldexp2(float x, int e) {
  const int e1 = e / 2, e2 = e - e1;
  return x * __int_as_float((127 + e1) << 23) * __int_as_float((127 + e2) << 23);
}
// exponent e with |x| < 2^e for finite nonzero x; -200 for zero
__device__ __forceinline__ int exp_of(float x) {
  const int E = (__float_as_int(x) >> 23) & 0xff;
  return E == 0 ? (x == 0.0f ? -200 : -126) : E - 126;
}

}  // namespace tc
}  // namespace dgx
