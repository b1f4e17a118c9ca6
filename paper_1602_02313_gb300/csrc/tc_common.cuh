// Blackwell (sm_100a / sm_103a) tensor-core building blocks in inline PTX:
// tcgen05 MMA with operands in shared memory and FP32 accumulators in tensor
// memory (TMEM), mbarrier waits with an iteration budget, and the canonical
// K-major 128-byte-swizzled shared-memory operand layout.
#pragma once
#include <cstdint>

namespace gwi {
namespace tc {

// ---------------------------------------------------------------- error flags
// Device-side error codes written into a global int by bounded waits.
constexpr int kErrTimeout = 1;
// mbarrier polls before a wait gives up (each poll is a try_wait, which itself
// suspends for a hardware-defined interval): ~seconds, far beyond a healthy wait.
constexpr long long kWaitBudget = 1ll << 26;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// ---------------------------------------------------------------- mbarrier
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.shared::cta.b64 st, [%0];\n}" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// The same, suspended for up to about `ns` nanoseconds.
__device__ __forceinline__ bool mbar_try_wait_for(uint64_t* bar, uint32_t parity, uint32_t ns) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity), "r"(ns)
      : "memory");
  return ok != 0;
}
// Wait for the phase with the given parity to complete; gives up after the
// budget, records kErrTimeout in *err and returns false.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int* err) {
  for (long long i = 0; i < kWaitBudget; ++i)
    if (mbar_try_wait(bar, parity)) return true;
  if (err) atomicExch(err, kErrTimeout);
  return false;
}

// Wait for work a block has already issued before it frees its resources; twice the budget of
// mbar_wait, and false if even that runs out.
__device__ __forceinline__ bool mbar_wait_drain(uint64_t* bar, uint32_t parity) {
  for (long long i = 0; i < 2 * kWaitBudget; ++i)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
}

constexpr long long kDrainCycles = 4000000000ll;  // ~2 s at 2 GHz: waits for work already issued

// Bounded mbarrier wait shared by all roles of a block: gives up after `budget` clock cycles
// (the context's wait budget, ~2 s by default), or at once if another thread of the block has
// given up; on giving up it raises the block's abort flag and records kErrTimeout in *err.
__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* err,
                                         long long budget) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (true) {
    // The abort flag and the clock are looked at once in eight polls: every look is a load through the data
    // pipe that the MMAs read their operands by (20 % of it, with eight warps waiting and a look per poll).
#pragma unroll 1
    for (int i = 0; i < 8; ++i)
      if (mbar_try_wait_for(bar, parity, 1000)) return true;
    if (*abort_flag) return false;
    if (clock64() - t0 > budget) {
      *abort_flag = 1;
      if (err) atomicExch(err, kErrTimeout);
      return false;
    }
  }
}

// Wait for work this block has already issued (bulk copies into its shared memory, MMAs into its
// TMEM) before the block gives up its resources; ignores the abort flag, bounded by kDrainCycles.
__device__ __forceinline__ bool drain_bar(uint64_t* bar, uint32_t parity) {
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity))
    if (clock64() - t0 > kDrainCycles) return false;
  return true;
}

// Arrive on an mbarrier and add `bytes` to the transaction count it waits for.
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

// Bulk copy global -> shared (async proxy), completion counted in bytes on an mbarrier.
// Addresses 16-byte aligned, size a multiple of 16.
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// ---------------------------------------------------------------- fences
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// ---------------------------------------------------------------- TMEM
// Allocate ncols (power of two >= 32) TMEM columns; whole warp executes. The
// base address is written to *slot (shared memory).
__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// 32 lanes x 16 consecutive 32-bit columns: thread t of the warp gets lane (base lane + t).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// ---------------------------------------------------------------- descriptors
// Shared-memory matrix descriptor, K-major operand in the 128-byte swizzle
// layout: rows of 128 bytes (64 fp16 / bf16 values), the 16-byte chunks of row r
// permuted by XOR with (r mod 8), groups of 8 rows 1024 bytes apart (stride
// byte offset), tile base 1024-byte aligned. Fields: start address >> 4 (bits
// 0-13), leading byte offset >> 4 (16-29, unused for this layout: 1), stride
// byte offset >> 4 (32-45), descriptor version 1 (46-47), base offset 0
// (49-51), layout type 2 = 128-byte swizzle (61-63).
__device__ __forceinline__ uint64_t sdesc_sw128(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// Same for rows of 64 bytes (32 fp16 values) in the 64-byte swizzle layout:
// 16-byte chunk c of row r stored at chunk c ^ ((r >> 1) & 3), groups of 8
// rows 512 bytes apart, layout type 4 = 64-byte swizzle; tile base 512-byte aligned.
__device__ __forceinline__ uint64_t sdesc_sw64(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(512 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)4 << 61;
  return d;
}

// K-major operand without swizzle: core matrices of 8 rows x 16 bytes (128 contiguous bytes), the
// row groups of 8 one after another (stride byte offset 128), the next 8 K values `lbo` bytes on;
// layout type 0.
__device__ __forceinline__ uint64_t sdesc_none(uint32_t saddr, uint32_t lbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
  d |= (uint64_t)(lbo >> 4) << 16;
  d |= (uint64_t)(128 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// Instruction descriptor of tcgen05.mma kind::f16: D = FP32 (bits 4-5 = 1),
// A / B format (bits 7-9 / 10-12: 0 = fp16, 1 = bf16), negate A (bit 13),
// K-major A and B (bits 15, 16 = 0), N >> 3 (bits 17-22), M >> 4 (bits 24-28).
__host__ __device__ constexpr uint32_t idesc_f16(int M, int N, bool bf16, bool negA) {
  return (1u << 4) | ((bf16 ? 1u : 0u) << 7) | ((bf16 ? 1u : 0u) << 10) | ((negA ? 1u : 0u) << 13) |
         ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// D[tmem] (+)= A[smem] * B[smem]^T, issued by one thread.
__device__ __forceinline__ void mma_f16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                       uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrive on an mbarrier when all previously issued MMAs of this thread complete.
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

// For an issuer warp that runs converged: the waits and the operands' arithmetic are the whole warp's (so
// that they stay in uniform registers), and only the MMAs and commits stand in a branch of the one elected
// lane. With the whole role in a lane == 0 branch the descriptors are per-thread values that cost a
// register-to-uniform move each (measured 98 clocks per MMA of distinct descriptors, against the 48 that
// the operands of a 128 x 64 x 16 MMA take to read). The branch is needed: uniform registers are the
// warp's, so lanes that left a wait at different times must not both run through the issue code.
// a_lo, b_lo: low 32 bits of the descriptors (address and leading offset), desc_hi: the high 32 of both.
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t r;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}" : "=r"(r));
  return r;
}
__device__ __forceinline__ void mma_f16_lo(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t desc_hi, uint32_t idesc,
                                           uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n .reg .b64 a, b;\n mov.b64 a, {%1, %3};\n mov.b64 b, {%2, %3};\n"
      " setp.ne.b32 p, %5, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %4, p;\n}" ::"r"(d_tmem),
      "r"(a_lo), "r"(b_lo), "r"(desc_hi), "r"(idesc), "r"(accumulate)
      : "memory");
}

// Byte offset of element (r, k), k in [0, 64), 2-byte elements, in a K-major
// 128-byte-swizzled tile (row pitch 128 bytes).
__device__ __forceinline__ uint32_t sw128_off(uint32_t r, uint32_t k) {
  return r * 128u + ((((k >> 3) ^ (r & 7u)) << 4) | ((k & 7u) << 1));
}

// Byte offset of element (r, k), k in [0, 32), 2-byte elements, in a K-major
// 64-byte-swizzled tile (row pitch 64 bytes).
__device__ __forceinline__ uint32_t sw64_off(uint32_t r, uint32_t k) {
  return r * 64u + ((((k >> 3) ^ ((r >> 1) & 3u)) << 4) | ((k & 7u) << 1));
}

}  // namespace tc
}  // namespace gwi
