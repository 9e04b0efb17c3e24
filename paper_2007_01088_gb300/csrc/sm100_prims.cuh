// Inline-PTX primitives for sm_100-family (sm_103a) kernels: mbarriers with
// bounded waits, bulk copies, tensor-memory allocation and loads, and the
// shared-memory / instruction descriptors of tcgen05.mma (kind::f16).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace cc3 {
namespace sm100 {

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
               : "memory");
}

__device__ __forceinline__ void fence_barrier_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
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

// Whether the phase of this parity has completed, without waiting.
__device__ __forceinline__ bool mbar_test(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

__device__ __forceinline__ uint64_t globaltimer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

// Bounded wait: polls until the phase completes, another role has failed
// (*err set), or about `limit_ns` nanoseconds pass; then sets *err and returns
// false.  Every spin in these kernels goes through here.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, volatile int *err,
                                          uint64_t limit_ns = 2000000000ull) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = globaltimer_ns();
  uint32_t n = 0;
  while (!mbar_try_wait(bar, parity)) {
    if (*err) return false;
    if ((++n & 255u) == 0 && globaltimer_ns() - t0 > limit_ns) {
      *err = 1;
      return false;
    }
  }
  return true;
}

// Contiguous bulk copy global -> shared (16-byte aligned, size % 16 == 0),
// completion counted on `bar` (transaction bytes).
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes,
                                          uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

// Bounded wait with back-off (nanosleep between polls) for threads that may
// wait for a whole main loop.
__device__ __forceinline__ bool mbar_wait_sleep(uint64_t *bar, uint32_t parity, volatile int *err,
                                                uint64_t limit_ns = 2000000000ull) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = globaltimer_ns();
  while (!mbar_try_wait(bar, parity)) {
    if (*err) return false;
    __nanosleep(256);
    if (globaltimer_ns() - t0 > limit_ns) {
      *err = 1;
      return false;
    }
  }
  return true;
}

// Bounded wait that ignores the error word: for the exit path of a CTA that
// has given up, which must still let its own bulk copies and tensor-core
// operations finish (they write shared and tensor memory) before it frees
// them.  Returns false after about limit_ns.
__device__ __forceinline__ bool mbar_wait_quiet(uint64_t *bar, uint32_t parity,
                                                uint64_t limit_ns) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = globaltimer_ns();
  while (!mbar_try_wait(bar, parity)) {
    __nanosleep(128);
    if (globaltimer_ns() - t0 > limit_ns) return false;
  }
  return true;
}

// ---- tensor memory -----------------------------------------------------------
// whole warp: allocate ncols columns, address written to *dst_smem
__device__ __forceinline__ void tmem_alloc(uint32_t *dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                   smem_u32(dst_smem)),
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

// One lane of a converged warp, the same one each time (1 there, 0 elsewhere).
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t l;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(l));
  return l;
}

// D[tmem] (+)= A[smem] * B[smem]^T, issued by the lane whose `lead` is 1 of a
// converged warp: with the whole warp at the instruction the compiler keeps
// the descriptors in uniform registers, which tcgen05.mma reads.  Issued from
// under a single-thread branch the same instruction took ~80 clocks instead
// of ~49 (128 x 96 x 16, the time of the product itself).
// U is a usage hint for the A operand's collector buffer: U = 1 reads A from
// shared memory and keeps it (fill), U = 2 reuses the kept A (use), U = 3
// reuses it for the last time (lastuse), U = 0 reads A and does not keep it
// (discard, the default).  A run fill, use..., lastuse must pass the same A
// descriptor and be consecutive MMAs of this thread.
#define CC3_UMMA(HINT)                                                             \
  asm volatile(                                                                    \
      "{\n\t.reg .pred p, l;\n\t"                                                  \
      "setp.ne.b32 p, %4, 0;\n\t"                                                  \
      "setp.ne.b32 l, %5, 0;\n\t"                                                  \
      "@l tcgen05.mma.cta_group::1.kind::f16" HINT " [%0], %1, %2, %3, p;\n\t}" ::"r"( \
          d_tmem),                                                                 \
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(lead))
template <int U>
__device__ __forceinline__ void umma_f16_a(uint32_t lead, uint32_t d_tmem, uint64_t a_desc,
                                           uint64_t b_desc, uint32_t idesc,
                                           uint32_t accumulate) {
  if constexpr (U == 1) {
    CC3_UMMA(".collector::a::fill");
  } else if constexpr (U == 2) {
    CC3_UMMA(".collector::a::use");
  } else if constexpr (U == 3) {
    CC3_UMMA(".collector::a::lastuse");
  } else {
    CC3_UMMA("");
  }
}
#undef CC3_UMMA

// arrive on `bar` when every previously issued tcgen05.mma of this thread completes
__device__ __forceinline__ void umma_commit(uint64_t *bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(bar))
      : "memory");
}

// The same from the lane whose `lead` is 1 of a converged warp, without a branch.
__device__ __forceinline__ void umma_commit_a(uint32_t lead, uint64_t *bar) {
  asm volatile(
      "{\n\t.reg .pred l;\n\t"
      "setp.ne.b32 l, %1, 0;\n\t"
      "@l tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(
          smem_u32(bar)),
      "r"(lead)
      : "memory");
}

// 32 lanes x 4 columns of 32 bit
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, float *v) {
  uint32_t r[4];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr)
               : "memory");
#pragma unroll
  for (int i = 0; i < 4; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_wait_ld() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// ---- descriptors ---------------------------------------------------------------
// Shared-memory matrix descriptor, canonical K-major layout without swizzle:
// core matrices of 8 rows x 16 bytes, the two K halves 128 bytes apart and
// consecutive 8-row groups `sbo` bytes apart.
__device__ __forceinline__ uint64_t smem_desc_kmajor(uint32_t saddr, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);          // start address
  d |= (uint64_t)((128 >> 4) & 0x3FFF) << 16;       // leading byte offset (K direction)
  d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;       // stride byte offset (M/N direction)
  d |= (uint64_t)1 << 46;                           // descriptor version (sm100)
  return d;                                         // layout type 0: no swizzle
}

// Instruction descriptor: BF16 x BF16 -> FP32, K-major A and B, M x N.
__host__ __device__ __forceinline__ uint32_t idesc_bf16(int M, int N, int negA) {
  return (1u << 4)                         // D format F32
         | (1u << 7)                       // A format BF16
         | (1u << 10)                      // B format BF16
         | ((uint32_t)(negA ? 1 : 0) << 13)  // negate A
         | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

}  // namespace sm100
}  // namespace cc3
