// Fifth-generation tensor-core primitives (sm_100-family tcgen05, TMEM, bulk
// copies) as inline PTX, for the surrogate network's inference kernel.
//
// Operand layout used throughout: K-major BF16 tiles with the 128-byte
// swizzle.  A tile of R rows and 64 K-elements (one "slab") occupies R * 128
// bytes: row r is 128 contiguous bytes (eight 16-byte chunks) and chunk j of
// row r is stored at chunk position j ^ (r % 8).  Slabs are 1024-byte aligned,
// so consecutive groups of 8 rows (1024 bytes) form one swizzle atom.  Longer
// K is a sequence of slabs.
#pragma once

#include <cstdint>
#include <cuda_bf16.h>

namespace casim_dev {

// byte offset of element (r, k) of a K-major swizzled slab sequence with R rows per slab
__host__ __device__ __forceinline__ uint32_t sw128_offset(int R, int r, int k) {
  const int slab = k >> 6, kk = k & 63;
  const int chunk = (kk >> 3) ^ (r & 7);
  return (uint32_t)(slab * R * 128 + r * 128 + chunk * 16 + (kk & 7) * 2);
}

// byte offset of element (r, k), k < 16, of a K-major tile of 16 K-elements
// with the 32-byte swizzle: row r is 32 contiguous bytes, its two 16-byte
// chunks exchanged in every second group of four rows
__host__ __device__ __forceinline__ uint32_t sw32_offset(int r, int k) {
  return (uint32_t)(r * 32 + (((k >> 3) ^ ((r >> 2) & 1)) << 4) + (k & 7) * 2);
}
// its matrix descriptor: 256 bytes between 8-row groups
__device__ __forceinline__ uint64_t umma_desc_sw32(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)(16u >> 4) << 16;
  d |= (uint64_t)(256u >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)6 << 61;
  return d;
}

// shared-memory matrix descriptor: start address, leading-dimension offset
// (unused by swizzled K-major layouts, set to 16 bytes), stride-dimension
// offset 1024 bytes (between 8-row groups), descriptor version 1, 128-byte
// swizzle
__device__ __forceinline__ uint64_t umma_desc_sw128(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)(16u >> 4) << 16;
  d |= (uint64_t)(1024u >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// MN-major tiles with the 128-byte swizzle: a block of 64 rows (m or n) and 64
// k is 64 k-rows of 128 contiguous bytes (eight 16-byte chunks of 8 rows
// each), chunk j of k-row k at chunk position j ^ (k % 8); further blocks of
// 64 rows follow 8192 bytes apart (the leading-dimension offset), groups of 8
// k-rows 1024 bytes apart (the stride-dimension offset).
__device__ __forceinline__ uint32_t sw128_mn_offset(int r, int k) {
  return (uint32_t)((r >> 6) * 8192 + k * 128 + (((r >> 3) & 7) ^ (k & 7)) * 16);
}
__device__ __forceinline__ uint64_t umma_desc_mn_sw128(uint32_t saddr) {
  return (umma_desc_sw128(saddr) & ~((uint64_t)0x3FFF << 16)) | (uint64_t)(8192u >> 4) << 16;
}

// instruction descriptor, kind::f16: BF16 A and B (K-major, or both MN-major),
// FP32 accumulator, M x N
__host__ __device__ constexpr uint32_t umma_idesc_bf16(int M, int N, bool mn_major = false) {
  return (1u << 4)            // D format: F32
         | (1u << 7)          // A format: BF16
         | (1u << 10)         // B format: BF16
         | (mn_major ? 3u << 15 : 0u)
         | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// Programmatic dependent launch: the next kernel of the stream may start its
// prologue (pdl_trigger) and waits for this one's completion before it touches
// memory (pdl_wait).
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// all prior tcgen05 operations of this thread arrive on the mbarrier when done
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// 32 lanes x 32 columns of 32-bit accumulators: this thread's lane, columns col..col+31
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float v[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// 32 lanes x 16 columns of 32-bit accumulators: this thread's lane, columns col..col+15
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float v[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// the same for 32 columns without the wait; tmem_wait32 names the registers,
// so that nothing that uses them can come before it
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t r[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_wait32(uint32_t r[32]) {
  asm volatile(
      "tcgen05.wait::ld.sync.aligned;"
      : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
        "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]),
        "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]),
        "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
      :
      : "memory");
}

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void bar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_fence_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void bar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool bar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
               : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// every wait on a barrier gives up after this long (or `spins` polls)
constexpr uint64_t kWaitLimitNs = 2000000000ull;

// bounded wait for phase `parity`; false if it gave up.  The first try comes
// before the timer is read.
__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity, unsigned spins) {
  if (bar_try(bar, parity)) return true;
  const uint64_t t0 = global_ns();
  for (unsigned i = 0; i < spins; ++i) {
    if (bar_try(bar, parity)) return true;
    if ((i & 63u) == 63u && global_ns() - t0 > kWaitLimitNs) return false;
  }
  return false;
}
// bounded wait that also gives up early once `abort` is set by another thread
__device__ __forceinline__ bool bar_wait_or_abort(uint32_t bar, uint32_t parity, unsigned spins,
                                                  const volatile int *abort, uint64_t limit_ns = kWaitLimitNs) {
  if (bar_try(bar, parity)) return true;
  const uint64_t t0 = global_ns();
  for (unsigned i = 0; i < spins; ++i) {
    if (bar_try(bar, parity)) return true;
    if ((i & 63u) == 63u && (*abort || global_ns() - t0 > limit_ns)) return false;
  }
  return false;
}

// The bounded wait on its own: one thread waits on an mbarrier that nothing
// arrives at (phase 0 never completes) through the waits' own code, gives up
// after limit_ns, and records that in the error word as the kernels do.  No
// copy, MMA or tensor memory is involved, so there is nothing to drain.
__global__ void k_wait_selftest(uint64_t limit_ns, unsigned *err, unsigned long long *elapsed) {
  __shared__ alignas(8) unsigned long long s_bar;
  __shared__ int s_abort;
  const uint32_t bar = smem_addr(&s_bar);
  if (threadIdx.x == 0) {
    s_abort = 0;
    bar_init(bar, 1);
    bar_fence_init();
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const uint64_t t0 = global_ns();
    const bool ok = bar_wait_or_abort(bar, 0u, 0xffffffffu, &s_abort, limit_ns);
    *elapsed = global_ns() - t0;
    if (!ok) atomicOr(err, 4u);
  }
}
// 1-D bulk copy global -> shared, completing on the mbarrier (16-byte aligned, size a multiple of 16)
__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

__device__ __forceinline__ float tanh_approx(float x) {
  float y;
  asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

}  // namespace casim_dev
