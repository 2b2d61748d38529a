// Fifth-generation tensor-core helpers (sm_103a): mbarriers with bounded waits,
// shared-memory and instruction descriptors of tcgen05.mma, TMEM loads and
// stores.  All operands are bf16, K-major; accumulators are fp32 in TMEM.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace mpnn {

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      "selp.b32 %0, 1, 0, p;\n}"
      : "=r"(done)
      : "r"(bar), "r"(parity)
      : "memory");
  return done != 0u;
}

// Waits for the phase of the given parity, a bounded number of tries (a try
// itself waits for a while): false if it did not come, or if another thread gave
// up (*failed).  A thread that gives up says so in *failed.
constexpr int kMbarTries = 1 << 18;
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* failed,
                                          int tries) {
  for (int i = 0; i < tries; ++i) {
    if (mbar_try(bar, parity)) return true;
    if (*failed) return false;
  }
  *failed = 1;
  return false;
}

// Waits for the phase whether or not another thread gave up: for the end of
// operations that must not outlive what they read and write.
__device__ __forceinline__ void mbar_drain(uint32_t bar, uint32_t parity) {
  for (int i = 0; i < kMbarTries && !mbar_try(bar, parity); ++i) {
  }
}

__device__ __forceinline__ void fence_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Shared-memory matrix descriptors (K-major).  Swizzled: rows of 128 bytes (64
// bf16), 16-byte piece c of row r at piece c ^ (r & 7), eight rows (1024 bytes)
// apart from the next eight; a chunk of 16 k further is 32 bytes further.  Plain:
// 16 k as two pieces, each piece's rows 16 bytes apart, `lead` bytes from the
// first piece's rows to the second's.
__device__ __forceinline__ uint64_t desc_sw128(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32) |
         (1ull << 46) | (2ull << 61);
}
__device__ __forceinline__ uint64_t desc_plain(uint32_t addr, uint32_t lead) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(lead >> 4) << 16) |
         ((uint64_t)(128 >> 4) << 32) | (1ull << 46);
}

// kind::f16 instruction descriptor: bf16 operands, fp32 accumulator, M x N
constexpr uint32_t tc_idesc(uint32_t M, uint32_t N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((N >> 3) << 17) | ((M >> 4) << 24);
}

// D (+)= A B^T over 16 k; one thread issues it
__device__ __forceinline__ void tc_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc,
                                       bool add) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(add ? 1 : 0)
      : "memory");
}
// the products issued so far arrive at the barrier when they are done
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
      : "memory");
}

// 16 columns of the warp's 32 TMEM lanes: v[c] of lane l
__device__ __forceinline__ void tc_ld16(uint32_t (&v)[16], uint32_t addr) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15}, [%16];\n"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
        "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
        "=r"(v[14]), "=r"(v[15])
      : "r"(addr)
      : "memory");
}
// one value to `cols` consecutive columns (cols is the same in all lanes)
__device__ __forceinline__ void tc_fill(uint32_t addr, uint32_t v, int cols) {
  for (; cols >= 8; cols -= 8, addr += 8)
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%1], {%0,%0,%0,%0,%0,%0,%0,%0};" ::"r"(v),
                 "r"(addr)
                 : "memory");
  if (cols & 4) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%1], {%0,%0,%0,%0};" ::"r"(v), "r"(addr)
                 : "memory");
    addr += 4;
  }
  if (cols & 2) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%1], {%0,%0};" ::"r"(v), "r"(addr)
                 : "memory");
    addr += 2;
  }
  if (cols & 1)
    asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%1], {%0};" ::"r"(v), "r"(addr)
                 : "memory");
}
__device__ __forceinline__ void tc_wait_st() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// All 512 columns of TMEM (one block an SM), by one warp; the address goes to
// shared memory.
__device__ __forceinline__ void tc_alloc(uint32_t dst, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst),
               "r"(cols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
__device__ __forceinline__ void tc_dealloc(uint32_t addr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(cols));
}

}  // namespace mpnn
