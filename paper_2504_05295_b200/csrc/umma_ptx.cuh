// tcgen05 / TMEM / mbarrier instructions shared by the contraction engine and the data-flow Cholesky, sm_100a only.
#pragma once

#include "dion_common.cuh"

namespace dion {
namespace umma {

constexpr int BM = 128;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void fence_barrier_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_alloc(uint32_t slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
template <bool BF16>
__device__ __forceinline__ void umma(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  if (BF16) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
  } else {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
  }
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

// Shared-memory matrix descriptor.
// K-major (any type) and MN-major bf16: 128-byte swizzle (16-byte units XORed with
//   the row index mod 8); rows of 128 bytes, 8-row groups 1024 bytes apart.
// MN-major TF32: the only layout the hardware takes is the 128-byte swizzle with a
//   32-byte base: atoms of 4 k-rows x 128 bytes, 32-byte units XORed with the row
//   index mod 4; groups of 4 k-rows are 512 bytes apart.
// For MN-major operands `lbo_bytes` is the distance between consecutive 128-byte
// chunks along M/N (32 fp32 or 64 bf16 elements).
template <bool BF16>
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr, bool mn_major, uint32_t lbo_bytes) {
  const bool base32 = mn_major && !BF16;
  const uint64_t lbo = mn_major ? (uint64_t)(lbo_bytes >> 4) : 1ull;
  const uint64_t sbo = base32 ? (512 >> 4) : (1024 >> 4);
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= lbo << 16;
  d |= sbo << 32;
  d |= 1ull << 46;                      // descriptor version of sm_100
  d |= (base32 ? 1ull : 2ull) << 61;    // SWIZZLE_128B_BASE32B or SWIZZLE_128B
  return d;
}

// Instruction descriptor: fp32 accumulate, TF32 or BF16 operands, M = 128, N = BN.
// f16 (with bf16): the 16-bit operands are IEEE half values (kind::f16 takes either format)
__device__ __forceinline__ uint32_t make_idesc(bool bf16, bool a_mn, bool b_mn, int bn, int bm = BM, bool f16 = false) {
  uint32_t d = 0;
  const uint32_t fmt = bf16 ? (f16 ? 0u : 1u) : 2u;   // 0 F16, 1 BF16 (kind::f16); 2 TF32 (kind::tf32)
  d |= 1u << 4;                         // D format: F32
  d |= fmt << 7;                        // A format
  d |= fmt << 10;                       // B format
  d |= (a_mn ? 1u : 0u) << 15;
  d |= (b_mn ? 1u : 0u) << 16;
  d |= (uint32_t)(bn >> 3) << 17;
  d |= (uint32_t)(bm >> 4) << 24;
  return d;
}

}  // namespace umma
}  // namespace dion
