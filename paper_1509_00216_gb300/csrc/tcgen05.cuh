// Device-side building blocks of the tensor-core kernels (sm_103a): bounded
// mbarrier waits, shared-memory operand descriptors, tcgen05 products and
// tensor-memory loads.
#pragma once
#include <cstdint>

#include "mpslcc.h"

namespace mpslcc {
namespace {

constexpr unsigned long long WAIT_NS = 2000000000ull;   // default bound on every mbarrier wait (2 s)
constexpr unsigned long long DRAIN_NS = 2000000000ull;  // bound on the drain of issued work after an abort

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n"
      ".reg .pred p;\n"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      "selp.u32 %0, 1, 0, p;\n"
      "}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// The same without the suspension.
__device__ __forceinline__ bool mbar_test_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n"
      ".reg .pred p;\n"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      "selp.u32 %0, 1, 0, p;\n"
      "}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

__device__ __forceinline__ unsigned long long gtimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Bounded wait; on expiry sets *err and returns false.  try_wait suspends the
// thread for longer than the few microseconds that one step's products take, so
// bounds of that order poll instead.
__device__ bool mbar_wait(uint64_t* bar, uint32_t parity, int* err, int code, unsigned long long limit_ns) {
  constexpr unsigned long long SHORT_NS = 10000;
  auto try_wait = [&]() {
    return limit_ns < SHORT_NS ? mbar_test_wait(bar, parity) : mbar_try_wait(bar, parity);
  };
  if (try_wait()) return true;
  const unsigned long long t0 = gtimer();
  for (;;) {
    if (try_wait()) return true;
    if (gtimer() - t0 > limit_ns) break;
    __nanosleep(32);
  }
  atomicExch(err, code);
  return false;
}

__device__ __forceinline__ uint64_t sdesc(const void* p) {
  // K-major operand tile, 128-byte swizzle: 8-row groups of 1024 bytes
  uint64_t a = smem_u32(p);
  uint64_t d = (a >> 4) & 0x3FFFull;
  d |= 1ull << 16;                    // leading byte offset (unused with swizzle)
  d |= (uint64_t)(1024 >> 4) << 32;   // stride byte offset
  d |= 1ull << 46;                    // descriptor version
  d |= 2ull << 61;                    // SWIZZLE_128B
  return d;
}

// The same for rows of ROW = 128 bytes, or of 64 bytes with 64-byte swizzle
// (8-row groups of 512 bytes).
template <int ROW>
__device__ __forceinline__ uint64_t sdesc_k(const void* p) {
  static_assert(ROW == 128 || ROW == 64, "operand row bytes");
  uint64_t d = ((uint64_t)smem_u32(p) >> 4) & 0x3FFFull;
  d |= 1ull << 16;
  d |= (uint64_t)(8 * ROW >> 4) << 32;
  d |= 1ull << 46;
  d |= (ROW == 128 ? 2ull : 4ull) << 61;   // SWIZZLE_128B or SWIZZLE_64B
  return d;
}

template <int PREC>
__device__ __forceinline__ uint32_t idesc(int M, int N) {
  uint32_t f = PREC == MPSLCC_BF16 ? 1u : 2u;  // BF16 or TF32 operands
  uint32_t d = 1u << 4;                        // FP32 accumulator
  d |= f << 7;
  d |= f << 10;
  d |= (uint32_t)(N >> 3) << 17;
  d |= (uint32_t)(M >> 4) << 24;
  return d;
}

// FP16 operands, FP32 accumulator (issued by umma<MPSLCC_BF16>: the same kind::f16).
__device__ __forceinline__ uint32_t idesc_f16(int M, int N) {
  return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

template <int PREC>
__device__ __forceinline__ void umma(uint32_t tmem, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
  if (PREC == MPSLCC_BF16)
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
        "l"(a), "l"(b), "r"(id), "r"(acc));
  else
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
        "l"(a), "l"(b), "r"(id), "r"(acc));
}

__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
        "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
        "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

}  // namespace
}  // namespace mpslcc
