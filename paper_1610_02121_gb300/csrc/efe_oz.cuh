// Device helpers and constants shared by the FP64 engine's kernels (efe_oz.cu,
// efe_oz_cell.cu): mbarriers, bulk copies, tcgen05 issue and the exact recombination
// of digit products.
#pragma once

#include <stdint.h>

namespace efe {

constexpr int OZ_S = 7;            // digits per operand
constexpr int OZ_M = 128;          // MMA rows
constexpr int OZ_KC = 16;          // K per chunk (one BF16 MMA)
constexpr int OZ_NACC = 5;         // accumulators: t = 2, 3, 4, 5 exact; t = 6..8 shared
constexpr uint32_t OZ_ASL = OZ_M * OZ_KC * 2;   // one A slice of a chunk, 4 KB
constexpr uint32_t OZ_TMEM_COLS = 512;
constexpr long long OZ_WAIT = 2000000000LL;     // bound of every wait, about one second of clocks

namespace {

__device__ __forceinline__ uint32_t su32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void bar_init(uint64_t* b, uint32_t n) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(b)), "r"(n) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint64_t* b) {
  asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(su32(b)) : "memory");
}
__device__ __forceinline__ bool bar_try(uint64_t* b, uint32_t parity) {
  uint32_t done = 0;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(su32(b)), "r"(parity)
      : "memory");
  return done != 0;
}
// one thread's bounded wait
__device__ __forceinline__ bool bar_wait(uint64_t* b, uint32_t parity) {
  const long long t0 = clock64();
  do {
    if (bar_try(b, parity)) return true;
  } while (clock64() - t0 < OZ_WAIT);
  return false;
}
// the same for a warp that goes on together.  Every lane has its own clock and its own view of
// the barrier, so the lanes vote: one that left alone could not take part in the warp's next
// collective step, and the others would wait for it there without a bound.
__device__ __forceinline__ bool warp_wait(uint64_t* b, uint32_t parity) {
  const long long t0 = clock64();
  do {
    if (__all_sync(0xffffffffu, bar_try(b, parity))) return true;
  } while (__all_sync(0xffffffffu, clock64() - t0 < OZ_WAIT));
  return false;
}
// the abort flag, one answer for the whole warp
__device__ __forceinline__ bool warp_aborted(const volatile int* flag) {
  return __any_sync(0xffffffffu, *flag != 0);
}
__device__ __forceinline__ void mma_bf16(uint32_t d, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
      "l"(a), "l"(b), "r"(id), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void bar_expect_tx(uint64_t* b, uint32_t bytes) {
  asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(su32(b)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(su32(dst)),
      "l"(src), "r"(bytes), "r"(su32(bar))
      : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* b) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(su32(b))
               : "memory");
}

// scale exponent of one value: |x| < 2^E (zero -> very small)
__device__ __forceinline__ int exp_of(double x) {
  const int ex = (int)((__double_as_longlong(x) >> 52) & 0x7FF);
  return ex == 0 ? -2000 : ex - 1022;
}

// x * 2^k in FP64, built from the bit pattern of x (exact; no FP64 arithmetic).
// Every accumulator value and error term here is zero or at least 2^-42 in
// magnitude (the smallest digit-product unit), so x is never subnormal;
// results outside the normal FP64 range take ldexp.
__device__ __forceinline__ double f32_scaled(float x, int k) {
  const uint32_t b = __float_as_uint(x);
  const int e = (int)((b >> 23) & 0xFFu);
  if (e == 0) return 0.0;
  const int E = e - 127 + 1023 + k;
  if (E < 1 || E > 2046) return ldexp((double)x, k);
  return __longlong_as_double((long long)(((unsigned long long)(b >> 31) << 63) | ((unsigned long long)E << 52) |
                                          ((unsigned long long)(b & 0x7FFFFFu) << 29)));
}

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}


}  // namespace
}  // namespace efe
