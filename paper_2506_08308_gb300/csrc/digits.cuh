// Exact products on the tensor cores from integer digits.
//
// A column (or row) of floating-point values is written in fixed point
// relative to its largest magnitude, x = X 2^(e - c), and the integer X is
// cut into balanced 8-bit digits, X = sum_k d_k 2^(8 (ND-1-k)) with -128 <=
// d_k <= 128.  A digit is exact in FP16, the product of two digits has at
// most 15 bits, and the FP32 accumulator of tcgen05.mma (kind::f16) adds
// such products without rounding as long as the sum stays below 2^24, that
// is for (summed rows) x (digit pairs) <= 1024.  All digit pairs (i, j) of
// equal i + j have equal weight and share one accumulator.  Pairs with i + j
// >= ND lie below the last digit; with seven digits the first such weight is
// kept as well, the others are left out.  What is lost is the cut of the inputs,
// at most a unit of X (bits below are dropped, a negative value is one too low).
#pragma once

#include <cuda_fp16.h>

#include "common.cuh"

namespace bdg {

constexpr long long MMA_WAIT_LIMIT = 1LL << 22;  // polls of an MMA barrier before giving up

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor (no swizzle): start address, byte offset
// between core matrices along K (lbo) and along M or N (sbo), version 1
__device__ __forceinline__ uint64_t mma_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) | (1ull << 46);
}
// instruction descriptor of kind::f16: D FP32, A and B FP16; MN-major
// operands when `mn` (bits 15, 16), N >> 3 at bit 17, M >> 4 at bit 24
__device__ __forceinline__ uint32_t mma_idesc_f16(int M, int N, bool a_mn, bool b_mn) {
  return (1u << 4) | ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}
__device__ __forceinline__ void mma_f16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, bool accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"((uint32_t)accumulate)
      : "memory");
}
// one lane of a converged warp (the same one every time)
__device__ __forceinline__ bool elect_one() {
  uint32_t r;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(r));
  return r != 0;
}
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ bool mma_wait(uint64_t* bar, uint32_t parity) {
  for (long long it = 0; it < MMA_WAIT_LIMIT; ++it) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}
__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t ncols) {  // one warp
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_free(uint32_t tmem, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// four accumulator columns of the thread's lane
__device__ __forceinline__ void tmem_ld4(uint32_t addr, float (&v)[4]) {
  uint32_t u[4];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3])
               : "r"(addr)
               : "memory");
#pragma unroll
  for (int q = 0; q < 4; ++q) v[q] = __uint_as_float(u[q]);
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// ---------------------------------------------------------------------------
// fixed point
// ---------------------------------------------------------------------------
// An integer in the order of |x|, zero for zero only; an FP64 value's exponent
// field is in its bits 20..30, an FP32 value's in 23..30.
__device__ __forceinline__ unsigned magnitude(double x) {
  return ((unsigned)__double2hiint(x) & 0x7FFFFFFFu) | min((unsigned)__double2loint(x), 1u);
}
__device__ __forceinline__ unsigned magnitude(float x) { return __float_as_uint(x) & 0x7FFFFFFFu; }
// Biased FP64 exponent of the largest value of a column from its magnitude: 0
// for zeros only, 1 (897 for FP32) where all are subnormal, 2047 for an
// infinity or NaN.
template <typename R>
__device__ __forceinline__ int biased_exponent(unsigned m) {
  if (m == 0) return 0;
  if constexpr (sizeof(R) == 8) return max((int)(m >> 20), 1);
  return m >= 0x7F800000u ? 2047 : max((int)(m >> 23), 1) + 896;
}
// Zeros and subnormals have no implicit bit, which to_fixed sets for all: it
// falls below the last digit unless the column's largest value is very small.
// Such a column (magnitude below LIMIT) is multiplied by 2^GROW first.
template <typename R> struct Tiny;
template <> struct Tiny<double> {
  static constexpr unsigned LIMIT = 128u << 20;
  static constexpr int GROW = 200;
  static constexpr double FACTOR = 0x1p200;
};
template <> struct Tiny<float> {
  static constexpr unsigned LIMIT = 64u << 23;
  static constexpr int GROW = 64;
  static constexpr float FACTOR = 0x1p64f;
};
template <typename R>
__device__ __forceinline__ bool is_tiny(unsigned m) {
  return m - 1u < Tiny<R>::LIMIT - 1u;   // (a column of zeros is not)
}

// Fixed point of x relative to 2^(emax - 1022), emax the largest biased
// exponent of its column, which is not a tiny one.  e20 holds emax in bits
// 20..30 (the bits below may be anything, as in a magnitude).
// ND = 6, 7: the value's 53 bits with two more below, |X| < 2^55, x = X
//   2^(emax - 1077), as seven bytes; six digits leave out the lowest byte,
//   which the bias of 0x80 per byte turns into rounding to nearest.
// ND = 4: |X| < 2^30, x = X 2^(emax - 1052), rounded down.
// Zeros and subnormals come out as at most one unit.  A column of zeros has
// emax = 0, whose X is finite and means nothing: the caller leaves it out.
template <int ND> struct Fixed { typedef long long I; };
template <> struct Fixed<4> { typedef int I; };

template <int ND>
__device__ __forceinline__ typename Fixed<ND>::I to_fixed(double x, int e20) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  const int sm = hi >> 31, d = (e20 - (hi & 0x7FF00000)) >> 20;
  if constexpr (ND == 4) {
    const int m = ((int)(__funnelshift_l((unsigned)lo, (unsigned)hi, 9) & 0x1FFFFFFFu) | 0x20000000) ^ sm;
    return m >> min(d, 31);
  } else {
    const unsigned mh = ((hi & 0xFFFFF) | 0x100000) ^ sm, ml = lo ^ sm;
    // the two bits below are the sign's, so that a negative value is off by one unit of X at most
    const unsigned h2 = __funnelshift_l(ml, mh, 2), l2 = __funnelshift_l((unsigned)sm, ml, 2);
    return (long long)(((unsigned long long)h2 << 32) | l2) >> min(d, 63);
  }
}
template <int ND>
__device__ __forceinline__ typename Fixed<ND>::I to_fixed(float x, int e20) {
  static_assert(ND == 4, "FP32 values have 24 bits");
  const int b = __float_as_int(x), sm = b >> 31;
  const int d = (e20 - (((b >> 3) & 0x0FF00000) + (896 << 20))) >> 20;
  const int m = (((b << 6) & 0x1FFFFFFF) | 0x20000000) ^ sm;
  return m >> min(d, 31);
}
// binary exponent of the unit of the top digits' product
template <int ND>
__host__ __device__ constexpr int product_unit(int ea, int eb) {
  return ND == 4 ? ea + eb - 2 * 1052 + 48 : ea + eb - 2 * 1077 + 96;
}

// The digits of two values as FP16 pairs (first value in the low half).
// Adding 128 to every digit makes the bytes of X + 0x80..80 the digits plus
// 128 (the top one up to 256, so 9 bits are taken there); 0x6400 | u is the
// FP16 number 1024 + u.
template <int ND>
__device__ __forceinline__ void digit_pairs(typename Fixed<ND>::I x, typename Fixed<ND>::I y, uint32_t (&d)[ND]) {
  const __half2 off = __half2half2(__ushort_as_half(0x6480));  // 1024 + 128
  auto put = [&](int k, uint32_t w) {
    const __half2 h = __hsub2(*reinterpret_cast<__half2*>(&w), off);
    d[k] = *reinterpret_cast<const uint32_t*>(&h);
  };
  // selectors put the wanted byte of the first value in byte 0 and that of
  // the second in byte 2
  if constexpr (ND == 4) {
    const unsigned a = (unsigned)x + 0x80808080u, b = (unsigned)y + 0x80808080u;
#pragma unroll
    for (int k = 0; k < 4; ++k) put(k, (__byte_perm(a, b, (3 - k) | ((7 - k) << 8)) & 0x00FF00FFu) | 0x64006400u);
  } else {
    const unsigned long long u = (unsigned long long)x + 0x80808080808080ull;
    const unsigned long long v = (unsigned long long)y + 0x80808080808080ull;
    const unsigned ul = (unsigned)u, uh = (unsigned)(u >> 32), vl = (unsigned)v, vh = (unsigned)(v >> 32);
    put(0, __byte_perm(uh, vh, 0x7632) | 0x64006400u);
    put(1, (__byte_perm(uh, vh, 0x0501) & 0x00FF00FFu) | 0x64006400u);
    put(2, (__byte_perm(uh, vh, 0x0400) & 0x00FF00FFu) | 0x64006400u);
#pragma unroll
    for (int k = 3; k < ND; ++k) put(k, (__byte_perm(ul, vl, (6 - k) | ((10 - k) << 8)) & 0x00FF00FFu) | 0x64006400u);
  }
}

}  // namespace bdg
