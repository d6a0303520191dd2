// fp64_int.cuh -- FP64 products on the integer pipes.
//
// GB300 issues one FP64 instruction of a warp in 16 cycles of an SM (2 lanes
// per clock, 1/64 of the FP32 rate), while the integer pipes of the FP64-bound
// kernels are nearly idle.  A double product is 4 multiply-adds of 32-bit
// halves and some 30 integer instructions: measured at 15.2 against 19.2
// cycles per warp and SM for the native multiply, and the two overlap (4
// integer products beside 4 FMAs took 79.5 cycles, 4 FMAs alone 76.9), so a
// kernel that takes its plain products here leaves the FP64 pipe to the FMAs.
//
// mul_int gives the correctly rounded product (round to nearest, ties to even),
// the bits of the native multiply, for normal operands whose product is normal.
// mul_int0 is for operands that may be tiny or zero: subnormal operands count
// as zero, and a product below 2^-1022 is zero; mul_fp64_0 is the same on the
// FP64 pipe.  Neither takes infinities, NaN or products of 2^1024 and more:
// callers make sure of that and use the FP64 pipe otherwise.
#pragma once
#ifndef FP64_INT_HOST  // (the CPU test compiles mul_bits alone)
#include <cuda_runtime.h>
#endif
#include <stdint.h>

namespace amr {

// the product of two doubles, given as bit patterns; ZERO: they or their
// product may lie below the normal range (see above)
template <bool ZERO>
__host__ __device__ __forceinline__ uint64_t mul_bits(uint64_t x, uint64_t y) {
  const uint32_t ah = uint32_t(x >> 32), bl = uint32_t(y), bh = uint32_t(y >> 32);
  // A = mantissa of x (53 bits) 2^11, B = mantissa of y: A B in [2^115, 2^117)
  const uint64_t A = (x << 11) | (uint64_t(1) << 63);
  const uint32_t Al = uint32_t(A), Ah = uint32_t(A >> 32), Bh = (bh & 0xFFFFFu) | 0x100000u;
  const uint64_t t0 = uint64_t(Al) * bl;
  const uint64_t t1 = uint64_t(Ah) * bl + uint32_t(t0 >> 32);
  const uint64_t t2 = uint64_t(Al) * Bh + uint32_t(t1);
  const uint64_t H = uint64_t(Ah) * Bh + uint32_t(t1 >> 32) + uint32_t(t2 >> 32);
  // the upper 64 bits H in [2^51, 2^53), below them Lh and Ll; shifted so that
  // 54 bits remain (53 and the rounding bit), the others in `rest`
  const uint32_t Hl = uint32_t(H), Hh = uint32_t(H >> 32), Lh = uint32_t(t2), Ll = uint32_t(t0);
  const uint32_t c = Hh >> 20;  // the product of the mantissas is 2 or more (0 or 1)
  const uint32_t sh = 2u - c;
#ifdef __CUDA_ARCH__
  const uint32_t h1 = __funnelshift_l(Hl, Hh, sh), h0 = __funnelshift_l(Lh, Hl, sh);
#else
  const uint32_t h1 = (Hh << sh) | (Hl >> (32 - sh)), h0 = (Hl << sh) | (Lh >> (32 - sh));
#endif
  const uint32_t rest = (Lh << sh) | Ll;
  const uint64_t r = (((uint64_t(h1) << 32) | h0) + 1u) >> 1;
  uint32_t m = uint32_t(r);
  if (rest == 0 && (h0 & 1u)) m &= ~1u;  // half-way: to the even neighbour
  const uint32_t ea = ah & 0x7FF00000u, eb = bh & 0x7FF00000u, e = ea + eb + (c << 20) - (1024u << 20);
  const uint32_t sign = (ah ^ bh) & 0x80000000u;
  uint32_t hi = (uint32_t(r >> 32) + e) | sign;
  if (ZERO && (ea == 0 || eb == 0 || int32_t(e) < 0)) {
    hi = sign;
    m = 0;
  }
  return (uint64_t(hi) << 32) | m;
}

// a + b + c of doubles given as bit patterns, rounded once, on the integer pipes: the
// mantissas, shifted to the largest exponent with 8 bits below its last place, add up
// in 64 bits.  Each term loses less than 2^-8 units in the last place of the largest;
// a rounded addition loses up to half a unit of its result, and two are saved.  `ok`:
// false where an operand is infinite, NaN or too large for the sum, where the result
// lies below the normal range, or where the terms cancel to less than 2^-12 of the
// largest (what they lost is then more than 2^-46 of the result, and two of them may
// cancel exactly beside a small third); the caller then adds on the FP64 pipe.
__host__ __device__ __forceinline__ uint64_t sum3_bits(const uint64_t (&x)[3], bool &ok) {
  constexpr uint32_t one = 1u << 20;  // one step of the exponent in a double's upper half
  uint32_t e[3], top = one;           // (subnormal numbers have the smallest normal exponent)
  uint64_t m[3], sum = 0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const uint32_t field = uint32_t(x[k] >> 32) & 0x7FF00000u;
    m[k] = ((x[k] & 0xFFFFFFFFFFFFFull) | (field ? uint64_t(1) << 52 : 0)) << 8;
    e[k] = field ? field : one;
    top = e[k] > top ? e[k] : top;
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const uint32_t d = (top - e[k]) >> 20;
    const uint64_t t = m[k] >> (d < 63 ? d : 63);
    sum = x[k] >> 63 ? sum - t : sum + t;
  }
  const uint64_t neg = sum >> 63, a = neg ? 0 - sum : sum;
  ok = top < 2042u * one && (a >> 48 || (m[0] | m[1] | m[2]) == 0);  // the largest is 2^60 and more
  if (a == 0) return 0;
#ifdef __CUDA_ARCH__
  const int z = __clzll((long long)a);
#else
  const int z = __builtin_clzll(a);
#endif
  const uint64_t n = a << z;
  const uint64_t r = (n >> 11) + ((n >> 10) & 1);
  const int es = int(top >> 20) + 2 - z;  // of the sum, less one (the mantissa's leading bit adds it)
  ok = ok && es >= 0;
  return (neg << 63) | ((uint64_t(uint32_t(es)) << 52) + r);
}

#ifndef FP64_INT_HOST
__device__ __forceinline__ double mul_int(double x, double y) {
  return __longlong_as_double(
      (long long)mul_bits<false>(uint64_t(__double_as_longlong(x)), uint64_t(__double_as_longlong(y))));
}
__device__ __forceinline__ double mul_int0(double x, double y) {
  return __longlong_as_double(
      (long long)mul_bits<true>(uint64_t(__double_as_longlong(x)), uint64_t(__double_as_longlong(y))));
}
// a value below the normal range is zero
__device__ __forceinline__ double normal_or_zero(double x) {
  const int h = __double2hiint(x);
  return (h & 0x7FF00000) ? x : __hiloint2double(h & int(0x80000000u), 0);
}
__device__ __forceinline__ double mul_fp64_0(double x, double y) {
  return normal_or_zero(__dmul_rn(normal_or_zero(x), normal_or_zero(y)));
}

// not inlined: both sums would be formed and one chosen
__device__ __noinline__ double sum3_fp64(double a, double b, double c) { return __dadd_rn(__dadd_rn(a, b), c); }
__device__ __forceinline__ double sum3_int(double a, double b, double c) {
  const uint64_t x[3] = {uint64_t(__double_as_longlong(a)), uint64_t(__double_as_longlong(b)),
                         uint64_t(__double_as_longlong(c))};
  bool ok;
  const uint64_t s = sum3_bits(x, ok);
  return ok ? __longlong_as_double((long long)s) : sum3_fp64(a, b, c);
}

// x in [2^-E, 2^E)
template <int E>
__device__ __forceinline__ bool within(double x) {
  return uint32_t(__double2hiint(x)) - (uint32_t(1023 - E) << 20) < (uint32_t(2 * E) << 20);
}
// |x| < 2^E
template <int E>
__device__ __forceinline__ bool below(double x) {
  return (uint32_t(__double2hiint(x)) & 0x7FFFFFFFu) < (uint32_t(1023 + E) << 20);
}
#endif

}  // namespace amr
