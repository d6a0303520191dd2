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

// Sum of six doubles (bit k of NEG: the k-th is subtracted), rounded once, on the
// integer pipes: the mantissas, shifted to the largest exponent with 7 bits below
// its last place, add up in 64 bits (some 120 instructions; 5 additions hold the
// FP64 pipe for 80 cycles of an SM).  Each term loses less than 2^-7 units in the
// last place of the largest, the sum is then rounded to the nearest double:
// against the exact sum at most 0.05 of those units more than one rounding, where
// a chain of five additions rounds five times.  As in the products, what lies below
// the normal range is zero.  `ok`: false where an operand is infinite, NaN or too
// large for the sum; the caller then adds them on the FP64 pipe.
template <unsigned NEG>
__host__ __device__ __forceinline__ uint64_t sum6_bits(const uint64_t (&x)[6], bool &ok) {
  uint32_t top = 0;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const uint32_t e = uint32_t(x[k] >> 32) & 0x7FF00000u;
    top = e > top ? e : top;
  }
  ok = top < (2042u << 20);
  uint64_t sum = 0;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const uint32_t h = uint32_t(x[k] >> 32), e = h & 0x7FF00000u;
    const uint64_t m = e ? ((x[k] & 0xFFFFFFFFFFFFFull) | (uint64_t(1) << 52)) << 7 : 0;
    const uint32_t d = (top - e) >> 20;
    const uint64_t t = m >> (d < 63 ? d : 63);
    const bool minus = (h >> 31) != ((NEG >> k) & 1u);
    sum = minus ? sum - t : sum + t;
  }
  const uint64_t neg = sum >> 63, a = neg ? 0 - sum : sum;
  if (a == 0) return 0;
#ifdef __CUDA_ARCH__
  const int z = __clzll((long long)a);
#else
  const int z = __builtin_clzll(a);
#endif
  const uint64_t n = a << z;
  const uint64_t r = (n >> 11) + ((n >> 10) & 1);
  const int e = int(top >> 20) + 3 - z;  // of the sum, less one (the mantissa's leading bit adds it)
  return e < 0 ? 0 : (neg << 63) | ((uint64_t(e) << 52) + r);
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

// not inlined: both sums would be formed and one chosen, five FP64 issues each time
// (Sedov 7-10, update per coarse step: 450 instead of 359 us)
__device__ __noinline__ double sum6_fp64(double a, double b, double c, double d, double e, double f) {
  return __dadd_rn(__dadd_rn(__dadd_rn(a, b), __dadd_rn(c, d)), __dadd_rn(e, f));
}
template <unsigned NEG>
__device__ __forceinline__ double sum6_int(double a, double b, double c, double d, double e, double f) {
  const uint64_t x[6] = {uint64_t(__double_as_longlong(a)), uint64_t(__double_as_longlong(b)),
                         uint64_t(__double_as_longlong(c)), uint64_t(__double_as_longlong(d)),
                         uint64_t(__double_as_longlong(e)), uint64_t(__double_as_longlong(f))};
  bool ok;
  const uint64_t s = sum6_bits<NEG>(x, ok);
  if (ok) return __longlong_as_double((long long)s);
  return sum6_fp64(NEG & 1 ? -a : a, NEG & 2 ? -b : b, NEG & 4 ? -c : c, NEG & 8 ? -d : d, NEG & 16 ? -e : e,
                   NEG & 32 ? -f : f);
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
