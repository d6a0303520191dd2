// cic_weights.cuh -- the 8 FP64 Cloud-in-Cell contributions of a particle on the
// integer pipes.
//
// A particle's contributions m wx wy wz cost 22 FP64 instructions (the source
// cell, 6 weights and 14 products), which bounded every FP64 deposit at 16
// cycles of an SM per instruction and warp; the integer pipes were idle.  Here a
// weight is a fixed-point fraction: x n - 1/2 has at most 63 bits after the point
// for every x that matters (the bits of x n below 2^-63 belong to x below 2^-10 /
// n, whose weights are near 1/2).  The weights are those of the definition in
// FP64, f = s - floor(s) and 1 - f, each rounded to 53 bits; weights and mass are
// then 64-bit mantissas, a product keeps the upper 64 bits (relative error below
// 2^-60 after three), and each contribution is rounded to FP64 once: within 0.51
// units in the last place of m wx wy wz, where three FP64 products are within 1.5.
//
// Positions in [0, 1) and masses that are zero or of magnitude 2^-400 .. 2^400;
// callers take the FP64 pipe for anything else.
#pragma once
#include <stdint.h>
#ifndef FP64_INT_HOST
#include <cuda_runtime.h>
#endif

namespace amr {

__host__ __device__ __forceinline__ uint64_t cic_mulhi(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return uint64_t((unsigned __int128)a * b >> 64);
#endif
}
__host__ __device__ __forceinline__ int cic_clz(uint64_t a) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)a);
#else
  return a ? __builtin_clzll(a) : 64;
#endif
}

// a non-negative number m 2^(e - 64), m normalised (its top bit set) or zero
struct CicNum {
  uint64_t m;
  int e;
};

// a fraction f 2^-63 <= 1 rounded to 53 significant bits (to nearest, ties to even)
__host__ __device__ __forceinline__ uint64_t cic_round53(uint64_t f) {
  const int drop = 11 - cic_clz(f);
  if (drop <= 0) return f;
  const uint64_t low = (uint64_t(1) << drop) - 1;
  return (f + (low >> 1) + ((f >> drop) & 1)) & ~low;
}

// the source cell floor(x n - 1/2) (n = 2^bits, unmasked) and the weights of the
// cells i0 and i0 + 1 of a position in [0, 1), given by its bits
__host__ __device__ __forceinline__ int cic_axis_int(uint64_t x, int bits, CicNum (&w)[2]) {
  const int E = int(x >> 52);
  const uint64_t M = E ? (x & 0xFFFFFFFFFFFFFull) | (uint64_t(1) << 52) : 0;  // subnormal: 0
  // x n + 1/2 with 63 bits after the point: M 2^sh + 2^62 in (hi, lo)
  const int sh = E - 1075 + bits + 63;
  uint64_t lo, hi = 0;
  if (sh >= 0) {  // at most bits + 10
    lo = M << sh;
    hi = sh ? M >> (64 - sh) : 0;
  } else {  // x below 2^(-10 - bits): f is 1/2 and more; bits shifted out only turn a tie
    lo = sh > -64 ? (M >> -sh) | ((M << (64 + sh)) != 0) : M != 0;
  }
  const uint64_t l2 = lo + (uint64_t(1) << 62);
  hi += l2 < lo;
  const uint64_t f = cic_round53(l2 & 0x7FFFFFFFFFFFFFFFull), g = cic_round53((uint64_t(1) << 63) - f);
  const int zf = cic_clz(f), zg = cic_clz(g);
  w[1].m = f << (zf & 63);
  w[1].e = 1 - zf;
  w[0].m = g << (zg & 63);
  w[0].e = 1 - zg;
  return int((hi << 1) | (l2 >> 63)) - 1;
}

// floor(x n): the cell that contains the position
__host__ __device__ __forceinline__ int cic_floor_int(uint64_t x, int bits) {
  const int E = int(x >> 52), sh = 1075 - E - bits;  // x < 1: sh is at least 53 - bits
  return E && sh < 64 ? int(((x & 0xFFFFFFFFFFFFFull) | (uint64_t(1) << 52)) >> sh) : 0;
}

// |m| n^3 (n^3 = 2^(3 bits)) of a mass given by its bits
__host__ __device__ __forceinline__ CicNum cic_mass_int(uint64_t m, int bits) {
  const int E = int(m >> 52) & 0x7FF;
  return CicNum{E ? (m << 11) | (uint64_t(1) << 63) : 0, E - 1022 + 3 * bits};
}

__host__ __device__ __forceinline__ CicNum cic_mul(CicNum a, CicNum b) {
  return CicNum{cic_mulhi(a.m, b.m), a.e + b.e};  // not normalised: at most one bit lost
}

// to the nearest double, with the sign bit given
__host__ __device__ __forceinline__ uint64_t cic_round(CicNum a, uint64_t sign) {
  const int z = cic_clz(a.m);
  const uint64_t m = a.m << (z & 63);
  const uint64_t r = (m >> 11) + ((m >> 10) & 1);
  const int E = a.e - z + 1022;  // a = 1.frac 2^(E - 1023)
  return a.m && E > 0 ? sign | ((uint64_t(E - 1) << 52) + r) : sign;
}

// the contributions ((m n^3 wx) wy) wz, corner c = cx + 2 cy + 4 cz, as bits
__host__ __device__ __forceinline__ void cic_weights_int(uint64_t x, uint64_t y, uint64_t z, uint64_t m, int bits,
                                                         int &i, int &j, int &k, uint64_t (&w)[8]) {
  CicNum wx[2], wy[2], wz[2], b[4];
  i = cic_axis_int(x, bits, wx);
  j = cic_axis_int(y, bits, wy);
  k = cic_axis_int(z, bits, wz);
  const CicNum ms = cic_mass_int(m, bits);
  const uint64_t sign = m & (uint64_t(1) << 63);
  for (int q = 0; q < 4; ++q) b[q] = cic_mul(cic_mul(ms, wx[q & 1]), wy[q >> 1]);
  for (int c = 0; c < 8; ++c) w[c] = cic_round(cic_mul(b[c & 3], wz[c >> 2]), sign);
}

#ifndef FP64_INT_HOST
// positions in [0, 1) (not -0) and a mass of the range above
__device__ __forceinline__ bool cic_in_range(double x, double y, double z, double m) {
  const uint32_t one = 0x3FF00000u, h = uint32_t(__double2hiint(m)) & 0x7FFFFFFFu;
  return uint32_t(__double2hiint(x)) < one && uint32_t(__double2hiint(y)) < one && uint32_t(__double2hiint(z)) < one &&
         (h - (uint32_t(1023 - 400) << 20) < (uint32_t(800) << 20) || m == 0.0);
}
#endif

}  // namespace amr
