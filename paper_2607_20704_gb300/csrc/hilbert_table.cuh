// hilbert_table.cuh -- 3-D Hilbert indices by a table of states.
//
// 3-D Hilbert index of (x, y, z), x most significant: the same curve as
// hilbert_index (Skilling's transposed construction) as a state machine.  What
// the construction has done to the lower bits of the three axes when it comes to
// a level -- exchanged them (6 orders), inverted them (8 masks) -- and the
// Gray-code parity of the levels above are one of 96 states; a state and the
// level's three bits give an octal digit and the next state.  Two levels per
// lookup, from a table in shared memory: the key of a 256^3 cell takes 4 lookups
// and some 50 instructions instead of 150 (the keys' kernel, bound by its integer
// work, took 142 us for 16.8 M FP32 particles; 77 us now).
#pragma once
#include <stddef.h>
#include <stdint.h>

namespace amr {

struct alignas(16) HilbertTable {  // read as words of 32 bits
  uint16_t two[96 * 64];  // [state][x1 x0 y1 y0 z1 z0]: two digits, next state << 6
  uint16_t one[96 * 8];   // [state][x y z]: digit, next state << 6
};
constexpr int hilbert_step(int state, int x, int y, int z, int &digit) {
  int g = state & 1, inv[3] = {(state >> 1) & 1, (state >> 2) & 1, (state >> 3) & 1};
  // axis held by each slot: the order's two-step code (first slot, swap of the rest)
  const int o = state >> 4, first = o >> 1;
  int ax[3] = {first, (first + 1) % 3, (first + 2) % 3};
  if (o & 1) {
    const int t = ax[1];
    ax[1] = ax[2];
    ax[2] = t;
  }
  const int raw[3] = {x, y, z};
  const int a0 = raw[ax[0]] ^ inv[0], a1 = raw[ax[1]] ^ inv[1], a2 = raw[ax[2]] ^ inv[2];
  if (a0) inv[0] ^= 1;
  for (int k = 1; k < 3; ++k) {
    if (k == 1 ? a1 : a2) {
      inv[0] ^= 1;
    } else {
      const int t = ax[0], u = inv[0];
      ax[0] = ax[k];
      inv[0] = inv[k];
      ax[k] = t;
      inv[k] = u;
    }
  }
  const int b1 = a1 ^ a0, b2 = a2 ^ b1;
  digit = (a0 ^ g) << 2 | (b1 ^ g) << 1 | (b2 ^ g);
  g ^= b2;
  return (ax[0] << 1 | (ax[1] != (ax[0] + 1) % 3)) << 4 | inv[2] << 3 | inv[1] << 2 | inv[0] << 1 | g;
}
constexpr HilbertTable hilbert_table() {
  HilbertTable t{};
  for (int s = 0; s < 96; ++s) {
    for (int q = 0; q < 8; ++q) {
      int d = 0;
      const int n = hilbert_step(s, q >> 2, (q >> 1) & 1, q & 1, d);
      t.one[8 * s + q] = uint16_t(n << 6 | d);
    }
    for (int q = 0; q < 64; ++q) {
      int d1 = 0, d0 = 0;
      const int m = hilbert_step(s, q >> 5, (q >> 3) & 1, (q >> 1) & 1, d1);
      const int n = hilbert_step(m, (q >> 4) & 1, (q >> 2) & 1, q & 1, d0);
      t.two[64 * s + q] = uint16_t(n << 6 | d1 << 3 | d0);
    }
  }
  return t;
}

}  // namespace amr
