"""The FP64 Cloud-in-Cell contributions on the integer pipes
(``csrc/cic_weights.cuh``, compiled for the host): the source cell of the
definition, and each contribution within 0.51 units in the last place of the
exact product m wx wy wz n^3 of the FP64 weights f = s - floor(s) and 1 - f
(each product keeps 64 bits, 2^-60 after three, and one rounding follows)."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2607_20704_gb300", "csrc")
SRC = """
#include <cstdint>
#define __host__
#define __device__
#define __forceinline__ inline
#define FP64_INT_HOST
#include "cic_weights.cuh"
extern "C" void weights(const uint64_t *p, uint64_t m, int bits, int *cell, uint64_t *w) {
  uint64_t v[8];
  amr::cic_weights_int(p[0], p[1], p[2], m, bits, cell[0], cell[1], cell[2], v);
  for (int c = 0; c < 8; ++c) w[c] = v[c];
  for (int d = 0; d < 3; ++d) cell[3 + d] = amr::cic_floor_int(p[d], bits);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("cic_weights")
    (d / "w.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "w.cpp"), "-o",
                    str(d / "w.so")], check=True)
    return ctypes.CDLL(str(d / "w.so"))


def _positions(rng, n):
    """In [0, 1): spread, tiny, on cell faces and centres and beside them, near 1."""
    x = rng.random(3)
    for d in range(3):
        k = rng.integers(0, 7)
        if k == 1:
            x[d] *= 2.0 ** -float(rng.integers(0, 70))
        elif k == 2:
            x[d] = np.floor(x[d] * n) / n
        elif k >= 3:
            x[d] = (np.floor(x[d] * n) + 0.5) / n
            if k >= 4:
                x[d] = np.nextafter(x[d], (2.0, -1.0)[k & 1])
        if k == 6:
            x[d] = 1.0 - rng.random() * 2.0 ** -float(rng.integers(0, 53))
    return np.clip(x, 0.0, np.nextafter(1.0, 0.0))


@pytest.mark.parametrize("bits", [1, 2, 5, 7, 10, 15])
def test_contributions_are_rounded_once(lib, bits):
    rng = np.random.default_rng(bits)
    n = 1 << bits
    for it in range(600):
        x = _positions(rng, n)
        m = float(np.exp(3 * rng.standard_normal())) * (-1 if it % 7 == 0 else 1) * (it % 41 != 0)
        cell, w = np.zeros(6, np.int32), np.zeros(8, np.uint64)
        lib.weights(x.view(np.uint64).ctypes.data_as(ctypes.c_void_p), ctypes.c_uint64(int(np.float64(m).view(np.uint64))),
                    bits, cell.ctypes.data_as(ctypes.c_void_p), w.ctypes.data_as(ctypes.c_void_p))
        wt = []
        for d in range(3):
            s = Fraction(float(x[d])) * n - Fraction(1, 2)
            i0 = s.numerator // s.denominator
            assert cell[d] == i0 and cell[3 + d] == int(np.floor(x[d] * n))
            f = float(s - i0)  # correctly rounded
            wt.append((Fraction(1.0 - f), Fraction(f)))
        for c in range(8):
            want = Fraction(m) * n ** 3 * wt[0][c & 1] * wt[1][(c >> 1) & 1] * wt[2][c >> 2]
            got = float(w[c:c + 1].view(np.float64)[0])
            ulp = Fraction(float(np.spacing(abs(float(want))))) if want else Fraction(0)
            assert abs(Fraction(got) - want) <= Fraction(51, 100) * ulp, (x, m, c)
