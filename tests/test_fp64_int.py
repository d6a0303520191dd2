"""FP64 arithmetic on the integer pipes (``csrc/fp64_int.cuh``) on the CPU (the
header compiled for the host): products with the same bits as the native product
for normal operands with a normal product; sums of six against the exact sum."""
import ctypes
import math
import os
import subprocess

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
#include "fp64_int.cuh"
extern "C" void mul_many(const uint64_t *a, const uint64_t *b, uint64_t *c, long n) {
  for (long i = 0; i < n; ++i) c[i] = amr::mul_bits<false>(a[i], b[i]);
}
extern "C" void mul_many0(const uint64_t *a, const uint64_t *b, uint64_t *c, long n) {
  for (long i = 0; i < n; ++i) c[i] = amr::mul_bits<true>(a[i], b[i]);
}
extern "C" void sum_many(const uint64_t *a, uint64_t *c, unsigned char *ok, long n) {
  for (long i = 0; i < n; ++i) {
    const uint64_t x[6] = {a[6 * i], a[6 * i + 1], a[6 * i + 2], a[6 * i + 3], a[6 * i + 4], a[6 * i + 5]};
    bool o;
    c[i] = amr::sum6_bits<0x2A>(x, o);
    ok[i] = o;
  }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fp64_int")
    (d / "m.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "m.cpp"), "-o",
                    str(d / "m.so")], check=True)
    return ctypes.CDLL(str(d / "m.so"))


def _ptr(x):
    return x.ctypes.data_as(ctypes.c_void_p)


def _bits(rng, n, spread):
    """Doubles of exponents within +-spread: random mantissas, mantissas with
    few set bits (exact and half-way products) and with long runs of ones."""
    m = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    keep = rng.integers(0, 53, n).astype(np.uint64)
    low = (np.uint64(1) << keep) - np.uint64(1)
    kind = rng.integers(0, 3, n)
    m = np.where(kind == 1, m & ~low, np.where(kind == 2, m | low, m)) & np.uint64((1 << 52) - 1)
    e = rng.integers(1023 - spread, 1023 + spread + 1, n).astype(np.uint64)
    s = rng.integers(0, 2, n).astype(np.uint64)
    return (s << np.uint64(63)) | (e << np.uint64(52)) | m


@pytest.mark.parametrize("seed,spread", [(0, 1), (1, 30), (2, 500)])
def test_products_equal_the_native_ones(lib, seed, spread):
    rng = np.random.default_rng(seed)
    n = 1 << 20
    a, b = _bits(rng, n, spread), _bits(rng, n, spread)
    # squares, powers of two and neighbours of one: the edges of the rounding
    a[:8] = np.array([1.0, 2.0, -1.0, 1 + 2.0 ** -52, 2 - 2.0 ** -52, 0.5, 1.5, 1 + 2.0 ** -26]).view(np.uint64)
    b[:64] = np.repeat(a[:8], 8)
    a[8:64] = np.tile(a[:8], 7)
    c = np.zeros(n, np.uint64)
    lib.mul_many(_ptr(a), _ptr(b), _ptr(c), ctypes.c_long(n))
    want = a.view(np.float64) * b.view(np.float64)
    assert np.all(np.abs(want) >= 2.0 ** -1022) and np.all(np.isfinite(want))
    assert np.array_equal(c, want.view(np.uint64))
    lib.mul_many0(_ptr(a), _ptr(b), _ptr(c), ctypes.c_long(n))
    assert np.array_equal(c, want.view(np.uint64))


def test_products_below_the_normal_range_are_zero(lib):
    rng = np.random.default_rng(3)
    n = 1 << 18
    a, b, c = _bits(rng, n, 700), _bits(rng, n, 700), np.zeros(n, np.uint64)
    a[::7] &= np.uint64(1 << 63)                      # signed zeros
    a[3::7] &= np.uint64((1 << 63) | ((1 << 52) - 1))  # subnormal operands
    x, y = a.view(np.float64), b.view(np.float64)
    with np.errstate(over="ignore", under="ignore"):
        want = np.where(np.abs(x) < 2.0 ** -1022, np.copysign(0.0, x), x) * y
    want = np.where(np.abs(want) < 2.0 ** -1022, np.copysign(0.0, want), want)
    ok = np.isfinite(want) & (np.abs(want) != 2.0 ** -1022)  # (rounded up from below: either is right)
    lib.mul_many0(_ptr(a), _ptr(b), _ptr(c), ctypes.c_long(n))
    assert ok.sum() > n // 2 and np.count_nonzero(want[ok] == 0) > n // 4
    assert np.array_equal(c[ok], want.view(np.uint64)[ok])


@pytest.mark.parametrize("spread", [0, 2, 30, 60, 500])
def test_sums_of_six_round_once(lib, spread):
    rng = np.random.default_rng(5 + spread)
    n = 20000
    a = _bits(rng, 6 * n, spread).reshape(n, 6)
    a[::3, 1] = a[::3, 0]                              # differences that cancel
    a[1::3, 3] = a[1::3, 2] ^ np.uint64(1)             # nearly
    a[::5, 4:] &= np.uint64(1 << 63)                   # zeros of either sign
    a[:9] &= np.uint64(1 << 63)
    x, c, ok = a.view(np.float64), np.zeros(n, np.uint64), np.zeros(n, np.uint8)
    lib.sum_many(_ptr(a), _ptr(c), _ptr(ok), ctypes.c_long(n))
    assert ok.all()
    got = c.view(np.float64)
    for r, t in zip(got, x * [1, -1, 1, -1, 1, -1]):
        # five terms lose less than 2^-7 units in the last place of the largest each
        assert abs(math.fsum([r, *-t])) <= 0.5 * math.ulp(r) + 5 * 2.0 ** -7 * math.ulp(abs(t).max())


def test_sums_at_the_ends_of_the_range(lib):
    a = np.zeros((7, 6))
    a[0, 2], a[1, 5], a[2, 0] = np.inf, np.nan, 2.0 ** 1020  # refused
    a[3, 1] = 5e-324                                         # below the normal range: zero
    a[4, 3], a[5, 2] = 2.0 ** -1022, -(2.0 ** -960)          # exact
    a[6, :] = 2.0 ** 1018
    c, ok = np.zeros(7, np.uint64), np.zeros(7, np.uint8)
    lib.sum_many(_ptr(a), _ptr(c), _ptr(ok), ctypes.c_long(7))
    assert ok.tolist() == [0, 0, 0, 1, 1, 1, 1]
    assert c.view(np.float64)[3:].tolist() == [0.0, -(2.0 ** -1022), -(2.0 ** -960), 0.0]
