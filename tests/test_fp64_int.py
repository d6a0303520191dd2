"""FP64 arithmetic on the integer pipes (``csrc/fp64_int.cuh``) on the CPU (the
header compiled for the host): products with the same bits as the native product
for normal operands with a normal product; the sum of three flux differences against
the exact one."""
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
#include <cstring>
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
extern "C" void sum_many(const double *a, double *c, unsigned char *ok, long n) {
  for (long i = 0; i < n; ++i) {
    uint64_t x[3], s;
    for (int k = 0; k < 3; ++k) {
      const double d = a[6 * i + 2 * k] - a[6 * i + 2 * k + 1];
      std::memcpy(&x[k], &d, 8);
    }
    bool o;
    s = amr::sum3_bits(x, o);
    std::memcpy(&c[i], &s, 8);
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


def _check_sums(lib, a, most):
    """The sum of the three (rounded) differences within half a unit in the last place
    of the result and 3 2^-8 units of the largest difference: what three terms lose.
    Refused only where they cancel to less than 2^-12 of the largest (2^-11 for the
    terms' own loss and the largest mantissa); `most`: the share that may."""
    n = len(a)
    x, c, ok = a.view(np.float64), np.zeros(n), np.zeros(n, np.uint8)
    lib.sum_many(_ptr(x), _ptr(c), _ptr(ok), ctypes.c_long(n))
    d = x[:, ::2] - x[:, 1::2]
    assert np.count_nonzero(ok == 0) <= most * n
    for r, o, t in zip(c, ok, d):
        exact, big = math.fsum(t), abs(t).max()
        if o:
            assert abs(math.fsum([r, *-t])) <= 0.5 * math.ulp(r) + 3 * 2.0 ** -8 * math.ulp(big), (t, r)
            assert abs(math.fsum([r, *-t])) <= 2.0 ** -45 * abs(exact), (t, r)
        else:
            assert big > 0 and abs(exact) <= 2.0 ** -11 * big, (t, r)


@pytest.mark.parametrize("spread", [0, 2, 30, 60, 500])
def test_sums_of_three_differences_round_once(lib, spread):
    rng = np.random.default_rng(5 + spread)
    n = 20000
    a = _bits(rng, 6 * n, spread).reshape(n, 6)
    a[::3, 1] = a[::3, 0]                              # differences that cancel
    a[1::3, 3] = a[1::3, 2] ^ np.uint64(1)             # nearly
    a[::5, 4:] &= np.uint64(1 << 63)                   # zeros of either sign
    a[:9] &= np.uint64(1 << 63)
    _check_sums(lib, a, 0.02)


@pytest.mark.parametrize("pair", [0, 2, 4])
def test_a_large_pair_takes_nothing_from_a_small_difference(lib, pair):
    """A flux that is (nearly) the same on both faces of one axis beside fluxes 2^40 to
    2^400 times smaller along the others: the small difference is what moves the cell."""
    rng = np.random.default_rng(11 + pair)
    n = 20000
    a = _bits(rng, 6 * n, 20).reshape(n, 6)
    a[:, pair] += rng.integers(60, 400, n).astype(np.uint64) << np.uint64(52)
    a[:, pair + 1] = a[:, pair]
    a[::7, pair + 1] += np.uint64(1)                   # one unit in the last place apart
    near = (pair + 2) % 6
    a[1::2, near + 1] = a[1::2, near] + rng.integers(0, 1 << 20, len(a[1::2])).astype(np.uint64)
    _check_sums(lib, a, 0.02)


@pytest.mark.parametrize("axes", [(0, 2), (0, 4), (2, 4)])
def test_differences_that_cancel_are_left_to_the_fp64_pipe(lib, axes):
    """Two axes whose differences are (nearly) opposite beside a small third."""
    rng = np.random.default_rng(17 + sum(axes))
    n = 20000
    a = _bits(rng, 6 * n, 20).reshape(n, 6)
    p, q = axes
    a[:, [p, p + 1]] += (rng.integers(42, 400, n).astype(np.uint64) << np.uint64(52))[:, None]
    a[:, q], a[:, q + 1] = a[:, p + 1], a[:, p]
    a[::7, q] ^= np.uint64(1)
    _check_sums(lib, a, 1.0)


def test_sums_at_the_ends_of_the_range(lib):
    a = np.zeros((9, 6))
    a[0, 2], a[1, 5], a[2, 0] = np.inf, np.nan, 2.0 ** 1020  # refused
    a[3, 1], a[4, 2:4] = 5e-324, (2.0 ** -1022, 5e-324)      # a result below the normal range: refused
    a[5, 3], a[6, 2] = 2.0 ** -1022, -(2.0 ** -960)          # exact
    a[7, :] = 2.0 ** 1018
    a[8, :] = 5e-324
    c, ok = np.zeros(9), np.zeros(9, np.uint8)
    lib.sum_many(_ptr(a), _ptr(c), _ptr(ok), ctypes.c_long(9))
    assert ok.tolist() == [0, 0, 0, 0, 0, 1, 1, 1, 1]
    assert c[5:].tolist() == [-(2.0 ** -1022), -(2.0 ** -960), 0.0, 0.0]
