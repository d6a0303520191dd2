"""The particle keys' Hilbert table (``csrc/hilbert_table.cuh``, compiled for the
host): aligned for the 32-bit words in which the kernel reads it, and walked two
levels per lookup it gives the oracle's index."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2607_20704_gb300", "csrc")
SRC = """
#include "hilbert_table.cuh"
static const amr::HilbertTable table = amr::hilbert_table();
extern "C" long table_align() { return alignof(amr::HilbertTable); }
extern "C" unsigned index_of(unsigned x, unsigned y, unsigned z, int bits) {
  unsigned key = 0, s = 0;
  if (bits & 1) {
    const int b = bits - 1;
    const unsigned v = table.one[((x >> b) & 1) << 2 | ((y >> b) & 1) << 1 | ((z >> b) & 1)];
    key = v & 7;
    s = v >> 6;
  }
  for (int b = (bits & ~1) - 2; b >= 0; b -= 2) {
    const unsigned v = table.two[s << 6 | ((x >> b) & 3) << 4 | ((y >> b) & 3) << 2 | ((z >> b) & 3)];
    key = key << 6 | (v & 63);
    s = v >> 6;
  }
  return key;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("hilbert")
    (d / "h.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "h.cpp"), "-o",
                    str(d / "h.so")], check=True)
    return ctypes.CDLL(str(d / "h.so"))


def test_the_table_is_aligned_for_its_word_reads(lib):
    assert lib.table_align() >= 4


@pytest.mark.parametrize("bits", range(1, 11))
def test_index_equals_the_oracle(lib, orc, bits):
    c = np.random.default_rng(bits).integers(0, 1 << bits, (2000, 3))
    c[:8] = [[i & 1, (i >> 1) & 1, i >> 2] for i in range(8)]
    c[8:16] = (1 << bits) - 1 - c[:8]
    for x, y, z in c.tolist():
        assert lib.index_of(x, y, z, bits) == orc.hilbert3(x, y, z, bits)
