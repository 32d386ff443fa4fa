"""The kernels' shared index arithmetic (csrc/index.h), compiled for the host."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = """
#include "index.h"
extern "C" int64_t piece_row(int64_t q, int64_t n) { return tvcg::piece_row(q, n); }
extern "C" int arrivals_reached(uint32_t v, uint32_t want) { return tvcg::arrivals_reached(v, want); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("index")
    (d / "index.cpp").write_text(SOURCE)
    so = d / "index.so"
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2501_03121_gb300", "csrc"), str(d / "index.cpp"), "-o", str(so)], check=True)
    lib = ctypes.CDLL(str(so))
    lib.piece_row.argtypes = [ctypes.c_int64, ctypes.c_int64]
    lib.piece_row.restype = ctypes.c_int64
    lib.arrivals_reached.argtypes = [ctypes.c_uint32, ctypes.c_uint32]
    return lib


@pytest.mark.parametrize("n", [1, 2, 3, 2**31, 2**32 - 1, 2**32, 2**32 + 1, 2**32 + 5, 2**33, 3 * 2**33 + 1])
def test_row_of_a_piece(lib, n):
    # rows of 2^32 pieces and more: 2^34 FP32, 2^35 BF16 or 2^33 FP64 elements
    for q in (0, 1, n - 1, n, n + 1, 2 * n - 1, 2**32 - 1, 2**32, 2**32 + 7, 5 * n + n // 2):
        assert lib.piece_row(q, n) == q // n, q


@pytest.mark.parametrize("phase", [1, 2, 2**32 // 152, 2**32 // 152 + 1, 2 * 2**32 // 152 + 1])
def test_barrier_arrivals_past_the_word(lib, phase):
    blocks = 152
    want = phase * blocks
    for missing in (0, 1, blocks - 1, blocks):
        assert bool(lib.arrivals_reached((want - missing) % 2**32, want % 2**32)) == (missing == 0), missing
