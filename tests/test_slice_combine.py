"""The combination of the seven diagonal sums of the FP64 tensor-core kernels as they do it
(csrc/oz_combine.h, compiled here for the host; CPU only), over the range of two merged chunks,
K = 128: diagonals 0 and 1 as FP32 bit patterns with an offset, 2 to 6 as integers."""
import ctypes
import os
import struct
import subprocess

import numpy as np
import pytest

from conftest import ROOT

SOURCE = """
#include "oz_combine.h"
extern "C" long long combine(const unsigned* f, const int* d) {
  return chol::oz_high(chol::oz_low(d[4], d[5], d[6]), f[0], f[1], d[2], d[3]);
}
"""
OFFSET = np.float32(12582912.0)  # 1.5 * 2^23
BOUND = [128 * (d + 1) * 2**14 for d in range(7)]  # K = 128, |s_p| <= 2^7


@pytest.fixture(scope="module")
def combine(tmp_path_factory):
    d = tmp_path_factory.mktemp("combine")
    src, so = d / "combine.cpp", d / "combine.so"
    src.write_text(SOURCE)
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-fwrapv", "-shared", "-fPIC", "-I",
                           os.path.join(ROOT, "paper_2202_09288_gb300", "csrc"), str(src), "-o", str(so)])
    f = ctypes.CDLL(str(so)).combine
    f.restype = ctypes.c_longlong

    def run(D):
        bits = [struct.unpack("<I", struct.pack("<f", float(np.float32(x) + OFFSET)))[0] for x in D[:2]]
        return f((ctypes.c_uint * 2)(*bits), (ctypes.c_int * 7)(*D))

    return run


def test_ranges():
    assert max(BOUND) < 2**24       # every partial sum is an exact FP32 integer
    assert max(BOUND[:2]) <= 2**22  # and these two keep it beside the offset


def test_combination(combine):
    rng = np.random.default_rng(11)
    cases = [[0] * 7, BOUND, [-b for b in BOUND]]
    cases += [[s * b if i == d else 0 for i in range(7)] for d, b in enumerate(BOUND) for s in (1, -1)]
    cases += [[int(rng.integers(-b, b + 1)) for b in BOUND] for _ in range(20000)]
    cases += [[int(rng.choice([-b, -1, 0, 1, b])) for b in BOUND] for _ in range(3000)]
    for D in cases:
        low = sum(D[d] << (8 * (6 - d)) for d in range(4, 7))
        w = (sum(D[d] << (8 * (3 - d)) for d in range(4)) << 17) + ((low + 64) >> 7)
        assert abs(w) < 1.01 * 2**62 and combine(D) == w, D
