"""Integer arithmetic of the FP64 tensor-core kernels' 8-bit slices, restated on the host (CPU
only): rounding to 55 bits, seven balanced digits (least significant first: one from the 64-bit
integer, then three from each 24-bit half) stored as bf16, and the combination of the seven
diagonal sums, three of them as integers and four as FP32 bit patterns with a folded offset."""
import struct

import numpy as np

MASK64 = (1 << 64) - 1
OFF = 0x4B400000
HI_BIAS = (-(OFF * ((1 << 17) + (1 << 25) + (1 << 33) + (1 << 41)))) % (1 << 64) >> 32
BOUND = [64 * (d + 1) * 2**14 for d in range(7)]  # K = 64, |s_p| <= 2^7


def fixed(x, e):
    """x 2^(55 - e) rounded half away from zero, from the bits of x."""
    bits = struct.unpack("<q", struct.pack("<d", x))[0]
    exb = (bits >> 52) & 0x7FF
    if exb == 0:
        return 0
    mant = (bits & ((1 << 52) - 1)) | (1 << 52)
    sh = exb - 1020 - e
    m = mant << sh if sh >= 0 else ((mant + (1 << (-sh - 1))) >> -sh if sh >= -53 else 0)
    return -m if bits < 0 else m


def digits(R):
    d = [0] * 7
    d[6] = ((R + 128) & 255) - 128
    r = (R - d[6]) >> 8
    lo, hi = r & 0xFFFFFF, r >> 24
    for p in (5, 4, 3):
        d[p] = ((lo + 128) & 255) - 128
        lo = (lo - d[p]) >> 8
    assert lo in (0, 1) and abs(hi) < 2**31
    hi += lo
    for p in (2, 1):
        d[p] = ((hi + 128) & 255) - 128
        hi = (hi - d[p]) >> 8
    d[0] = hi
    return d


def combine(D):
    f = [(OFF + x) & 0xFFFFFFFF for x in D[:4]]
    lo = ((D[4] * 65536 + (D[5] * 256 + (D[6] + 64))) >> 7) & MASK64
    w = (f[3] * 131072 + lo) & MASK64
    w = (f[2] * 33554432 + w) & MASK64
    w = (w + (((f[1] * 2 + f[0] * 512 + HI_BIAS) & 0xFFFFFFFF) << 32)) & MASK64
    return w - (1 << 64) if w >> 63 else w


def test_fixed_point_error():
    rng = np.random.default_rng(3)
    for x in list(rng.uniform(-1, 1, 3000) * 2.0 ** rng.integers(-80, 1, 3000)) + [0.0, 1 - 2.0**-53]:
        m = fixed(float(x), 0)
        assert abs(m) <= 2**55
        assert abs(m - float(x) * 2.0**55) <= 0.5  # exact in FP64: |x| 2^55 has at most 56 bits kept


def test_digits():
    rng = np.random.default_rng(7)
    cases = [0, 1, -1, 2**55, -(2**55), 2**55 - 1, 2**47, -(2**47), 127, 128, -128, -129, 2**31, 2**32 - 1]
    cases += [int(x) for x in rng.integers(-(2**55), 2**55, size=20000, dtype=np.int64)]
    cases += [int(s) * int(rng.integers(0, 2 ** int(b))) for s, b in
              zip(rng.choice([-1, 1], 5000), rng.integers(1, 56, 5000))]
    for R in cases:
        d = digits(R)
        assert sum(d[p] << (48 - 8 * p) for p in range(7)) == R
        assert all(-128 <= x <= 128 for x in d)
        for x in d:  # bf16: eight significant bits
            b = struct.unpack("<I", struct.pack("<f", float(x)))[0]
            assert b & 0xFFFF == 0


def test_combination():
    # FP32 sums of integers are exact below 2^24; the offset form needs |D| <= 2^22
    assert max(BOUND) < 2**24 and max(BOUND[:4]) <= 2**22
    for d in range(4):
        for s in (BOUND[d], -BOUND[d]):
            r = np.float32(s) + np.float32(12582912.0)
            assert struct.unpack("<I", struct.pack("<f", float(r)))[0] == (OFF + s) & 0xFFFFFFFF
    rng = np.random.default_rng(11)
    cases = [[0] * 7, BOUND, [-b for b in BOUND]]
    cases += [[int(rng.integers(-b, b + 1)) for b in BOUND] for _ in range(20000)]
    cases += [[int(rng.choice([-b, -1, 0, 1, b])) for b in BOUND] for _ in range(2000)]
    for D in cases:
        v = sum(D[d] << (8 * (6 - d)) for d in range(4, 7))
        w = (sum(D[d] << (8 * (3 - d)) for d in range(4)) << 17) + ((v + 64) >> 7)
        assert abs(w) < 2**62 and combine(D) == w, D
