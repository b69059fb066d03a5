"""The binary64 Box–Muller tables that build.py writes for the reference stepper.

The logarithm from the table, -2 ln((w + 1/2) 2^-32), against longer
arithmetic at the ends of the words' range, around powers of two (where the
leading bit moves) and on random words: the two constants and the sum err by
half a unit in the last place each (2^-53 relative), the series by less than
one, so 2.5 x 2^-52 relative in all.  The angles: cosines and sines of the
binary64 product 2 pi u1 to half a unit in the last place, i.e. at most one unit
from the C library's.
"""
import re
import struct

import numpy as np
import pytest

from paper_2206_11234_gb300 import build


@pytest.fixture(scope="module")
def tables():
    out = {}
    for line in build.f64_tables().splitlines():
        name = re.search(r"k\w+64", line).group(0)
        out[name] = np.array([struct.unpack("<d", struct.pack("<Q", int(x, 16)))[0]
                              for x in re.findall(r"0x(\w+)ull", line)])
    return out


def words():
    rng = np.random.default_rng(3)
    w = [np.arange(0, 4096), 2**32 - 1 - np.arange(0, 4096), rng.integers(0, 2**32, 200000)]
    for p in range(1, 32):
        w.append(np.clip(2**p + np.arange(-3, 4), 0, 2**32 - 1))
        w.append(rng.integers(2 ** (p - 1), 2**p, 500))
    return np.unique(np.concatenate(w).astype(np.uint64))


def test_logarithm(tables):
    log, ln2n = tables["kLog64"].reshape(-1, 2), tables["kLn2N64"]
    w = words()
    U = 2 * w + 1
    top = np.floor(np.log2(U.astype(np.float64))).astype(np.int64)
    top -= (U < (np.uint64(1) << top.astype(np.uint64))).astype(np.int64)
    m = U.astype(np.float64) * np.exp2(-top.astype(np.float64))  # exact: U has 33 bits
    assert np.all((m >= 1.0) & (m < 2.0))
    i = ((m - 1.0) * 1024).astype(np.int64)
    x = 2.0 + m * log[i, 0]  # exact: 33 x 20 bits
    assert np.abs(x).max() <= 2.0**-10 * 1.002
    L = (log[i, 1] + ln2n[32 - top]) + (x + x * x * (0.25 + x * (1 / 12 + x * (1 / 32 + x / 80))))
    ref = -2.0 * np.log((w.astype(np.longdouble) + np.longdouble(0.5)) / np.longdouble(2**32))
    assert np.max(np.abs((L - ref) / ref)) <= 2.5 * 2.0**-52


def test_angles(tables):
    t = tables["kTrig64"].reshape(-1, 2)
    a = 6.283185307179586 * ((np.arange(65536) + 0.5) / 65536)
    for k, f in ((0, np.cos), (1, np.sin)):
        assert np.all(np.abs(t[:, k] - f(a)) <= np.spacing(np.abs(t[:, k])))
