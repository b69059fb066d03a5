"""The histogram's exponential of a number <= 0, in integers (csrc/histogram.cu), restated
with the tables that build.py writes.

Every rounding of the integer steps is restated, and the result compared with
50-digit arithmetic: within 0.77 units in the last place, the bound that the kernel's
comment gives, over all table entries, at the steps of ln 2 / 4096 and halfway between them,
around the powers of two, for tiny arguments and up to 512, where the library's
exponential takes over (the largest exponent the integer form has to assemble is
that of exp(-512) = 2^-739).
"""
import decimal
import math
import re
import struct

import numpy as np
import pytest

from paper_2206_11234_gb300 import build

M64 = (1 << 64) - 1


@pytest.fixture(scope="module")
def tables():
    text = build.exp_table()
    words = [int(x) for x in re.findall(r"(\d+)ull", text)]
    const = {k: int(v) for k, v in re.findall(r"(kExp\w+) = (\d+)u", text)}
    assert len(words) == 4096
    return words, const


def exp_neg(x, tables):
    """csrc/histogram.cu's exp_neg for -512 < x <= 0."""
    table, c = tables
    bits = struct.unpack("<Q", struct.pack("<d", x))[0] & ((1 << 63) - 1)
    hi = bits >> 32
    assert hi < 0x40800000
    m = (((((hi & 0xFFFFF) | 0x100000) << 32) | (bits & 0xFFFFFFFF)) << 11) & M64
    z = m >> min(1031 - (hi >> 20), 63)
    k = ((z >> 32) * c["kExpPerStep"] + (1 << 41)) >> 42
    kstep = (k * c["kExpStep1"] + (k * c["kExpStep0"] >> 32) + (((k * c["kExpStep2"]) & 0xFFFFFFFF) << 32)) & M64
    r = ((z << 11) - kstep) & M64
    r -= (r >> 63) << 64
    assert abs(r) < 1 << 53
    rs = r >> 22
    assert -(1 << 31) <= rs < 1 << 31
    r2 = (rs * rs) >> 32
    w = (0x80000000 - (rs * 174763 >> 32)) & 0xFFFFFFFF
    p = r - ((r2 * w & M64) >> 22)
    T = table[k & 4095]
    Th, ph = T >> 32, p >> 32
    assert Th < 1 << 31 and -(1 << 31) <= ph < 1 << 31
    Tp = Th * ph + (Th * (p & 0xFFFFFFFF) >> 32) + 2 * ((((T & 0xFFFFFFFF) >> 1) * ph) >> 32)
    e = T - (Tp >> 2)
    over = e >> 62
    e = (e >> over) + 256
    out = ((1021 + over - (k >> 12)) << 52) + (e >> 9)
    assert 0 < out < 1 << 63
    return struct.unpack("<d", struct.pack("<Q", out))[0]


def arguments():
    rng = np.random.default_rng(7)
    step = math.log(2.0) / 4096
    k = np.concatenate([np.arange(0, 4097), 4096 * np.arange(1, 738), rng.integers(1, 3_025_000, 2000)]).astype(np.float64)
    a = [k * step, np.nextafter(k * step, 0), np.nextafter(k * step, 1e9), (k + 0.5) * step,
         2.0 ** -np.arange(0.0, 60.0), 2.0 ** np.arange(0.0, 9.0), np.nextafter(2.0 ** np.arange(-30.0, 10.0), 0),
         10.0 ** -np.arange(0.0, 320.0, 4.0), 512 * rng.random(3000), 40 * rng.random(2000), rng.random(2000),
         [511.9999999999999, np.nextafter(512.0, 0), 5e-324, 0.0]]
    a = np.unique(np.concatenate([np.asarray(x, dtype=np.float64) for x in a]))
    return a[a < 512.0]


def test_exponential_in_units_in_the_last_place(tables):
    ctx = decimal.Context(prec=50)
    worst = 0.0
    for a in arguments():
        got = exp_neg(-float(a), tables)
        exact = ctx.exp(decimal.Decimal(-float(a)))
        ulp = decimal.Decimal(math.ulp(float(exact)) if float(exact) < 1.0 else 2.0 ** -53)
        worst = max(worst, abs(float(ctx.divide(ctx.subtract(decimal.Decimal(got), exact), ulp))))
    assert worst <= 0.77, worst


def test_exponential_of_zero_is_one(tables):
    assert exp_neg(0.0, tables) == 1.0 and exp_neg(-0.0, tables) == 1.0
