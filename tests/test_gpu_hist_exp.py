"""The histogram's exponential and its fixed-point bins at their edges."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def histogram(N, lw, lo, hi, n_bins):
    """(counts, s1, s2) per bin."""
    import torch
    from paper_2206_11234_gb300 import native as nat
    bins = torch.zeros(n_bins, 8, dtype=torch.float64, device="cuda")
    counts = torch.zeros(4, dtype=torch.int64, device="cuda")
    nat.fpt_histogram(torch.as_tensor(N).cuda(), torch.as_tensor(lw).cuda(), n_bins, lo, hi, bins, counts)
    h = bins.cpu().numpy()
    return h[:, 7].copy().view(np.int64), h[:, 1], h[:, 2]


def test_exponential_by_record():
    """Bins of two records, ln w = 0 and y: s1 = 1 + exp(y) and s2 = 1 + exp(2 y), each rounded
    from an exp(y) within a unit in the last place; around the steps of ln 2 / 4096 and the
    powers of 2, for tiny |y|, up to and beyond 512, and for a zero weight."""
    rng = np.random.default_rng(5)
    step = math.log(2.0) / 4096
    k = np.concatenate([np.arange(1, 40), 4096 * np.arange(1, 40), rng.integers(1, 3_000_000, 400)])
    y = np.concatenate([-k * step, -np.nextafter(k * step, 0), -np.nextafter(k * step, 1e9), -(k + 0.5) * step,
                        -rng.random(500), -30 * rng.random(500), -10.0 ** -np.arange(0, 320, 8),
                        [-0.0, -511.9999999999999, -512.0, -700.0, -745.0, -800.0, -math.inf]])
    for i in range(0, len(y), 2000):
        part = y[i:i + 2000]
        n = len(part)
        _, s1, s2 = histogram(np.repeat(np.arange(n) + 0.5, 2), np.stack([np.zeros(n), part], 1).ravel().copy(),
                              0.0, float(n), n)
        e = np.array([math.exp(v) for v in part])
        assert np.all(np.abs(s1 - (1.0 + e)) <= 2 * 2.0 ** -52)
        assert np.all(np.abs(s2 - (1.0 + e * e)) <= 4 * 2.0 ** -52)


@pytest.mark.parametrize("lo,hi,n_bins", [(7.0, 10.0, 4095), (-24.0, -21.0, 4095), (0.1, 0.4, 97), (31.9, 32.0, 100),
                                          (-32768.0, -32767.0, 1), (32766.0, 32768.0, 2), (3e5, 3e5 + 1, 4)])
def test_bins_as_the_division_gives_them(lo, hi, n_bins):
    """Bins of values at, next to and between the edges are ceil((N - lo) / d) - 1, also
    where |lo| / d is up to and beyond the fixed point's range."""
    d = (hi - lo) / n_bins
    edges = lo + d * np.arange(n_bins + 1)
    N = np.concatenate([edges, np.nextafter(edges, -np.inf), np.nextafter(edges, np.inf),
                        lo + (hi - lo) * np.random.default_rng(3).random(20000)])
    count, _, _ = histogram(N, np.zeros(len(N)), lo, hi, n_bins)
    inside = N[(N > lo) & (N <= hi)]
    want = np.bincount(np.clip(np.ceil((inside - lo) / d).astype(int) - 1, 0, n_bins - 1), minlength=n_bins)
    assert np.array_equal(count, want)
