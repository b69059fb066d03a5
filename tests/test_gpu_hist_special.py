"""Weights that are not numbers, infinite or zero in the sorted second pass of the histogram.

ln w = -inf is a run of weight zero; NaN and +inf are a caller's mistake that must
stay in its own bin: the other bins, which share tiles and threads with it, keep
their exact values.  Sizes with one, eight and 32 records per thread.
"""
import math

import numpy as np
import pytest

import oracle
from paper_2206_11234_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nat(cuda_device):
    from paper_2206_11234_gb300 import native
    return native


@pytest.mark.parametrize("n", [3000, 100_000, 6_000_000])
@pytest.mark.parametrize("n_bins", [24, 3000])
def test_special_weights_stay_in_their_bins(nat, n, n_bins):
    import torch
    N, lw = W.random_records(n, seed=n_bins, lo=0.0, hi=6.0)
    inside = np.isfinite(N) & (N > 0.0) & (N <= 6.0)
    j = np.where(inside, np.clip(np.ceil(N / (6.0 / n_bins)).astype(float) - 1, 0, n_bins - 1), -1).astype(int)
    some, _ = oracle.histogram(N, lw, n_bins, 0.0, 6.0)
    full = np.flatnonzero(some[0, :, 7].astype(int) >= 3)
    b_nan, b_inf, b_zero, b_only = full[[1, len(full) // 3, len(full) // 2, -2]]
    assert len({b_nan, b_inf, b_zero, b_only}) == 4
    for b, v in ((b_nan, math.nan), (b_inf, math.inf), (b_zero, -math.inf)):
        lw[np.flatnonzero(j == b)[1]] = v
    lw[j == b_only] = -math.inf
    bins, counts = nat.empty_bins(n_bins), nat.empty_counts(1)
    nat.fpt_histogram(torch.from_numpy(N).cuda(), torch.from_numpy(lw).cuda(), n_bins, 0.0, 6.0, bins, counts)
    got = bins.cpu().numpy()
    ref = some[0]
    assert np.array_equal(got.view(np.int64)[:, 7], ref[:, 7].astype(np.int64))
    rest = np.ones(n_bins, dtype=bool)
    rest[[b_nan, b_inf, b_zero, b_only]] = False
    assert np.array_equal(got[rest, 0], ref[rest, 0])
    np.testing.assert_allclose(got[rest, 1:7], ref[rest, 1:7], rtol=1e-12, atol=1e-300)
    assert math.isnan(got[b_nan, 0]) and np.all(np.isnan(got[b_nan, 1:7]))
    assert got[b_inf, 0] == math.inf and np.all(np.isnan(got[b_inf, 1:7]))
    assert got[b_only, 0] == -math.inf and np.all(np.isnan(got[b_only, 1:7]))
    x = lw[j == b_zero]
    x = x[np.isfinite(x)]
    assert got[b_zero, 0] == x.max()
    np.testing.assert_allclose(got[b_zero, 1:3], [np.exp(x - x.max()).sum(), np.exp(2 * (x - x.max())).sum()], rtol=1e-12)
    assert list(got[b_zero, 3:7]) == [-math.inf, math.inf, -math.inf, math.inf]
