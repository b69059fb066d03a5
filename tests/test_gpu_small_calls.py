"""Calls on little data: the launches chosen for them, at the edges of their ranges, and their
times against calls of the same box (best of many; the faults they were written for were
1.2 to 1.6 times as slow)."""
import numpy as np
import pytest

import oracle
from oracle import estimate as OE
from paper_2206_11234_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nat(cuda_device):
    from paper_2206_11234_gb300 import native
    return native


def best_us(f, passes=30):
    import torch
    f()
    out = []
    for _ in range(passes):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(5):
            f()
        b.record()
        torch.cuda.synchronize()
        out.append(200.0 * a.elapsed_time(b))
    return min(out)


def test_many_sets_cost_little_on_the_host(nat):
    """64 sets of 100 runs of one step against one set of 6400: 44 and 31 us when
    ordering the sets took sixteen nodes of each."""
    import torch

    def call(n_sets):
        sets = nat.make_sets([W.SetSpec(phi_in=1.5, m=0.01, b=0.0, dN=0.5, n_max=1.0, n_traj=6400 // n_sets, set_id=i)
                              for i in range(n_sets)])
        N = torch.empty(6400, dtype=torch.float64, device="cuda")
        lw = torch.empty_like(N)
        p = nat.make_params(precision="f32_kahan", m=0.01, n_max=1.0)
        return lambda: nat.fpt_simulate_batch(p, sets, 3, N, lw)

    assert best_us(call(64)) < 1.3 * best_us(call(1))


@pytest.mark.parametrize("n_bins,n_sub", [(1, 1), (3, 1), (5, 1), (1021, 1), (1025, 1), (4096, 1), (64, 64), (7, 3)])
@pytest.mark.parametrize("size", [1, 2, 255, 256, 257, 8192, "wave", "wave+1"])
def test_histograms_of_few_records(nat, n_bins, n_sub, size):
    """Counts and maxima exactly, sums to rounding (as the larger ones), with one
    record per thread up to a CTA per SM and eight from there on."""
    import torch
    wave = 256 * torch.cuda.get_device_properties(0).multi_processor_count
    n = {"wave": wave, "wave+1": wave + 1}.get(size, size)
    N, lw = W.random_records(n, seed=n_bins, lo=0.0, hi=6.0)
    bins, counts = nat.empty_bins(n_bins * n_sub), nat.empty_counts(1)
    nat.fpt_histogram(torch.from_numpy(N).cuda(), torch.from_numpy(lw).cuda(), n_bins, 0.0, 6.0, bins, counts, n_sub=n_sub,
                      id_offset=5)
    ref, ref_counts = oracle.histogram(N, lw, n_bins, 0.0, 6.0, n_sub=n_sub, id_offset=5)
    ref, got = ref.reshape(-1, 8), bins.cpu().numpy()
    assert np.array_equal(counts.cpu().numpy()[0], ref_counts)
    assert np.array_equal(got.view(np.int64)[:, 7], ref[:, 7].astype(np.int64))
    assert np.array_equal(got[:, 0], ref[:, 0])
    np.testing.assert_allclose(got[:, 1:7], ref[:, 1:7], rtol=1e-12, atol=1e-300)


def test_many_bins_cost_few_records_little(nat):
    """100 records into 4096 bins and into one: calls of 57 and 46 us with eight records
    per thread and a bin per thread of the scan."""
    import torch
    N, lw = (torch.from_numpy(x).cuda() for x in W.random_records(100, seed=1, lo=0.0, hi=6.0))

    def call(nb):
        bins, counts = nat.empty_bins(nb), nat.empty_counts(1)
        return lambda: nat.fpt_histogram(N, lw, nb, 0.0, 6.0, bins, counts)

    assert best_us(call(4096)) < 1.13 * best_us(call(1))


def test_gradient_of_medium_batches(nat):
    """100,000 rows against 20,000: 98 and 60 us with three CTAs per SM, each of which
    adds its 4489 sums to the one gradient."""
    import torch
    w = nat.mlp_pack(W.mlp_params(seed=11, gain=1.5, out_scale=0.5), (5.2, 0.5, 30.0, 1 / 15.0))

    def call(n):
        x = [torch.rand(n, device="cuda") + 1.5 for _ in range(3)]
        grad = torch.zeros(nat.MLP_NPARAM, device="cuda")
        return lambda: nat.fpt_mlp_backward(w, *x, grad)

    assert best_us(call(100000)) < 1.3 * best_us(call(20000))


@pytest.mark.parametrize("n_bins,n_sub", [(2048, 2), (15, 2), (16, 2), (17, 2), (33, 1), (5, 3), (9, 8), (3, 9), (2, 33)])
def test_estimates_at_the_edges_of_the_lane_groups(nat, n_bins, n_sub):
    """A group of 1, 2, 8 or 32 lanes per bin: every field as the oracle has it from
    the raw records (tolerances as in test_gpu_estimate.py)."""
    import torch
    rng = np.random.default_rng(n_bins)
    N = rng.normal(8.5, 0.6, 60000)
    lw = -30.0 - 4.0 * (N - 7.0) + 0.8 * rng.standard_normal(N.size) + 0.3 * rng.exponential(1.0, N.size)
    bins, counts, est = nat.empty_bins(n_bins * n_sub), nat.empty_counts(1), nat.empty_estimates(n_bins)
    nat.fpt_histogram(torch.from_numpy(N).cuda(), torch.from_numpy(lw).cuda(), n_bins, 7.0, 10.0, bins, counts,
                      n_sub=n_sub, id_offset=3)
    nat.fpt_estimate(bins, n_bins, 7.0, 10.0, N.size, est, n_sub=n_sub, id_offset=3)
    got, ref = nat.estimates_to_dict(est), OE.estimate(N, lw, n_bins, 7.0, 10.0, n_sub=n_sub, id_offset=3)
    for f, x in ref.items():
        if f in ("bias_ln", "p_normal"):  # their errors are those of k4 and of K^2, compared as k2 and bias_se
            continue
        tol = 1e-7 if f in ("skew", "kurt", "z_skew", "z_kurt", "k2", "bias_se") else 1e-9
        np.testing.assert_allclose(got[f], x, rtol=tol, atol=tol if tol > 1e-9 else 1e-300, equal_nan=True, err_msg=f)


def test_two_subsets_cost_no_more_than_one(nat):
    """2048 bins of two subsets against 4096 bins: 60 and 17 us with eight lanes per bin."""
    bins = nat.empty_bins(4096)
    bins.zero_()

    def call(nb, ns):
        est = nat.empty_estimates(nb)
        return lambda: nat.fpt_estimate(bins, nb, 0.0, 1.0, 1000, est, n_sub=ns)

    assert best_us(call(2048, 2)) < 1.8 * best_us(call(4096, 1))
