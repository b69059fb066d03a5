"""Records do not depend on how a launch is laid out: the order in which the
sets' tickets are handed out, the threads per block and the resident warps the
library picks for a given number of runs, or the scheduling block the
binary32 stepper works in.

Sets of very different lengths (so that their tickets are reordered), with an
empty set and one that starts at its end, must leave the records of one call
per set, bit for bit; every block size gives the same records at run counts
around warp, block and wave edges; and first-passage times do not depend on
k_steps, which only sets where ln w is rounded.
"""
import math

import numpy as np
import pytest

from paper_2206_11234_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nat(cuda_device):
    from paper_2206_11234_gb300 import native
    return native


def batch(nat, specs, precision, **kw):
    import torch
    n = sum(s.n_traj for s in specs)
    N = torch.full((n,), -1.0, dtype=torch.float64, device="cuda")
    lw = torch.full_like(N, -1.0)
    nat.fpt_simulate_batch(nat.make_params(precision=precision, m=specs[0].m, n_max=specs[0].n_max, **kw),
                           nat.make_sets(specs), 3, N, lw)
    return N, lw


@pytest.mark.parametrize("precision", ["f64", "f32_kahan", "f32_f64acc"])
def test_sets_of_rising_length_equal_one_call_per_set(nat, precision):
    import torch
    spec = dict(dN=2e-3, n_max=8.0)
    specs = [W.SetSpec(phi_in=1.6, m=0.1, b=0.0, n_traj=333, set_id=0, **spec),
             W.SetSpec(phi_in=3.0, m=1.0, b=0.0, n_traj=0, set_id=1, **spec),
             W.SetSpec(phi_in=2.5, m=1.0, b=1.0, n_traj=1025, set_id=2, phi_uv=2.6, **spec),
             W.SetSpec(phi_in=1.2, m=1.0, b=0.0, n_traj=65, set_id=3, **spec),  # starts past the end: N = 0
             W.SetSpec(phi_in=4.0, m=1.0, b=30.0, n_traj=129, set_id=4, **spec),  # escapes: censored
             W.SetSpec(phi_in=4.0, m=0.01, b=0.0, n_traj=31, set_id=5, **spec)]
    N, lw = batch(nat, specs, precision)
    off = 0
    for s in specs:
        if s.n_traj:
            N1, l1 = batch(nat, [s], precision)
            # the wall of another set makes the kernel mirror at infinity too, which changes nothing
            assert torch.equal(N[off:off + s.n_traj], N1), s.set_id
            assert torch.equal(lw[off:off + s.n_traj], l1), s.set_id
        off += s.n_traj
    assert torch.all(N[-31 - 129 - 65:-31 - 129] == 0.0)
    assert torch.all(torch.isinf(N[-31 - 129:-31]))


@pytest.mark.parametrize("precision", ["f64", "f32_kahan"])
@pytest.mark.parametrize("n", [1, 31, 33, 4865, 20001])
def test_any_block_size_gives_the_same_records(nat, precision, n):
    import torch
    s = W.SetSpec(phi_in=1.8, m=1.0, b=0.5, dN=2e-3, n_max=3.0, n_traj=n)
    N, lw = batch(nat, [s], precision)
    for block in (32, 96, 512):
        N1, l1 = batch(nat, [s], precision, block_dim=block)
        assert torch.equal(N, N1) and torch.equal(lw, l1), block


@pytest.mark.parametrize("precision", ["f32_kahan", "f32_f64acc"])
@pytest.mark.parametrize("n_max", [0.002, 0.03, 0.034, 0.128, 0.13, 3.0])
def test_block_lengths_agree(nat, precision, n_max):
    """Caps below, at and past 16- and 64-step edges; ln w agrees to the
    rounding of its binary32 block sums (at most 64 terms of a few units each:
    64 x 4 x 2^-24 x b sqrt(dN) per block, and at most n_max / dN / 16 blocks)."""
    dN, b = 2e-3, 0.5
    s = W.SetSpec(phi_in=1.45, m=1.0, b=b, dN=dN, n_max=n_max, n_traj=5000)
    N, lw = batch(nat, [s], precision)
    steps = math.ceil(n_max / dN)
    tol = 64 * 4 * 2.0 ** -24 * b * math.sqrt(dN) * math.ceil(steps / 16)
    for ks in (16, 32, 64):
        N1, l1 = batch(nat, [s], precision, k_steps=ks)
        assert np.array_equal(N.cpu().numpy(), N1.cpu().numpy()), ks
        assert float((lw - l1).abs().max()) <= tol, ks


@pytest.mark.parametrize("precision", ["f32_kahan", "f32_f64acc"])
@pytest.mark.parametrize("c", [[0, 0, 0, 0, 0.0125], [0.02, 0, 0.1, 0.01], [0, 0, 0.15, 0, 0.005]])
@pytest.mark.parametrize("phi_uv", [math.inf, 4.6])
def test_low_degree_polynomial_is_the_general_one(nat, precision, c, phi_uv):
    """A potential of degree <= 4 starts Horner's rule at its own degree; with a
    coefficient of phi^7 that is zero in binary32 only, the general kernel runs
    the same potential: the same records, bit for bit."""
    import torch
    out = []
    for poly in (c, c + [0.0] * (7 - len(c)) + [1e-300]):
        N = torch.empty(4097, dtype=torch.float64, device="cuda")
        lw = torch.empty_like(N)
        p = nat.make_params(model=nat.MODEL_POLYNOMIAL, precision=precision, poly=poly, n_max=6.0)
        nat.fpt_simulate(p, N.numel(), 4.0, 2.5, phi_uv, 1e-3, 0.6, 9, N, lw)
        out.append((N, lw))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])


def test_binary64_normals_over_all_angles_and_table_entries(nat):
    """2^19 binary64 normals (every 16-bit angle about four times, every entry of
    the logarithm's table) against the oracle's library functions: a few units in
    the last place, as for the smaller sample of test_gpu_parity."""
    import torch
    import oracle
    nb = 1 << 17
    z = torch.empty(4 * nb, dtype=torch.float64, device="cuda")
    nat.fpt_normals(11, 5, 1, 0, nb, "f64", z)
    ref = np.concatenate([oracle.normals4(11, 5, 1, k) for k in range(nb)])
    assert np.max(np.abs(z.cpu().numpy() - ref) / np.maximum(np.abs(ref), 1e-3)) < 4e-15


@pytest.mark.parametrize("ks", [4, 8])
@pytest.mark.parametrize("n_max", [0.006, 0.03, 0.032, 0.034, 1.0])
def test_binary64_caps_inside_a_block(nat, ks, n_max):
    """Caps at and beside the 4-, 8- and 16-step edges of the binary64 stepper against the oracle, run by run."""
    import oracle
    dN, b = 2e-3, 0.5
    s = W.SetSpec(phi_in=1.45, m=1.0, b=b, dN=dN, n_max=n_max, n_traj=3000, phi_uv=1.5)
    N, lw = batch(nat, [s], "f64", k_steps=ks)
    r = oracle.make_run(m=1.0, phi_in=1.45, phi_uv=1.5, dN=dN, b=b, n_max=n_max, seed=3)
    No, lwo, so = oracle.simulate(r, 3000)
    N, lw = N.cpu().numpy(), lw.cpu().numpy()
    fin = np.isfinite(No)
    assert np.array_equal(np.isfinite(N), fin)
    assert np.all(np.abs(N[fin] - No[fin]) <= 1e-12 * np.maximum(No[fin], dN))
    assert np.all(np.abs(lw - lwo) <= 1e-12 * np.maximum(1.0, so * b * math.sqrt(dN)))


@pytest.mark.parametrize("kind", ["f32_kahan", "f32_f64acc", "power", "quartic"])
@pytest.mark.parametrize("n", [19457, 20011, 24000, 38913, 40001, 60000])
def test_runs_that_take_turns(nat, kind, n):
    """Run counts just above a whole number of warps per scheduler, with runs of one
    length: the library lets a few runs per warp take turns.  The same records,
    bit for bit, as in calls small enough that none has to (runs 0 .. n by their
    offsets), with a second set of runs that start past their end."""
    import torch
    kw = {"power": dict(precision="f32_kahan", bias_p=3.0), "quartic": dict(precision="f32_kahan", model=2,
          poly=[0, 0, 0, 0, 1e-7])}.get(kind, dict(precision=kind))
    end = 1.8 if kind == "quartic" else W.PHI_END
    base = dict(m=0.01, dN=5e-4, n_max=0.4 if n == 24000 else 1.0, phi_end=end)  # 24000: censored at the cap
    specs = [W.SetSpec(phi_in=2.0, b=1e-3, n_traj=n, set_id=4, **base),
             W.SetSpec(phi_in=1.0, b=1e-3, n_traj=70, set_id=5, **base)]
    p = nat.make_params(m=0.01, n_max=1.0, **kw)

    def run(sp, seed=6):
        N = torch.full((sum(s.n_traj for s in sp),), -1.0, dtype=torch.float64, device="cuda")
        lw = torch.full_like(N, -1.0)
        nat.fpt_simulate_batch(p, nat.make_sets(sp), seed, N, lw)
        return N, lw

    N, lw = run(specs)
    assert torch.all(N[n:] == 0.0) and torch.all(lw[n:] == 0.0)
    step = 4096
    for off in range(0, n, step):
        k = min(step, n - off)
        N1, l1 = run([W.SetSpec(phi_in=2.0, b=1e-3, n_traj=k, set_id=4, traj_offset=off, **base)])
        assert torch.equal(N[off:off + k], N1) and torch.equal(lw[off:off + k], l1), off


@pytest.mark.parametrize("k_eval", [16, 32, 64, 128])
def test_learned_bias_few_and_many_runs(nat, k_eval):
    """A learned-bias call of few runs takes the kernel with held-back records, one
    of many runs (more than two tiles of 128 per SM) the other: the same runs and the
    same set of training records, bit for bit, split at an odd place."""
    import torch
    n, cut = 45001, 20011
    w = nat.mlp_pack(W.mlp_params(seed=21, gain=1.0, out_scale=0.6), (3.0, 1.0, 2.0, 0.5))
    base = dict(phi_in=2.4, m=1.0, b=0.0, dN=2e-3, n_max=1.0, phi_uv=2.6, set_id=2)
    p = nat.make_params(precision="f32_f64acc", m=1.0, n_max=1.0, mlp=w, k_eval=k_eval)

    def run(off, k):
        N = torch.empty(k, dtype=torch.float64, device="cuda")
        lw = torch.empty_like(N)
        rec = torch.empty((k * (500 // k_eval + 2), 4), dtype=torch.float32, device="cuda")
        m = nat.fpt_simulate_mlp(p, nat.make_sets([W.SetSpec(n_traj=k, traj_offset=off, **base)]), 8, N, lw, rec)
        r = rec[:m].cpu().numpy().view(np.uint32).copy()
        r[:, 3] += off  # runs are numbered within a call
        return N, lw, r

    N, lw, r = run(0, n)
    a, b = run(0, cut), run(cut, n - cut)
    assert torch.equal(N, torch.cat([a[0], b[0]])) and torch.equal(lw, torch.cat([a[1], b[1]]))
    both = np.concatenate([a[2], b[2]])
    order = lambda q: q[np.lexsort(q.T)]  # noqa: E731
    assert r.shape == both.shape and np.array_equal(order(r), order(both))


@pytest.mark.parametrize("kind", ["f32_kahan", "f32_f64acc", "power", "power_real", "quartic"])
@pytest.mark.parametrize("n", [1, 31, 33, 4097])
@pytest.mark.parametrize("k_steps", [16, 32, 64])
def test_few_runs(nat, kind, n, k_steps):
    """Few runs take the stepper with separate noise warps; a caller's block_dim
    keeps the persistent one.  The same records, bit for bit: sets with and without
    a wall, at the cap, ended at their start, and an empty one, with caps at and off
    the edges of 16 and k_steps."""
    import torch
    kw = {"power": dict(precision="f32_kahan", bias_p=3.0), "power_real": dict(precision="f32_f64acc", bias_p=2.5),
          "quartic": dict(precision="f32_kahan", model=2, poly=[0, 0, 0, 0, 0.01])}.get(kind, dict(precision=kind))
    ks = 32 if kind.startswith("power") else k_steps
    base = dict(m=1.0, dN=2e-3, phi_end=1.8)
    specs = [W.SetSpec(phi_in=2.0, b=0.02, n_traj=n, set_id=1, n_max=3.0, **base),
             W.SetSpec(phi_in=1.9, b=0.01, n_traj=n, set_id=2, n_max=0.13, phi_uv=1.95, **base),
             W.SetSpec(phi_in=1.7, b=0.01, n_traj=5, set_id=3, n_max=0.13, **base),
             W.SetSpec(phi_in=1.9, b=0.0, n_traj=0, set_id=4, n_max=0.13, **base),
             W.SetSpec(phi_in=4.0, b=0.0, n_traj=n, set_id=5, n_max=0.128, **base)]
    total = 3 * n + 5
    out = []
    for block in (0, 128):
        N = torch.full((total,), -1.0, dtype=torch.float64, device="cuda")
        lw = torch.full_like(N, -1.0)
        steps = torch.zeros(1, dtype=torch.int64, device="cuda")
        p = nat.make_params(m=1.0, n_max=3.0, block_dim=block, k_steps=ks, steps_out=steps, **kw)
        nat.fpt_simulate_batch(p, nat.make_sets(specs), 12, N, lw)
        out.append((N, lw, int(steps.item())))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert out[0][2] == out[1][2]
    assert torch.all(out[0][0][2 * n:2 * n + 5] == 0.0) and torch.all(torch.isinf(out[0][0][2 * n + 5:]))


@pytest.mark.parametrize("n", [1, 33, 4097])
@pytest.mark.parametrize("k_steps", [4, 8])
def test_few_runs_f64(nat, n, k_steps):
    """As above for the binary64 mode; walls, and caps at and off the edges of 4, 8 and 16."""
    import torch
    base = dict(m=1.0, dN=2e-3, phi_end=1.8)
    specs = [W.SetSpec(phi_in=2.0, b=0.02, n_traj=n, set_id=1, n_max=3.0, **base),
             W.SetSpec(phi_in=1.9, b=0.01, n_traj=n, set_id=2, n_max=0.13, phi_uv=1.95, **base),
             W.SetSpec(phi_in=1.7, b=0.01, n_traj=5, set_id=3, n_max=0.13, **base),
             W.SetSpec(phi_in=1.9, b=0.0, n_traj=0, set_id=4, n_max=0.13, **base),
             W.SetSpec(phi_in=4.0, b=0.0, n_traj=n, set_id=5, n_max=0.128, **base)]
    for some in (specs, specs[:1]):
        total = sum(s.n_traj for s in some)
        out = []
        for block in (0, 128):
            N = torch.full((total,), -1.0, dtype=torch.float64, device="cuda")
            lw = torch.full_like(N, -1.0)
            steps = torch.zeros(1, dtype=torch.int64, device="cuda")
            p = nat.make_params(m=1.0, n_max=3.0, precision="f64", block_dim=block, k_steps=k_steps, steps_out=steps)
            nat.fpt_simulate_batch(p, nat.make_sets(some), 12, N, lw)
            out.append((N, lw, int(steps.item())))
        assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
        assert out[0][2] == out[1][2]
