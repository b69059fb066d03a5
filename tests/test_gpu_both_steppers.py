"""Caps, folds and set orders in each stepper that a call may take.

A call of few runs takes the stepper with separate noise warps; a caller's
block_dim keeps the persistent one, in 64-step blocks beside long runs and in blocks
of one fold without.  The same sets go through all of them: the same records and step
counts, bit for bit, and binary64 run by run against the oracle.
"""
import math

import numpy as np
import pytest

import oracle
from paper_2206_11234_gb300 import workloads as W

pytestmark = pytest.mark.gpu

DN = 2e-3
CAPS = (1, 2, 15, 16, 17, 31, 32, 33, 47, 48, 63, 64, 65, 79, 80, 95, 96, 97, 127, 128, 129)
KINDS = {"f64": dict(precision="f64"), "f32_kahan": dict(precision="f32_kahan"), "f32_f64acc": dict(precision="f32_f64acc"),
         "power": dict(precision="f32_kahan", bias_p=3.0), "power_real": dict(precision="f32_f64acc", bias_p=2.5),
         "quartic": dict(precision="f32_f64acc", model=2, poly=[0, 0, 0, 0, 0.01]),
         "general": dict(precision="f32_kahan", model=2, poly=[0, 0, 0.1, 0, 0, 0, 1e-4])}


@pytest.fixture(scope="module")
def nat(cuda_device):
    from paper_2206_11234_gb300 import native
    return native


def run(nat, specs, **kw):
    import torch
    n = sum(s.n_traj for s in specs)
    N = torch.full((n,), -1.0, dtype=torch.float64, device="cuda")
    lw = torch.full_like(N, -1.0)
    steps = torch.zeros(1, dtype=torch.int64, device="cuda")
    p = nat.make_params(m=1.0, n_max=6.0, steps_out=steps, **kw)
    nat.fpt_simulate_batch(p, nat.make_sets(specs), 9, N, lw)
    return N.cpu().numpy(), lw.cpu().numpy(), int(steps.item())


def same(a, b):
    """Bit for bit; a run that escapes past the largest float has ln w = NaN in both."""
    return np.array_equal(a, b, equal_nan=True)


def capped(cap, phi_in, n, i, phi_uv, b):
    return W.SetSpec(phi_in=phi_in, phi_uv=phi_uv, m=1.0, b=b, dN=DN, n_max=(cap - 0.5) * DN, n_traj=n, set_id=i)


@pytest.mark.parametrize("kind,k_steps", [(k, ks) for k in KINDS for ks in
                                          ((4, 8) if k == "f64" else (32,) if k.startswith("power") else (16, 32, 64))])
@pytest.mark.parametrize("wall", [False, True])
def test_caps_at_the_edges_of_groups_folds_and_blocks(nat, kind, k_steps, wall):
    kw = dict(KINDS[kind], k_steps=k_steps)
    b = 0.02 if kind.startswith("power") else 0.5
    # runs that mostly reach their cap, runs that mostly end before, then long ones
    sets = [capped(c, 2.2, 37, 2 * i, 2.25 if wall else math.inf, b) for i, c in enumerate(CAPS)]
    sets += [capped(c, 1.47, 41, 2 * i + 1, 1.5 if wall else math.inf, b) for i, c in enumerate(CAPS)]
    sets += [W.SetSpec(phi_in=3.0, phi_uv=3.1 if wall else math.inf, m=1.0, b=b, dN=DN, n_max=6.0, n_traj=501, set_id=60)]
    N, lw, steps = run(nat, sets, **kw)
    for block in (32, 128):
        N1, lw1, steps1 = run(nat, sets, block_dim=block, **kw)
        assert same(N, N1) and same(lw, lw1) and steps == steps1, block
    N1, lw1, _ = run(nat, sets[:-1], **kw)  # without the long ones
    assert same(N[:-501], N1) and same(lw[:-501], lw1)
    if kind != "f64":
        return
    at = 0
    for s in sets:
        r = oracle.make_run(m=1.0, phi_in=s.phi_in, phi_uv=s.phi_uv, dN=DN, b=b, n_max=s.n_max, seed=9, set_id=s.set_id)
        No, lwo, so = oracle.simulate(r, s.n_traj)
        Ng, lg = N[at:at + s.n_traj], lw[at:at + s.n_traj]
        fin = np.isfinite(No)
        assert np.array_equal(np.isfinite(Ng), fin)
        assert np.all(np.abs(Ng[fin] - No[fin]) <= 1e-12 * np.maximum(No[fin], DN))
        assert np.all(np.abs(lg - lwo) <= 1e-12 * np.maximum(1.0, so * b * math.sqrt(DN)))
        at += s.n_traj


@pytest.mark.parametrize("kind", ["f64", "f32_kahan", "f32_f64acc"])
@pytest.mark.parametrize("block", [0, 32, 128, 512])
def test_sets_of_rising_length_in_any_block(nat, kind, block):
    """Tickets out of the sets' order (the longest first), an empty set, one that starts
    at its end and one that escapes: one call per set gives the same records."""
    spec = dict(dN=DN, n_max=6.0)
    sets = [W.SetSpec(phi_in=1.6, m=0.1, b=0.0, n_traj=333, set_id=0, **spec),
            W.SetSpec(phi_in=3.0, m=1.0, b=0.0, n_traj=0, set_id=1, **spec),
            W.SetSpec(phi_in=2.5, m=1.0, b=1.0, n_traj=1025, set_id=2, phi_uv=2.6, **spec),
            W.SetSpec(phi_in=1.2, m=1.0, b=0.0, n_traj=65, set_id=3, **spec),
            W.SetSpec(phi_in=4.0, m=1.0, b=30.0, n_traj=129, set_id=4, **spec),
            W.SetSpec(phi_in=4.0, m=0.01, b=0.0, n_traj=31, set_id=5, **spec)]
    N, lw, steps = run(nat, sets, block_dim=block, **KINDS[kind])
    at = total = 0
    for s in sets:
        if s.n_traj:
            N1, lw1, steps1 = run(nat, [s], block_dim=block, **KINDS[kind])
            assert same(N[at:at + s.n_traj], N1) and same(lw[at:at + s.n_traj], lw1), s.set_id
            total += steps1
        at += s.n_traj
    assert steps == total and np.all(N[-31 - 129 - 65:-31 - 129] == 0.0) and np.all(np.isinf(N[-31 - 129:-31]))


def test_64_binary64_sets(nat):
    """As many sets as a call may have, few runs each, in both steppers."""
    sets = [W.SetSpec(phi_in=1.8 + 0.02 * i, m=1.0, b=0.3, dN=DN, n_max=6.0, n_traj=1 + i % 5, set_id=i) for i in range(64)]
    a, b = run(nat, sets, precision="f64"), run(nat, sets, precision="f64", block_dim=128)
    assert same(a[0], b[0]) and same(a[1], b[1]) and a[2] == b[2]
