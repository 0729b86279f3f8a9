"""Tile passes whose shared memory lies just below the limit without the split
stages' phase tables (complex128, tiles of 2^11, 11 stages of 33 groups): they
run, with and without those tables, as one call and as a batch of circuits,
against the oracle.  Tolerances as in test_gpu_parity."""
import numpy as np
import pytest

import oracle
import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sv():
    import torch  # noqa: F401
    import paper_2406_03466_gb300 as m
    return m


def close(got, want, tol=1e-12):
    got, want = np.asarray(got), np.asarray(want)
    assert float(np.max(np.abs(got - want))) <= tol * max(1.0, float(np.max(np.abs(want))))


@pytest.mark.parametrize("ops", [("RX", "RZ", "RX"), ("RX",)])  # four sums a group, one
@pytest.mark.parametrize("no_relabel", [False, True])
def test_largest_complex128_pass(sv, ops, no_relabel):
    import torch
    n = 11
    rng = np.random.default_rng(len(ops))
    gates = wl.layered_ansatz(n, 3, ops, "ladder")
    p = 3 * n * len(ops)
    letters = rng.choice([0, 1, 2, 3], size=(5, n)).astype(np.int8)
    w = wl.Workload("limit", n, gates, p, rng.uniform(-3, 3, p), letters, rng.normal(size=5),
                    np.array([0, 5]), weights=np.array([0.4, 0.9]))
    prob = sv.Problem.from_spec(w, "c128", opts=sv.plan_opts(tile_bits=11, reg_bits=3, no_relabel=no_relabel))
    theta = torch.as_tensor(w.theta, dtype=torch.float64, device="cuda")
    _, e_, g_ = sv.sv_grad_adjoint(prob, theta)
    ks = [0, p // 2, p - 1]
    _, E, g = oracle.grad_param_shift(w, params=ks)
    close(e_.cpu(), E)
    close(g_.cpu()[ks], g)
    close(sv.sv_energies(prob, theta)[1].cpu(), E)
