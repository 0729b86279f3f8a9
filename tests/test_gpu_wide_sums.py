"""Pauli sums of many terms on either side of what an H pass can hold: the
12-qubit complex128 adjoint of a batch, which tile passes take where their H passes fit,
against the oracle and the engine a fixed shape selects, and tile-tier energies
of hundreds of terms over 26 qubits.  Tolerances as in test_gpu_parity."""
import numpy as np
import pytest

import oracle
import workloads as wl

pytestmark = pytest.mark.gpu

TOL = {"c128": 1e-12, "c64": 1e-5}


@pytest.fixture(scope="module")
def sv():
    import torch  # noqa: F401
    import paper_2406_03466_gb300 as m
    return m


def close(got, want, tol):
    got, want = np.asarray(got), np.asarray(want)
    assert float(np.max(np.abs(got - want))) <= tol * max(1.0, float(np.max(np.abs(want))))


def molecular(n, masks, terms, seed):
    """Z strings on `masks` flip masks (few diagonal tables, many terms)."""
    rng = np.random.default_rng(seed)
    xs = np.concatenate([[0], rng.choice((1 << n) - 1, masks - 1, replace=False) + 1])
    x = xs[rng.integers(0, masks, terms)]
    z = rng.integers(0, 1 << n, terms)
    q = np.arange(n)
    xb, zb = (x[:, None] >> q) & 1, (z[:, None] >> q) & 1
    return np.where(xb & zb, 2, np.where(xb, 1, np.where(zb, 3, 0))).astype(np.int8), rng.normal(size=terms) / terms


@pytest.mark.parametrize("terms", [100, 1000, 2500])
def test_batch_of_complex128_states(sv, terms):
    import torch
    w = wl.qcl(12, 3, 24)
    w.pauli_letters, w.pauli_coeffs = molecular(12, 40, terms, terms)
    theta = torch.as_tensor(w.theta, dtype=torch.float64, device="cuda")
    _, e_, g_ = sv.sv_grad_adjoint(sv.Problem.from_spec(w, "c128"), theta)
    close(e_.cpu(), oracle.instance_energies(w), 1e-12)
    fixed = sv.Problem.from_spec(w, "c128", opts=sv.plan_opts(reg_bits=3))
    close(g_.cpu(), sv.sv_grad_adjoint(fixed, theta)[2].cpu(), 1e-12)


@pytest.mark.parametrize("terms", [620, 660])
def test_tile_energies_of_wide_sums(sv, terms):
    """<H> is the sum of the halves' <H>, which fit an H pass with room to spare."""
    import torch
    w = wl.qcl(26, 1, 1)
    letters, coeffs = wl.random_pauli_sum(26, terms, 1)
    theta = torch.as_tensor(w.theta, dtype=torch.float64, device="cuda")
    got = []
    for part in (slice(None), slice(0, terms // 2), slice(terms // 2, None)):
        w.pauli_letters, w.pauli_coeffs = letters[part], coeffs[part]
        prob = sv.Problem.from_spec(w, "c64")
        got.append(float(sv.sv_energies(prob, theta)[1]))
        got.append(float(sv.sv_grad_adjoint(prob, theta)[1]))
    scale = max(1.0, float(np.linalg.norm(coeffs)))
    for k in (0, 1):
        assert abs(got[k] - got[2 + k] - got[4 + k]) <= TOL["c64"] * scale
