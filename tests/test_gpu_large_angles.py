"""Angles of many turns: theta + 4 pi k (rounded to double) against the oracle at
the same angle, by every engine that forms gate matrices in single precision
(on chip) or by table (tile passes), and in complex128.  A matrix must stay
unitary whatever its angle's size; tolerances as in test_gpu_parity, for gradients
plus the rounding of theta +- pi / 2, which the oracle's shift rule sees and the
adjoint does not."""
import numpy as np
import pytest

import oracle
import workloads as wl

pytestmark = pytest.mark.gpu

TOL = {"c128": dict(E=1e-12, G=1e-12), "c64": dict(E=1e-5, G=1e-4)}


@pytest.fixture(scope="module")
def sv():
    import torch  # noqa: F401
    import paper_2406_03466_gb300 as m
    return m


def close(got, want, tol):
    got, want = np.asarray(got), np.asarray(want)
    scale = max(1.0, float(np.max(np.abs(want))))
    assert float(np.max(np.abs(got - want))) <= tol * scale


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("n", [4, 8, 14])
@pytest.mark.parametrize("turns", [100, 2000003])
def test_large_angles(sv, dtype, n, turns):
    import torch
    w = wl.qcl(n, 1, 2) if n > 4 else wl.qcl(n, 2, 2)
    k = np.where(np.arange(w.n_params) % 2, turns, -turns)
    w = wl.Workload(**{**w.__dict__, "theta": w.theta + 4 * np.pi * k})
    theta = torch.as_tensor(w.theta, dtype=torch.float64, device="cuda")
    prob = sv.Problem.from_spec(w, dtype)
    ks = sorted({0, w.n_params // 2, w.n_params - 1})
    L, E, g = oracle.grad_param_shift(w, params=ks)
    close(sv.sv_energies(prob, theta)[1].cpu(), E, TOL[dtype]["E"])
    for fn in (sv.sv_grad_adjoint, sv.sv_grad_param_shift):
        _, e_, g_ = fn(prob, theta)
        close(e_.cpu(), E, TOL[dtype]["E"])
        close(g_.cpu()[ks], g, TOL[dtype]["G"] + 2 * np.spacing(np.max(np.abs(w.theta))))


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("n", [5, 8])
def test_angles_and_inputs_at_the_edges(sv, dtype, n):
    """Angles on both sides of 8 (where whole turns start to come off), inputs at
    and next to +-1 and 0; an input that only rounds to 1 in float counts as 1
    in complex64."""
    import torch
    w = wl.qcl(n, 2, 8)
    theta = np.resize(np.array([8.0, -8.0, 7.99999, 8.00001, -8.00001, 4 * np.pi, -2 * np.pi, 0.0, 1e-9]), w.n_params)
    x = np.array([1.0, -1.0, 0.0, 0.9999999, -0.9999, 0.5, 1e-8, 1.0]).reshape(-1, 1)
    w = wl.Workload(**{**w.__dict__, "theta": theta, "inputs": x})
    E = oracle.instance_energies(w)
    given = x.copy()
    if dtype == "c64":
        given[-1] = 1.0 + 1e-9
    prob = sv.Problem.from_spec(wl.Workload(**{**w.__dict__, "inputs": given}), dtype)
    th = torch.as_tensor(theta, dtype=torch.float64, device="cuda")
    close(sv.sv_energies(prob, th)[1].cpu(), E, TOL[dtype]["E"])
    ks = sorted({0, w.n_params // 2, w.n_params - 1})
    g = oracle.grad_param_shift(w, params=ks)[2]
    for fn in (sv.sv_grad_adjoint, sv.sv_grad_param_shift):
        close(fn(prob, th)[2].cpu()[ks], g, TOL[dtype]["G"])
