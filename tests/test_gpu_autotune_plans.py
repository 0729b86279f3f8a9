"""sv_autotune of device-memory states times a shape on the plan that later calls
run with it: where the trailing CNOTs go into the observable, a candidate's
passes leave them out as well.  Results under the chosen shape match the oracle;
tolerances as in test_gpu_parity."""
import numpy as np
import pytest

import oracle
import workloads as wl

pytestmark = pytest.mark.gpu

TOL = {"c128": dict(E=1e-12, G=1e-12), "c64": dict(E=1e-5, G=1e-4)}
LAST = {"c64": (12, 4), "c128": (9, 2)}  # the last shape timed


@pytest.fixture(scope="module")
def sv():
    import torch  # noqa: F401
    import paper_2406_03466_gb300 as m
    return m


def close(got, want, tol):
    got, want = np.asarray(got), np.asarray(want)
    assert float(np.max(np.abs(got - want))) <= tol * max(1.0, float(np.max(np.abs(want))))


@pytest.mark.parametrize("dtype", ["c64", "c128"])
def test_candidates_run_the_later_plan(sv, dtype):
    import torch
    w = wl.qcl(16, 4, 2)
    theta = torch.as_tensor(w.theta, dtype=torch.float64, device="cuda")
    prob = sv.Problem.from_spec(w, dtype)
    t, R = LAST[dtype]
    whole = sv.sv_plan_info(prob.circuit, dtype, sv.plan_opts(tile_bits=t, reg_bits=R))["n_passes"]
    sv.sv_autotune(prob, theta, 2)
    assert sv.sv_last_moved()["passes"] < whole
    sv.sv_autotune(prob, theta, 1)
    t, R, tc, us = sv.sv_tuned_tile(prob, 2)
    _, e_, g_ = sv.sv_grad_adjoint(prob, theta)
    whole = sv.sv_plan_info(prob.circuit, dtype, sv.plan_opts(tile_bits=t, reg_bits=R))["n_passes"]
    assert sv.sv_last_moved()["passes"] < whole and us > 0
    ks = [0, w.n_params // 2, w.n_params - 1]
    _, E, g = oracle.grad_param_shift(w, params=ks)
    close(e_.cpu(), E, TOL[dtype]["E"])
    close(g_.cpu()[ks], g, TOL[dtype]["G"])
    close(sv.sv_energies(prob, theta)[1].cpu(), E, TOL[dtype]["E"])
