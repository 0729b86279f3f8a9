"""Gradients and energies whose trailing CNOTs are taken into the observable
(default tile shape only), against the oracle and against a fixed tile shape,
which keeps them as passes; Pauli sums of wide strings, whose partners come from
global memory.  Tolerances as in test_gpu_parity."""
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


def with_paulis(w, n_terms, seed):
    rng = np.random.default_rng(seed)
    w.pauli_letters = rng.integers(0, 4, size=(n_terms, w.n_qubits)).astype(np.int8)
    w.pauli_coeffs = rng.normal(size=n_terms)
    return w


CASES = {
    "mcvqe_ladder": lambda: wl.mcvqe(15, 4, "nn+nnn", n_refs=3),
    "qcl_ring": lambda: wl.qcl(15, 3, 2),
    "wide_strings": lambda: with_paulis(wl.qcl(16, 2, 2), 25, 4),
    "real_wide_strings": lambda: with_paulis(wl.mcvqe(15, 3, "nn+nnn", n_refs=2), 20, 5),
}


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("name", sorted(CASES))
def test_trailing_cnots_in_the_observable(sv, dtype, name):
    import torch
    w = CASES[name]()
    theta = torch.as_tensor(w.theta, dtype=torch.float64, device="cuda")
    prob = sv.Problem.from_spec(w, dtype)
    E = oracle.instance_energies(w)
    ks = sorted({0, w.n_params // 2, w.n_params - 1})
    g = oracle.grad_param_shift(w, params=ks)[2]
    for every in (1, 2):
        _, e_, g_ = sv.sv_grad_adjoint(prob, theta, checkpoint_every=every)
        close(e_.cpu(), E, TOL[dtype]["E"])
        close(g_.cpu()[ks], g, TOL[dtype]["G"])
    passes = sv.sv_last_moved()["passes"]
    _, e_ = sv.sv_energies(prob, theta)
    close(e_.cpu(), E, TOL[dtype]["E"])
    outs = sv.sv_grad_adjoint_multi([prob, prob], [theta, theta])
    for _, e_, gm in outs:
        close(e_.cpu(), E, TOL[dtype]["E"])
        close(gm.cpu()[ks], g, TOL[dtype]["G"])
    # the same tile shape, fixed by the caller: every gate in the passes
    opts = sv.plan_opts(tile_bits=11 if dtype == "c64" else 10)
    fixed = sv.Problem.from_spec(w, dtype, opts=opts)
    _, e2, g2 = sv.sv_grad_adjoint(fixed, theta)
    close(e2.cpu(), E, TOL[dtype]["E"])
    close(g2.cpu(), g_.cpu(), TOL[dtype]["G"])
    assert passes <= sv.sv_last_moved()["passes"]
