"""Real circuits whose states share one complex state two by two (tile passes):
odd and even slot counts, rotations with negative cos(theta/2), groups of several
rotations and of X / H / CZ, both costs, every entry point that pairs slots,
against the oracle.  Tolerances as in test_gpu_parity."""
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


def real_workload(n, n_gates, instances, seed, cost, encoding):
    """Random real circuit (angles beyond pi: cos(theta/2) of both signs) and a
    Pauli sum with even Y counts, over `instances` distinct references."""
    rng = np.random.default_rng(seed)
    ops = ("RY", "RY", "RY", "CNOT", "CNOT", "X", "H", "CZ")
    gates, P, theta = wl.random_circuit(n, n_gates, seed, ops=ops)
    inputs = None
    if encoding:
        gates = [wl.Gate("ENC_RY_ASIN", target=q, param=0) for q in range(n)] + gates
        inputs = rng.uniform(-1.0, 1.0, (instances, 1))
        inputs[0] = 1.0
    letters = rng.integers(0, 4, size=(8, n)).astype(np.int8)
    odd = (letters == 2).sum(1) % 2 == 1
    letters[odd, 0] = np.where(letters[odd, 0] == 2, 1, 2)
    refs = rng.integers(0, 1 << n, size=instances).astype(np.int64)
    return wl.Workload("real", n, gates, P, 2.5 * theta, letters, rng.normal(size=8), refs,
                       inputs=inputs, cost=cost,
                       weights=rng.uniform(0.2, 1.0, instances) if cost == "linear" else None,
                       targets=rng.normal(size=instances) if cost == "mse" else None)


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("n,instances,tile_bits,reg_bits,cost,encoding", [
    (7, 2, 7, 2, "linear", False), (8, 3, 7, 2, "mse", True), (9, 5, 8, 3, "linear", True),
    (10, 4, 9, 4, "mse", False), (11, 3, 10, 4, "linear", False), (9, 1, 7, 2, "linear", True)])
def test_paired_slots_match_oracle(sv, dtype, n, instances, tile_bits, reg_bits, cost, encoding):
    import torch
    reg_bits = min(reg_bits, 3) if dtype == "c128" else reg_bits
    w = real_workload(n, 70, instances, 7 * n + instances, cost, encoding)
    opts = sv.plan_opts(tile_bits=tile_bits, reg_bits=reg_bits)
    prob = sv.Problem.from_spec(w, dtype, opts=opts)
    theta = torch.as_tensor(w.theta, dtype=torch.float64, device="cuda")
    L, E, g = oracle.grad_param_shift(w)
    for every in (1, 2, 0):
        l_, e_, g_ = sv.sv_grad_adjoint(prob, theta, checkpoint_every=every)
        close(l_.cpu(), [L], TOL[dtype]["E"])
        close(e_.cpu(), E, TOL[dtype]["E"])
        close(g_.cpu()[: w.n_params], g, TOL[dtype]["G"])
    assert sv.sv_last_adjoint_states() == (instances + 1) // 2
    l_, e_, g_ = sv.sv_grad_param_shift(prob, theta)
    close(e_.cpu(), E, TOL[dtype]["E"])
    close(g_.cpu()[: w.n_params], g, TOL[dtype]["G"])
    l_, e_ = sv.sv_energies(prob, theta)
    close(e_.cpu(), E, TOL[dtype]["E"])
    # a segment of the shifted batch that begins and ends inside a pair
    full = sv.sv_param_shift_energies(prob, theta).cpu()
    part = sv.sv_param_shift_energies_range(prob, theta, 1, 6).cpu()
    close(part, full[1:7], TOL[dtype]["E"])


def test_complex_observable_is_not_paired(sv):
    """One Y in a term makes H complex: the instances keep a state each."""
    import torch
    w = real_workload(8, 40, 2, 5, "linear", False)
    w.pauli_letters[0] = 0
    w.pauli_letters[0, 3] = 2
    prob = sv.Problem.from_spec(w, "c128", opts=sv.plan_opts(tile_bits=7, reg_bits=2))
    _, e_, g_ = sv.sv_grad_adjoint(prob, torch.as_tensor(w.theta, device="cuda"))
    assert sv.sv_last_adjoint_states() == 2
    L, E, g = oracle.grad_param_shift(w)
    close(e_.cpu(), E, 1e-12)
    close(g_.cpu()[: w.n_params], g, 1e-12)
