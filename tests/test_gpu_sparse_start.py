"""Tile passes leave out amplitudes that are zero because a state starts as one
basis state: circuits that touch every qubit only late, some qubits never, or
none at all, with references that differ in every bit (also within a pair of
real circuits), against the oracle.  Tolerances as in test_gpu_parity."""
import numpy as np
import pytest

import oracle
import workloads as wl

pytestmark = pytest.mark.gpu

TOL = {"c128": dict(E=1e-12, G=1e-12, A=1e-12), "c64": dict(E=1e-5, G=1e-4, A=2e-5)}


@pytest.fixture(scope="module")
def sv():
    import torch  # noqa: F401
    import paper_2406_03466_gb300 as m
    return m


def close(got, want, tol):
    got, want = np.asarray(got), np.asarray(want)
    scale = max(1.0, float(np.max(np.abs(want))))
    assert float(np.max(np.abs(got - want))) <= tol * scale


def circuit(n, kind, real):
    """Gates that spread the state over more and more qubits ("chain"), over the
    top qubits only ("top"), or not at all ("none")."""
    rots = ("RY",) if real else ("RX", "RZ", "RY")
    gates, p = [], 0
    qubits = {"chain": range(n), "top": range(n - 3, n), "none": ()}[kind]
    for rep in range(2):
        for q in qubits:
            for op in rots:
                gates.append(wl.Gate(op, target=q, param=p))
                p += 1
            if q + 1 < n:
                gates.append(wl.Gate("CNOT", target=q + 1, control=q))
    return gates, p


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("real", [True, False])
@pytest.mark.parametrize("kind", ["chain", "top", "none"])
@pytest.mark.parametrize("refs", [[0, 0, 0], [0, 1023, 512, 5], [341, 682]])
def test_sparse_passes_match_oracle(sv, dtype, real, kind, refs):
    import torch
    n = 10
    gates, P = circuit(n, kind, real)
    rng = np.random.default_rng(3)
    letters = rng.choice([0, 1, 3], size=(6, n)).astype(np.int8)
    I = len(refs)
    w = wl.Workload("sparse", n, gates, P, rng.uniform(-3, 3, P), letters, rng.normal(size=6),
                    np.array(refs, dtype=np.int64), weights=rng.uniform(0.2, 1.0, I))
    theta = torch.as_tensor(w.theta, dtype=torch.float64, device="cuda")
    opts = sv.plan_opts(tile_bits=7, reg_bits=2)
    # leave nonzero states of another problem in the library's scratch
    other = wl.qcl(n, 3, 8)
    sv.sv_grad_adjoint(sv.Problem.from_spec(other, dtype, opts=opts),
                       torch.as_tensor(other.theta, device="cuda"), checkpoint_every=1)
    prob = sv.Problem.from_spec(w, dtype, opts=opts)
    E = oracle.instance_energies(w)
    for every in (1, 2):
        _, e_, g_ = sv.sv_grad_adjoint(prob, theta, checkpoint_every=every)
        close(e_.cpu(), E, TOL[dtype]["E"])
        if P:
            close(g_.cpu()[:P], oracle.grad_param_shift(w)[2], TOL[dtype]["G"])
    _, e_ = sv.sv_energies(prob, theta)
    close(e_.cpu(), E, TOL[dtype]["E"])
    # the same states written out into a buffer of garbage, and a batch of
    # problems in one sweep
    st = sv.sv_alloc(n, I, dtype)
    st.tensor.fill_(7.0)
    circ = sv.Circuit(n, gates, P, 0)
    sv.sv_apply_circuit_batch(st, [circ], sv.make_slots([(0, 0, -1, -1, r, 0.0) for r in refs]),
                              theta.reshape(1, -1) if P else None, None, opts)
    for i in range(I):
        close(st.tensor[i].cpu(), oracle.state(w, instance=i), TOL[dtype]["A"])
    if kind != "none":
        probs = [prob, sv.Problem.from_spec(other, dtype, opts=opts)]
        outs = sv.sv_grad_adjoint_multi(probs, [theta, torch.as_tensor(other.theta, device="cuda")])
        close(outs[0][1].cpu(), E, TOL[dtype]["E"])
        close(outs[0][2].cpu()[:P], oracle.grad_param_shift(w)[2], TOL[dtype]["G"])
