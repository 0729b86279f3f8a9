"""sv_autotune on chip remembers what later adjoint gradients run: the shape it
reports is the one of the engine that the next call takes, whichever engine that
is, and the results stay those of the untuned call.  Tolerances as in
test_gpu_parity."""
import ctypes

import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu

TOL = {"c128": dict(E=1e-12, G=1e-12), "c64": dict(E=1e-5, G=1e-4)}
FUSED, COMPLEX, PAIR, REAL, TILES = 1, 2, 3, 4, 5


@pytest.fixture(scope="module")
def sv():
    import torch  # noqa: F401
    import paper_2406_03466_gb300 as m
    return m


def last_adjoint(sv):
    v = [ctypes.c_int32() for _ in range(3)]
    assert sv.library().sv_debug_last_adjoint(*[ctypes.byref(x) for x in v]) == 0
    return tuple(x.value for x in v)


def close(got, want, tol):
    got, want = np.asarray(got), np.asarray(want)
    assert float(np.max(np.abs(got - want))) <= tol * max(1.0, float(np.max(np.abs(want))))


def layered(n, layers, ops, instances):
    rng = np.random.default_rng(1000 * n + instances)
    gates = wl.layered_ansatz(n, layers, ops, "ladder")
    p = layers * n * len(ops)
    letters = rng.choice([0, 1, 3], size=(6, n)).astype(np.int8)
    return wl.Workload("tuned", n, gates, p, rng.uniform(-3, 3, p), letters, rng.normal(size=6),
                       rng.integers(0, 1 << n, instances).astype(np.int64),
                       weights=rng.uniform(0.2, 1, instances))


@pytest.mark.parametrize("dtype,n,layers,ops,instances,engine", [
    ("c64", 5, 2, ("RY",), 3, FUSED), ("c64", 8, 3, ("RX", "RZ"), 7, FUSED),
    ("c64", 12, 4, ("RX", "RZ"), 2, COMPLEX), ("c64", 11, 3, ("RY",), 155, PAIR),
    ("c64", 11, 3, ("RY",), 3, REAL), ("c128", 9, 3, ("RX", "RZ"), 3, COMPLEX),
    ("c128", 8, 2, ("RY",), 3, REAL), ("c128", 12, 3, ("RX", "RZ"), 24, TILES)])
def test_tuned_adjoint_is_what_runs(sv, dtype, n, layers, ops, instances, engine):
    import torch
    w = layered(n, layers, ops, instances)
    theta = torch.as_tensor(w.theta, dtype=torch.float64, device="cuda")
    prob = sv.Problem.from_spec(w, dtype)
    want = sv.sv_grad_adjoint(prob, theta)
    assert last_adjoint(sv)[0] == engine
    sv.sv_autotune(prob, theta, 2)
    R, threads, us = sv.sv_tuned_shape(prob, 2)
    assert us > 0
    got = sv.sv_grad_adjoint(prob, theta)
    assert last_adjoint(sv)[0] in (FUSED, engine)
    assert last_adjoint(sv)[1:] == (R, threads)
    for a, b, k in zip(got, want, "EEG"):
        close(a.cpu(), b.cpu(), TOL[dtype][k])
