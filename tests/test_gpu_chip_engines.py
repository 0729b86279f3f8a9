"""Each kind of on-chip adjoint state (complex, paired real, single real) by the
default route, with the engine that ran asserted: both precisions, the register
widths the route picks, odd instance counts on both sides of one state an SM,
and groups of several rotations, of X and H, without parameters, and of shared
parameters.  Energies and some derivatives against the oracle, whole gradients
against the one-kernel engine in complex128.  Tolerances as in test_gpu_parity."""
import numpy as np
import pytest

import oracle
import workloads as wl
from test_gpu_autotune_engines import COMPLEX, FUSED, PAIR, REAL, TILES, last_adjoint

pytestmark = pytest.mark.gpu

TOL = {"c128": dict(E=1e-12, G=1e-12), "c64": dict(E=1e-5, G=1e-4)}


@pytest.fixture(scope="module")
def sv():
    import torch  # noqa: F401
    import paper_2406_03466_gb300 as m
    return m


def close(got, want, tol):
    got, want = np.asarray(got), np.asarray(want)
    assert float(np.max(np.abs(got - want))) <= tol * max(1.0, float(np.max(np.abs(want))))


def workload(n, layers, instances, real, shared=False, every=False):
    """`layers` layers of one group on every qubit (every: all with parameters),
    each ending in CNOTs."""
    rng = np.random.default_rng(100 * n + layers + instances)
    gates, p = [wl.Gate("ENC_RY_ASIN", target=0, param=0)], 0
    kinds = ([["RY"], ["RY", "RY"], ["fixed"], ["fixed", "RY"]] if real else
             [["RX", "RZ"], ["RY"], ["H", "RZ"], ["X", "RZ"] if every else ["X"], ["RZ", "RX", "RZ"],
              ["RY", "fixed", "H"]])
    for layer in range(layers):
        for q in range(n):
            for op in kinds[rng.integers(len(kinds))]:
                if op == "fixed":
                    gates.append(wl.Gate("RY", target=q, angle=0.7))
                elif op in ("X", "H"):
                    gates.append(wl.Gate(op, target=q))
                else:
                    gates.append(wl.Gate(op, target=q, param=p))
                    p += 1
        gates += wl.cnot_ring(n) if layer % 2 else wl.cnot_ladder(n)
    if shared:
        gates = [wl.Gate(g.op, g.target, g.control, g.param % 5, g.angle)
                 if g.param >= 0 and not g.op.startswith("ENC") else g for g in gates]
        p = min(p, 5)
    letters = rng.choice([0, 1, 3], size=(7, n)).astype(np.int8)
    if not real:
        letters[0, 0] = 2
    return wl.Workload("engines", n, gates, p, rng.uniform(-6, 6, p), letters, rng.normal(size=7),
                       rng.integers(0, 1 << n, instances).astype(np.int64),
                       inputs=rng.uniform(-1, 1, (instances, 1)), weights=rng.uniform(0.2, 1, instances))


CASES = [("c64", False, 8, 33, 2), ("c64", False, 10, 7, 3), ("c64", False, 11, 4, 2), ("c64", False, 10, 4, 305),
         ("c64", False, 12, 4, 3), ("c64", False, 12, 2, 153), ("c64", False, 13, 3, 1),
         ("c64", True, 11, 3, 152), ("c64", True, 11, 3, 153), ("c64", True, 11, 3, 305), ("c64", True, 12, 2, 3),
         ("c64", True, 12, 2, 153), ("c64", True, 12, 2, 306), ("c64", True, 13, 1, 1), ("c64", True, 13, 1, 155),
         ("c128", False, 7, 5, 3), ("c128", False, 9, 2, 153), ("c128", False, 11, 2, 2),
         ("c128", True, 7, 1, 1), ("c128", True, 7, 2, 153), ("c128", True, 9, 2, 305), ("c128", True, 12, 2, 2),
         ("c128", True, 11, 2, 155)]


@pytest.mark.parametrize("shared", [False, True])
@pytest.mark.parametrize("dtype,real,n,layers,instances", CASES)
def test_engine_of_the_default_route(sv, dtype, real, n, layers, instances, shared):
    import torch
    w = workload(n, layers, instances, real, shared, every=dtype == "c128")
    theta = torch.as_tensor(w.theta, dtype=torch.float64, device="cuda")
    _, e_, g_ = sv.sv_grad_adjoint(sv.Problem.from_spec(w, dtype), theta)
    few = dtype == "c128" and not real and n >= 11  # few large states: tile passes
    assert last_adjoint(sv)[0] == (TILES if few else COMPLEX if not real else PAIR if instances > 152 else REAL)
    close(e_.cpu(), oracle.instance_energies(w), TOL[dtype]["E"])
    if not shared:
        ks = sorted({0, w.n_params // 2, w.n_params - 1})
        close(g_.cpu()[ks], oracle.grad_param_shift(w, params=ks)[2], TOL[dtype]["G"])
    fixed = sv.Problem.from_spec(w, "c128", opts=sv.plan_opts(**(dict(reg_bits=3) if n < 13 else dict(tile_bits=10))))
    close(g_.cpu(), sv.sv_grad_adjoint(fixed, theta)[2].cpu(), TOL[dtype]["G"])


@pytest.mark.parametrize("dtype", ["c64", "c128"])
def test_ladder_runs_fewer_passes(sv, dtype):
    """The trailing CNOTs of a layered circuit really leave its passes."""
    import torch
    w = wl.qcl(15, 3, 2)
    theta = torch.as_tensor(w.theta, dtype=torch.float64, device="cuda")
    sv.sv_grad_adjoint(sv.Problem.from_spec(w, dtype), theta)
    passes = sv.sv_last_moved()["passes"]
    fixed = sv.Problem.from_spec(w, dtype, opts=sv.plan_opts(tile_bits=11 if dtype == "c64" else 10))
    sv.sv_grad_adjoint(fixed, theta)
    assert passes < sv.sv_last_moved()["passes"]


@pytest.mark.parametrize("n,layers,ops,engine", [
    (8, 2, ("RX", "RZ"), COMPLEX), (8, 7, ("H",), FUSED), (10, 3, ("mixed",), FUSED), (8, 1, ("RX", "RZ"), FUSED)])
def test_line_between_the_complex128_engines(sv, n, layers, ops, engine):
    """Complex circuits go to the engine of split stages when their groups carry
    parameters and there is enough of them."""
    import torch
    rng = np.random.default_rng(n + layers)
    gates, p = [], 0
    for layer in range(layers):
        for q in range(n):
            for op in (("X", "H") if (q + layer) % 3 else ("RZ", "RX")) if ops == ("mixed",) else ops:
                rot = op in ("RX", "RY", "RZ")
                gates.append(wl.Gate(op, target=q, param=p if rot else -1))
                p += rot
        gates += wl.cnot_ladder(n)
    gates.append(wl.Gate("RZ", target=0, param=p))
    w = wl.Workload("line", n, gates, p + 1, rng.uniform(-3, 3, p + 1),
                    rng.choice([0, 1, 2, 3], size=(5, n)).astype(np.int8), rng.normal(size=5),
                    rng.integers(0, 1 << n, 3).astype(np.int64), weights=np.ones(3))
    theta = torch.as_tensor(w.theta, dtype=torch.float64, device="cuda")
    _, e_, g_ = sv.sv_grad_adjoint(sv.Problem.from_spec(w, "c128"), theta)
    assert last_adjoint(sv)[0] == engine
    ks = sorted({0, w.n_params - 1})
    _, E, g = oracle.grad_param_shift(w, params=ks)
    close(e_.cpu(), E, 1e-12)
    close(g_.cpu()[ks], g, 1e-12)
