"""An instance whose encoded input lies outside [-1, 1] has NaN energies and
leaves every other instance alone, also where two real instances share one
state (on chip above one state an SM, tile passes) and where each has its own.
The others are compared with the same call on valid inputs; where the bad slot
turns shears into 2x2 products only rounding differs.  Tolerances as in
test_gpu_parity."""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu

TOL = {"c128": 1e-12, "c64": 1e-5}


@pytest.fixture(scope="module")
def sv():
    import torch  # noqa: F401
    import paper_2406_03466_gb300 as m
    return m


def ry_circuit(n, layers, instances):
    rng = np.random.default_rng(n + instances)
    gates, p = [wl.Gate("ENC_RY_ASIN", target=q, param=0) for q in range(n)], 0
    for _ in range(layers):
        for q in range(n):
            gates.append(wl.Gate("RY", target=q, param=p))
            p += 1
        gates += wl.cnot_ladder(n)
    letters = rng.choice([0, 1, 3], size=(6, n)).astype(np.int8)
    return wl.Workload("isolation", n, gates, p, rng.uniform(-3, 3, p), letters, rng.normal(size=6),
                       rng.integers(0, 1 << n, instances).astype(np.int64),
                       inputs=rng.uniform(-1, 1, (instances, 1)),
                       weights=rng.uniform(0.2, 1, instances))


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("n,instances", [(8, 2), (8, 305), (11, 155), (14, 3)])
@pytest.mark.parametrize("bad", [0, -1])  # the last of an odd count stands alone
def test_a_nan_instance_stays_alone(sv, dtype, n, instances, bad):
    import torch
    w = ry_circuit(n, 3, instances)
    theta = torch.as_tensor(w.theta, dtype=torch.float64, device="cuda")
    want = [sv.sv_grad_adjoint(sv.Problem.from_spec(w, dtype), theta)[1].cpu().numpy(),
            sv.sv_energies(sv.Problem.from_spec(w, dtype), theta)[1].cpu().numpy()]
    x = w.inputs.copy()
    bads = sorted({bad % instances, (bad + instances // 2) % instances})
    x[bads] = 1.5
    prob = sv.Problem.from_spec(wl.Workload(**{**w.__dict__, "inputs": x}), dtype)
    got = [sv.sv_grad_adjoint(prob, theta)[1].cpu().numpy(), sv.sv_energies(prob, theta)[1].cpu().numpy()]
    ok = np.setdiff1d(np.arange(instances), bads)
    for a, b in zip(got, want):
        assert np.isnan(a[bads]).all()
        scale = max(1.0, float(np.max(np.abs(b))))
        assert float(np.max(np.abs(a[ok] - b[ok]), initial=0.0)) <= TOL[dtype] * scale
