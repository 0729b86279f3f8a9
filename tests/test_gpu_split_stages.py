"""Complex groups run as real rotations between phase products (tile passes):
groups whose rotation is none, a quarter turn or a half turn (c or s exactly or
nearly zero), one to four groups a stage, mixed with real groups, against the
oracle.  Tolerances as in test_gpu_parity."""
import numpy as np
import pytest

import oracle
import workloads as wl

pytestmark = pytest.mark.gpu

TOL = {"c128": dict(E=1e-12, G=1e-12, A=1e-12), "c64": dict(E=1e-5, G=1e-4, A=2e-5)}
# single-qubit groups as (op, parametrised) lists; angles are drawn below
GROUPS = [["RZ"], ["RX", "RZ", "RX"], ["RZ", "RY", "RZ"], ["H", "RZ"], ["X", "RZ"], ["RY"],
          ["RX"], ["RZ", "H", "RX"], ["H"], ["RY", "RZ"]]
ANGLES = [0.0, np.pi, -np.pi, np.pi / 2, 1e-9, np.pi - 1e-7, 2.0, -3.0, 5.0]


@pytest.fixture(scope="module")
def sv():
    import torch  # noqa: F401
    import paper_2406_03466_gb300 as m
    return m


def close(got, want, tol):
    got, want = np.asarray(got), np.asarray(want)
    scale = max(1.0, float(np.max(np.abs(want))))
    assert float(np.max(np.abs(got - want))) <= tol * scale


def workload(n, layers, width, seed):
    """Per layer, groups on `width` neighbouring qubits, then CNOTs around them."""
    rng = np.random.default_rng(seed)
    gates, theta = [], []
    for layer in range(layers):
        for j in range(width):
            q = (layer * width + j) % n
            for op in GROUPS[rng.integers(len(GROUPS))]:
                if op in ("X", "H"):
                    gates.append(wl.Gate(op, target=q))
                else:
                    gates.append(wl.Gate(op, target=q, param=len(theta)))
                    theta.append(ANGLES[rng.integers(len(ANGLES))])
        for j in range(width):
            a = (layer * width + j) % n
            gates.append(wl.Gate("CNOT", target=(a + 1) % n, control=a))
    letters, coeffs = wl.random_pauli_sum(n, 6, seed)
    return wl.Workload("split", n, gates, len(theta), np.array(theta), letters, coeffs,
                       rng.integers(0, 1 << n, size=2).astype(np.int64),
                       weights=rng.uniform(0.2, 1.0, 2))


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("width", [1, 2, 3, 4])
@pytest.mark.parametrize("tile_bits,reg_bits", [(7, 2), (8, 3), (9, 4)])
def test_split_stages_match_oracle(sv, dtype, width, tile_bits, reg_bits):
    import torch
    reg_bits = min(reg_bits, 3) if dtype == "c128" else reg_bits
    w = workload(9, 10, width, 10 * width + tile_bits)
    opts = sv.plan_opts(tile_bits=tile_bits, reg_bits=reg_bits)
    prob = sv.Problem.from_spec(w, dtype, opts=opts)
    theta = torch.as_tensor(w.theta, dtype=torch.float64, device="cuda")
    L, E, g = oracle.grad_param_shift(w)
    for every in (1, 3):
        _, e_, g_ = sv.sv_grad_adjoint(prob, theta, checkpoint_every=every)
        close(e_.cpu(), E, TOL[dtype]["E"])
        close(g_.cpu()[: w.n_params], g, TOL[dtype]["G"])
    circ = sv.Circuit(w.n_qubits, w.gates, w.n_params, 0)
    st = sv.sv_alloc(w.n_qubits, 2, dtype)
    rows = [(0, 0, -1, -1, int(w.refs[i]), 0.0) for i in range(2)]
    sv.sv_apply_circuit_batch(st, [circ], sv.make_slots(rows), theta.reshape(1, -1), None, opts)
    for i in range(2):
        close(st.tensor[i].cpu(), oracle.state(w, instance=i), TOL[dtype]["A"])
