"""Batches of circuits (sv_grad_adjoint_multi) and the options of their problems:
a call with other options plans and records its own graph instead of replaying
that of an earlier call on the same pointers, and problems whose tile shapes
differ are refused.  Tolerances as in test_gpu_parity."""
import numpy as np
import pytest

import oracle
import workloads as wl

pytestmark = pytest.mark.gpu

KEEP = []  # the calls' tensors: another case's pointers must be others


@pytest.fixture(scope="module")
def sv():
    import torch  # noqa: F401
    import paper_2406_03466_gb300 as m
    return m


def close(got, want, tol):
    got, want = np.asarray(got), np.asarray(want)
    assert float(np.max(np.abs(got - want))) <= tol * max(1.0, float(np.max(np.abs(want))))


@pytest.mark.parametrize("opts", [dict(no_relabel=True), dict(no_fusion=True), dict(tile_bits=11, reg_bits=4),
                                  dict(coalesce_bits=3)])
def test_options_plan_anew(sv, opts):
    import torch
    w = wl.mcvqe(18, 2, "nn+nnn", n_refs=4)
    theta = torch.as_tensor(w.theta, dtype=torch.float64, device="cuda")
    E = oracle.instance_energies(w)
    f = dict(dtype=torch.float64, device="cuda")
    outs = [(torch.empty(1, **f), torch.empty(w.n_instances, **f), torch.empty(w.n_params, **f))]
    prob = sv.Problem.from_spec(w, "c64")
    KEEP.append((theta, outs, prob))
    held = []
    for o in (None, None, sv.plan_opts(**opts)):
        prob.struct.opts = None if o is None else sv.ctypes.pointer(o)
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        sv.sv_grad_adjoint_multi([prob], [theta], outputs=outs)
        torch.cuda.synchronize()
        held.append(before - torch.cuda.mem_get_info()[0])
        close(outs[0][1].cpu(), E, 1e-5)
    states = 2 * w.n_instances * 8 << w.n_qubits  # psi and lambda
    assert held[0] >= states and held[1] < states and held[2] >= states


def test_mixed_tile_shapes_are_refused(sv):
    """A fixed tile of 2^10 amplitudes is one of 2^9 for the 9-qubit problem."""
    import torch
    ws = [wl.mcvqe(n, 1, "nn", n_refs=2) for n in (9, 14)]
    probs = [sv.Problem.from_spec(w, "c64", opts=sv.plan_opts(tile_bits=10, reg_bits=4)) for w in ws]
    thetas = [torch.as_tensor(w.theta, dtype=torch.float64, device="cuda") for w in ws]
    for k in (1, -1):
        with pytest.raises(Exception, match="one tile shape"):
            sv.sv_grad_adjoint_multi(probs[::k], thetas[::k])


def test_default_shapes_of_complex128_agree(sv):
    """14 and 17 qubits alone have different default register bits."""
    import torch
    ws = [wl.mcvqe(n, 1, "nn", n_refs=2) for n in (14, 17)]
    thetas = [torch.as_tensor(w.theta, dtype=torch.float64, device="cuda") for w in ws]
    outs = sv.sv_grad_adjoint_multi([sv.Problem.from_spec(w, "c128") for w in ws], thetas)
    for w, (_, e_, _) in zip(ws, outs):
        close(e_.cpu(), oracle.instance_energies(w), 1e-12)
