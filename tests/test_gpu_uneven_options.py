"""Batches of circuits (sv_grad_adjoint_multi) and the options of their problems:
a call with other options plans and records its own graph instead of replaying
that of an earlier call on the same pointers.  Tolerances as in test_gpu_parity."""
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
