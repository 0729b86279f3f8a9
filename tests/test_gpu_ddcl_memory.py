"""sv_grad_ddcl keeps one set of states per stream: growing circuits leave no
outgrown buffer behind, and a repeated call stores as many states as the first."""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sv():
    import torch  # noqa: F401
    import paper_2406_03466_gb300 as m
    return m


def test_ddcl_keeps_one_buffer(sv):
    import torch
    sizes = (20, 21, 22)
    args = {}
    for n in sizes:
        w = wl.ddcl(n, 1, seed=n)
        args[n] = (sv.Problem.from_spec(w, "c64"), torch.as_tensor(w.theta, device="cuda"),
                   torch.as_tensor(w.target_dist, dtype=torch.float64, device="cuda"))
        sv.sv_grad_ddcl(*args[n])  # plans and descriptors
    torch.cuda.synchronize()

    def held(calls):  # device memory that the calls leave held on a new stream
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        out = [torch.empty(1, dtype=torch.float64, device="cuda"),
               torch.empty(max(a[1].numel() for a in args.values()), dtype=torch.float64, device="cuda")]
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        every = []
        for n in calls:
            prob, theta, target = args[n]
            sv.sv_grad_ddcl(prob, theta, target, js_out=out[0], grad_out=out[1][: theta.numel()], stream=s)
            s.synchronize()
            every.append(sv.sv_last_adjoint_info()["checkpoint_every"])
        return before - torch.cuda.mem_get_info()[0], every

    alone, _ = held([22])
    grown, every = held([20, 21, 22, 22])
    assert alone >= 3 * 8 << 22  # psi, lambda and a stored state
    assert grown <= alone + (4 << 20)  # allocation granularity
    assert every[2] == every[3]
