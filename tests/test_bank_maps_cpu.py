"""Bank maps of the tile passes' shared-memory exchanges, on CPU: in the layered
circuits the lanes of one wavefront (16 of 8 bytes, 8 of 16 bytes) hit distinct
banks on both sides of every exchange, so their address vectors are independent
in the low bits."""
import pytest

import workloads as wl
from test_tile_passes_cpu import export, sv


def rank(vectors, bits):
    basis = {}
    for x in vectors:
        x &= (1 << bits) - 1
        while x:
            h = x.bit_length()
            if h not in basis:
                basis[h] = x
                break
            x ^= basis[h]
    return len(basis)


@pytest.mark.parametrize("dtype,t,R", [(0, 11, 4), (0, 10, 4), (0, 12, 4), (1, 10, 3), (1, 10, 2)])
@pytest.mark.parametrize("make", [lambda: wl.mcvqe(16, 4, "nn+nnn", n_refs=1),
                                  lambda: wl.mcvqe(28, 8, "nn+nnn", n_refs=1), lambda: wl.qcl(20, 10, 1)])
def test_exchanges_have_no_conflicts(make, dtype, t, R):
    w = make()
    csz, bits = (16, 3) if dtype else (8, 4)
    circ = sv.Circuit(w.n_qubits, w.gates, w.n_params, 0 if w.inputs is None else 1)
    for relabel in (False, True):
        for P in export(circ, t, R, True, dtype, relabel)[2]:
            lanes = min(bits, P.t - P.R)
            for e in range(P.n_stages + 1):
                sides = (P.ldperm if e == 0 else P.st[e - 1].stt, P.nat if e == P.n_stages else P.st[e].ldt)
                for v in sides:
                    assert rank([v[k] // csz for k in range(lanes)], bits) == lanes
