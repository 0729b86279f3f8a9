"""Trailing CNOTs taken into the observable, on CPU: the Pauli strings U^dag P U
against dense matrices, and the plan that leaves the CNOTs out."""
import ctypes

import numpy as np
import pytest

from oracle import dense
import workloads as wl

sv = pytest.importorskip("paper_2406_03466_gb300")

I32 = ctypes.c_int32


def _conjugate(n, pairs, letters):
    f = sv.library().sv_debug_conjugate
    f.restype = I32
    tail = (I32 * max(1, 2 * len(pairs)))(*[v for p in pairs for v in p])
    bits = 1 << np.arange(n, dtype=np.uint64)
    x = (np.isin(letters, (1, 2)) * bits).sum(1).astype(np.uint64)
    z = (np.isin(letters, (2, 3)) * bits).sum(1).astype(np.uint64)
    sign = (I32 * len(letters))()
    assert f(tail, len(pairs), len(letters), x.ctypes.data_as(ctypes.c_void_p),
             z.ctypes.data_as(ctypes.c_void_p), sign) == 0
    xb, zb = (x[:, None] & bits) != 0, (z[:, None] & bits) != 0
    return np.where(xb & zb, 2, np.where(xb, 1, np.where(zb, 3, 0))).astype(np.int8), np.array(sign)


@pytest.mark.parametrize("seed", range(4))
def test_conjugated_strings_match_dense(seed):
    n = 4
    rng = np.random.default_rng(seed)
    pairs = [tuple(rng.choice(n, 2, replace=False)) for _ in range(6)]
    U = np.eye(1 << n)
    for c, t in pairs:  # time order: later gates multiply from the left
        j = np.arange(1 << n)
        G = np.zeros_like(U)
        G[j ^ (((j >> c) & 1) << t), j] = 1
        U = G @ U
    letters = rng.integers(0, 4, size=(40, n)).astype(np.int8)
    got, sign = _conjugate(n, pairs, letters)
    for row, new, s in zip(letters, got, sign):
        P = dense.hamiltonian(n, row[None], np.ones(1))
        Q = dense.hamiltonian(n, new[None], np.ones(1))
        np.testing.assert_allclose(U.T @ P @ U, s * Q, atol=1e-14)


@pytest.mark.parametrize("w", [wl.mcvqe(14, 3, "nn+nnn", n_refs=2), wl.qcl(14, 2, 1),
                               wl.ddcl(14, 2), wl.random_workload(14, 60, 4, 1, seed=9)],
                         ids=["ladder", "ring", "no_cnots_at_the_end", "random"])
def test_plan_leaves_out_the_trailing_cnots(w):
    f = sv.library().sv_debug_drop_tail
    f.restype = I32
    d = 0 if w.inputs is None else w.inputs.shape[1]
    circ = sv.Circuit(w.n_qubits, w.gates, w.n_params, d)
    n_passes, n_tail = I32(), I32()
    tail, lay = (I32 * (2 * len(w.gates) + 2))(), (I32 * w.n_qubits)()
    assert f(ctypes.byref(circ.struct), 11, 4, 0, ctypes.byref(n_passes), ctypes.byref(n_tail),
             tail, lay) == 0
    got = [(tail[2 * i], tail[2 * i + 1]) for i in range(n_tail.value)]
    busy, want = set(), []
    for g in reversed(w.gates):
        q = {g.target} | ({g.control} if g.control >= 0 else set())
        if g.op == "CNOT" and not (q & busy):
            want.append((g.control, g.target))
        else:
            busy |= q
    assert got == want[::-1]
    assert sorted(lay) == list(range(w.n_qubits))
    if w.name.startswith("ddcl"):
        assert not got
