"""The H passes of large Pauli sums stay within a block's shared memory, on CPU:
groups that a pass takes over from a later one must not push it past that."""
import ctypes

import numpy as np
import pytest

import workloads as wl
from test_tile_passes_cpu import HClass, HGroup, HRow, HTerm, export_h, sv

LIMIT = 227 * 1024  # bytes a block


def smem(P, csz):
    """Dynamic shared memory of one block of k_tile_h (tile_h_smem)."""
    vals = (1 << P.R) * (1 if P.real else 2)
    return (3 * (csz << P.t) + P.n_rows * (vals * csz // 2 + ctypes.sizeof(HRow))
            + P.n_groups * ctypes.sizeof(HGroup) + P.n_classes * (csz + 8 + ctypes.sizeof(HClass))
            + P.n_terms * ctypes.sizeof(HTerm) + 32 * 8 + 16)


def plan(n, terms, seed, c128, mask=None):
    """(every pass's bytes, groups moved into the first pass)"""
    letters, coeffs = wl.random_pauli_sum(n, terms, seed)
    if mask is not None:  # at most `mask` letters a string
        rng = np.random.default_rng(seed)
        for row in letters:
            row[rng.permutation(n)[mask:]] = 0
    t, c = (11, 3) if c128 else (12, 4)
    passes, groups = export_h(sv.PauliSum(n, letters, coeffs), t, c)[:2]
    g0 = passes[0].groups or 0
    moved = [g for g in groups[g0:g0 + passes[0].n_groups]
             if g.xfar and bin(g.xfar | (1 << c) - 1).count("1") <= t]
    assert sum(P.n_terms for P in passes) == terms
    return [smem(P, 16 if c128 else 8) for P in passes], moved


@pytest.mark.parametrize("c128,terms", [(False, 620), (False, 660), (False, 700), (True, 640)])
def test_large_sums_fit_a_block(c128, terms):
    need, _ = plan(26, terms, 1, c128)
    assert max(need) <= LIMIT


def test_small_sums_still_move():
    """40 strings of up to 10 letters over 22 qubits: later passes of one group are taken over."""
    _, moved = plan(22, 40, 22, False, 10)
    assert moved
