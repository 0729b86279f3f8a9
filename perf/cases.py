"""What the speed of this library is measured on: twelve calls through its public entry points.

Every case is one gradient, energy or state evaluation as a user's program
makes it, at sizes of this repository's own configurations (``workloads``,
``bench.py`` and the tests): the 4-qubit VQE, the 8- and 28-qubit
multi-contracted VQE, 12- and 20-qubit circuit learning, the 16-qubit
circuit with prepared references, data-driven circuit learning, and a batch of
circuits of different size.  ``draw`` gives sizes between them.

A call's results (loss, instance energies, gradient) lie one behind the other
in one buffer, as a program that fetches them with one transfer has them; a
complex64 problem's results are handed on as float32, the precision they are
computed in, a complex128 problem's as float64.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2406_03466_gb300 as sv

ON_CHIP = 13  # largest complex64 state (qubits) that never leaves the chip


# ------------------------------------------------------------------- the cases

def listed():
    return [
        # the smallest call: a VQE driven by a host optimiser, theta in host
        # memory, loss and gradient back in host memory
        dict(name="vqe4_shift_host_c128", family="vqe", call="shift_host", n=4, layers=2, terms=10,
             instances=1, dtype="c128"),
        # state-averaged MC-VQE on chip: 585 shifted circuits in one launch
        dict(name="mcvqe8_shift_c64", family="mcvqe", call="shift", n=8, layers=4, pairs="all",
             instances=9, dtype="c64"),
        # the same family in double precision by the reverse sweep, odd size
        dict(name="mcvqe11_adjoint_c128", family="mcvqe", call="adjoint", n=11, layers=3,
             pairs="all", instances=12, dtype="c128"),
        # circuit-learning regression on chip: one training step over 256 samples
        dict(name="qcl12_adjoint_c64", family="qcl", call="adjoint", n=12, layers=6, instances=256,
             dtype="c64"),
        # state preparation for later use: 64 states of 20 qubits, written out
        dict(name="qcl20_states_c64", family="qcl", call="states", n=20, layers=10, instances=64,
             dtype="c64"),
        # circuit-learning regression beyond on-chip size: one training step
        dict(name="qcl20_adjoint_c64", family="qcl", call="adjoint", n=20, layers=10, instances=64,
             dtype="c64"),
        # parameter shift of the circuit with prepared (CIS) references: 612
        # circuits of 16 qubits
        dict(name="cis16_shift_c64", family="cis", call="shift", n=16, instances=4, dtype="c64"),
        # double-precision MC-VQE in device memory, odd sizes
        dict(name="mcvqe19_adjoint_c128", family="mcvqe", call="adjoint", n=19, layers=5,
             pairs="nn+nnn", instances=5, dtype="c128"),
        # evaluating an observable with Y factors (no gradient): the forward path
        dict(name="vqe21_energies_c64", family="vqe", call="energies", n=21, layers=4, terms=40,
             instances=3, dtype="c64"),
        # data-driven circuit learning: JS divergence and its gradient
        dict(name="ddcl24_adjoint_c64", family="ddcl", call="adjoint", n=24, layers=10, instances=1,
             dtype="c64"),
        # circuits of different qubit counts and depths in one call
        dict(name="uneven_adjoint_c64", family="uneven", call="adjoint", n_low=15, n_high=19,
             layers_low=3, layers_high=8, circuits=5, instances=8, shapes=3, dtype="c64"),
        # the largest: MC-VQE of 28 qubits, eight references
        dict(name="mcvqe28_adjoint_c64", family="mcvqe", call="adjoint", n=28, layers=8,
             pairs="nn+nnn", instances=8, dtype="c64"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng: random.Random):
    kind = rng.choice(["vqe", "mcvqe_chip", "qcl_chip", "mcvqe_hbm", "mcvqe_hbm", "qcl_hbm", "cis",
                       "energies", "ddcl", "uneven"])
    dtype = rng.choice(["c64", "c64", "c128"])
    if kind == "vqe":
        n = rng.randint(3, 7)
        return dict(family="vqe", call=rng.choice(["shift_host", "shift", "adjoint"]), n=n,
                    layers=rng.randint(1, 4), terms=_log_int(rng, 6, 40), instances=1, dtype=dtype)
    if kind == "mcvqe_chip":
        n = rng.randint(6, 12 if dtype == "c64" else 11)
        return dict(family="mcvqe", call=rng.choice(["shift", "adjoint"]), n=n,
                    layers=rng.randint(2, 6), pairs=rng.choice(["all", "nn+nnn"]),
                    instances=rng.randint(1, n + 1), dtype=dtype)
    if kind == "qcl_chip":
        return dict(family="qcl", call=rng.choice(["adjoint", "adjoint", "energies"]),
                    n=rng.randint(5, 12), layers=rng.randint(2, 8), instances=_log_int(rng, 8, 256),
                    dtype=dtype)
    if kind == "mcvqe_hbm":
        n = rng.randint(14, 26 if dtype == "c64" else 21)
        return dict(family="mcvqe", call=rng.choice(["adjoint", "adjoint", "energies"]), n=n,
                    layers=rng.randint(2, 8), pairs="nn+nnn", instances=rng.randint(1, 8),
                    dtype=dtype)
    if kind == "qcl_hbm":
        n = rng.randint(14, 21 if dtype == "c64" else 19)
        return dict(family="qcl", call=rng.choice(["adjoint", "adjoint", "states"]), n=n,
                    layers=rng.randint(2, 10), instances=_log_int(rng, 2, 64 if n <= 20 else 32),
                    dtype=dtype)
    if kind == "cis":
        return dict(family="cis", call=rng.choice(["shift", "adjoint"]), n=rng.randint(14, 18),
                    instances=rng.randint(1, 6), dtype="c64")
    if kind == "energies":
        return dict(family="vqe", call=rng.choice(["energies", "adjoint"]), n=rng.randint(14, 23),
                    layers=rng.randint(1, 6), terms=_log_int(rng, 8, 60),
                    instances=rng.randint(1, 4), dtype=dtype if rng.random() < 0.5 else "c64")
    if kind == "ddcl":
        return dict(family="ddcl", call="adjoint", n=rng.randint(14, 25),
                    layers=rng.randint(2, 10), instances=1, dtype="c64")
    lo = rng.randint(14, 17)
    return dict(family="uneven", call="adjoint", n_low=lo, n_high=lo + rng.randint(1, 3),
                layers_low=2, layers_high=rng.randint(3, 8), circuits=rng.randint(2, 6),
                instances=_log_int(rng, 2, 16), shapes=rng.randint(0, 10 ** 6), dtype="c64")


# ----------------------------------------------------- circuits and their inputs
# gates are (op, target, control, param, angle), qubit q is bit q of an index

def _ladder(n):
    return [("CNOT", q + 1, q, -1, 0.0) for q in range(n - 1)]


def _layers(n, layers, rots, ring=False):
    gates, p = [], 0
    for _ in range(layers):
        for q in range(n):
            for op in rots:
                gates.append((op, q, -1, p, 0.0))
                p += 1
        gates += _ladder(n)
        if ring:
            gates.append(("CNOT", 0, n - 1, -1, 0.0))
    return gates, p


def _cis_circuit(n):
    """A CIS-like state sum_i c_i |e_i> from |e_0> (angles per instance, from
    inputs), then entanglers on neighbours that share their outer rotations."""
    gates = []
    for i in range(n - 1):
        gates += [("ENC_RY_ASIN", i + 1, -1, 2 * i, 0.0), ("CNOT", i + 1, i, -1, 0.0),
                  ("ENC_RY_ASIN", i + 1, -1, 2 * i + 1, 0.0), ("CNOT", i + 1, i, -1, 0.0),
                  ("CNOT", i, i + 1, -1, 0.0)]
    p = 0
    for a in range(n - 1):
        for q in ([a] if a == 0 else []) + [a + 1]:
            gates.append(("RY", q, -1, p, 0.0))
            p += 1
        for _ in range(2):
            gates.append(("CNOT", a + 1, a, -1, 0.0))
            for q in (a, a + 1):
                gates.append(("RY", q, -1, p, 0.0))
                p += 1
    return gates, p


def _ddcl_circuit(n, layers):
    gates, p = [], 0
    for q in range(0, n - 1, 2):  # neighbours as Bell pairs
        gates += [("H", q, -1, -1, 0.0), ("CNOT", q + 1, q, -1, 0.0)]
    for _ in range(layers):
        for half in range(2):
            for q in range(n):
                for op in ("RZ", "RY", "RZ"):
                    gates.append((op, q, -1, p, 0.0))
                    p += 1
            if half == 0:
                gates += _ladder(n)
    return gates, p


def _spin_rows(n, pairs):
    """Exciton Hamiltonian: Z_A, X_A, then XX, XZ, ZX, ZZ on each pair."""
    if pairs == "all":
        pl = [(a, b) for a in range(n) for b in range(a + 1, n)]
    else:
        pl = [(a, a + 1) for a in range(n - 1)]
        pl += [(a, a + 2) for a in range(n - 2)] if pairs == "nn+nnn" else []
    terms = [[(a, 3)] for a in range(n)] + [[(a, 1)] for a in range(n)]
    for a, b in pl:
        terms += [[(a, x), (b, y)] for x in (1, 3) for y in (1, 3)]
    rows = np.zeros((len(terms), n), dtype=np.int64)
    for t, term in enumerate(terms):
        for q, letter in term:
            rows[t, q] = letter
    return rows, 2 * n


class _Spec:
    """One problem in host memory: circuit, parameters, observable, instances."""

    def __init__(self, case, seed):
        f, n, I = case["family"], case["n"], case["instances"]
        rng = np.random.default_rng(seed)
        self.n, self.dtype = n, case["dtype"]
        self.inputs = self.targets = self.weights = None
        self.input_dim, self.cost = 0, "linear"
        self.refs = np.zeros(I, dtype=np.int64)
        if f == "vqe":
            self.gates, P = _layers(n, case["layers"], ("RY", "RZ"))
            # a random Pauli sum whose structure belongs to the case
            fixed = np.random.default_rng(1000 * n + case["terms"])
            self.letters = fixed.integers(0, 4, size=(case["terms"], n))
            self.coeffs = rng.normal(0.0, 1.0, case["terms"])
            self.refs = (np.arange(I) * 5) % (1 << n)
        elif f in ("mcvqe", "cis"):
            self.letters, one = _spin_rows(n, case.get("pairs", "nn"))
            self.coeffs = np.concatenate([rng.normal(0.0, 0.5, one),
                                          rng.normal(0.0, 0.05, len(self.letters) - one)])
            if f == "mcvqe":
                self.gates, P = _layers(n, case["layers"], ("RY",))
                self.refs = np.array([0] + [1 << i for i in range(I - 1)], dtype=np.int64)
            else:
                self.gates, P = _cis_circuit(n)
                self.refs = np.ones(I, dtype=np.int64)
                x = np.sin(rng.uniform(-np.pi, np.pi, (I, n - 1)) / 2)
                self.input_dim = 2 * (n - 1)
                self.inputs = np.stack([x, -x], axis=2).reshape(I, self.input_dim)
        elif f == "qcl":
            body, P = _layers(n, case["layers"], ("RX", "RZ", "RX"), ring=True)
            self.gates = [(op, q, -1, 0, 0.0) for q in range(n)
                          for op in ("ENC_RY_ASIN", "ENC_RZ_ACOS_SQ")] + body
            self.letters = np.zeros((1, n), dtype=np.int64)
            self.letters[0, 0] = 3
            self.coeffs = np.ones(1)
            x = rng.uniform(-1.0, 1.0, I)
            self.input_dim, self.inputs = 1, x.reshape(-1, 1)
            self.targets, self.cost = np.sin(np.pi * x) + rng.normal(0.0, 0.05, I), "mse"
        else:
            self.gates, P = _ddcl_circuit(n, case["layers"])
            self.letters = np.zeros((1, n), dtype=np.int64)
            self.letters[0, 0] = 3
            self.coeffs = np.ones(1)
        if self.cost == "linear":
            self.weights = np.full(I, 1.0 / I)
        self.n_params = P
        self.theta = rng.uniform(-np.pi, np.pi, P)


def _uneven(case):
    """The circuits of a batch, drawn from the case alone."""
    rng = random.Random(case["shapes"])
    return [dict(family="qcl", call="adjoint", n=rng.randint(case["n_low"], case["n_high"]),
                 layers=rng.randint(case["layers_low"], case["layers_high"]),
                 instances=case["instances"], dtype=case["dtype"])
            for _ in range(case["circuits"])]


def _ddcl_target(n, device):
    """Two discretised Gaussians over the 2^n bitstrings."""
    b = torch.arange(1 << n, dtype=torch.float64, device=device) / float(1 << n)
    p = torch.exp(-0.5 * ((b - 0.25) * 16) ** 2) + torch.exp(-0.5 * ((b - 0.75) * 16) ** 2)
    return p / p.sum()


# ----------------------------------------------------------------- one user call

class _Call:
    """A problem marshalled once, its parameters and its result buffer."""

    def __init__(self, case, seed):
        s = _Spec(case, seed)
        host = case["call"] == "shift_host"
        dev = "cpu" if host else "cuda"

        def on(a, where="cuda"):
            return None if a is None else torch.as_tensor(a, dtype=torch.float64, device=where).contiguous()

        self.single = s.dtype == "c64"
        circuit = sv.Circuit(s.n, s.gates, s.n_params, s.input_dim)
        self.inputs = on(s.inputs)
        self.theta = on(s.theta, dev)
        if case["call"] == "states":
            self.circuits = [circuit]
            self.theta = self.theta.reshape(1, -1)
            self.slots = sv.make_slots((0, 0, -1, i, 0, 0.0) for i in range(len(s.refs)))
            self.states = sv.sv_alloc(s.n, len(s.refs), s.dtype)
            return
        self.problem = sv.Problem(circuit, sv.PauliSum(s.n, s.letters, s.coeffs), s.refs, s.dtype,
                                  inputs=self.inputs, cost=s.cost, weights=on(s.weights),
                                  targets=on(s.targets))
        I, P = len(s.refs), 0 if case["call"] == "energies" else s.n_params
        E = 0 if case["family"] == "ddcl" else I
        self.record = torch.zeros(1 + E + P, dtype=torch.float64, device=dev)
        self.loss, self.energies, self.grad = self.record[:1], self.record[1:1 + E], self.record[1 + E:]
        if case["family"] == "ddcl":
            self.target = _ddcl_target(s.n, "cuda")

    def results(self):
        return self.record.float() if self.single else self.record


def prepare(case, seed):
    if case["family"] == "uneven":
        calls = [_Call(c, 1000 * seed + i) for i, c in enumerate(_uneven(case))]
        return dict(case=case, calls=calls)
    return dict(case=case, call=_Call(case, seed))


def run(state):
    case = state["case"]
    if case["family"] == "uneven":
        calls = state["calls"]
        sv.sv_grad_adjoint_multi([c.problem for c in calls], [c.theta for c in calls],
                                 outputs=[(c.loss, c.energies, c.grad) for c in calls])
        return [c.results() for c in calls]
    c, call = state["call"], case["call"]
    if call == "states":
        sv.sv_apply_circuit_batch(c.states, c.circuits, c.slots, c.theta, c.inputs)
        return c.states.tensor
    if case["family"] == "ddcl":
        sv.sv_grad_ddcl(c.problem, c.theta, c.target, js_out=c.loss, grad_out=c.grad)
    elif call == "energies":
        sv.sv_energies(c.problem, c.theta, energy_out=c.energies, loss_out=c.loss)
    else:
        entry = {"shift": sv.sv_grad_param_shift, "shift_host": sv.sv_grad_param_shift_host,
                 "adjoint": sv.sv_grad_adjoint}[call]
        entry(c.problem, c.theta, energy_out=c.energies, loss_out=c.loss, grad_out=c.grad)
    return c.results()


# ------------------------------------------------------- the work of one pass

_REAL_OPS = ("RY", "X", "H", "CNOT", "ENC_RY_ASIN")


def work(case):
    """Parameters, inputs and (DDCL) target read, results written; 2x2
    products of the rotations merged per qubit (3 operations per real
    amplitude, 14 per complex one), the observable once per set of flipped
    qubits.  A shifted circuit is a circuit of its own; the reverse sweep takes
    a circuit's rotations on two states back."""
    if case["family"] == "uneven":
        parts = [work(c) for c in _uneven(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    s = _Spec(case, 0)
    I, P, dim = len(s.refs), s.n_params, 1 << s.n
    real = all(g[0] in _REAL_OPS for g in s.gates) and not np.any((s.letters == 2).sum(1) % 2)
    merged, open_ = 0, set()
    for g in s.gates:
        if g[0] == "CNOT":
            open_ -= {g[1], g[2]}
        elif g[1] not in open_:
            open_.add(g[1])
            merged += 1
    sweep = merged * dim * (3 if real else 14)
    flips = len({tuple(np.isin(r, (1, 2))) for r in s.letters})
    expect = 0 if case["family"] == "ddcl" else flips * dim * (2 if real else 4)
    io = 8 * (P + 1 + I * (1 + s.input_dim))
    call = case["call"]
    if call == "states":
        return {"bytes": io + I * dim * (8 if s.dtype == "c64" else 16), "flops": I * sweep}
    if call == "energies":
        return {"bytes": io, "flops": I * (sweep + expect)}
    if call in ("shift", "shift_host"):
        return {"bytes": io + 8 * P, "flops": (2 * P + 1) * I * (sweep + expect)}
    target = 8 * dim if case["family"] == "ddcl" else 0
    return {"bytes": io + 8 * P + target, "flops": I * (3 * sweep + expect + P * dim * 2)}


# ------------------------------------------- the same results, in 64 bits

def _seconds(case):
    """About what a 64-bit evaluation of the case takes."""
    if case["family"] == "uneven":
        return sum(_seconds(c) for c in _uneven(case))
    s = _Spec(case, 0)
    real = all(g[0] in _REAL_OPS for g in s.gates) and not np.any((s.letters == 2).sum(1) % 2)
    size = len(s.refs) * (1 << s.n) * (8 if real else 16)
    return (len(s.gates) * (6 if case["call"] in ("states", "energies") else 24)
            + 8 * len(s.letters)) * size / 2.5e12


def _matrix(op, a, real):
    """exp(-i a P / 2) for angles a [B], as [B, 2, 2]."""
    c, s = torch.cos(a / 2), torch.sin(a / 2)
    o = torch.zeros_like(c)
    if op == "RY":
        m = torch.stack([torch.stack([c, -s], -1), torch.stack([s, c], -1)], -2)
        return m if real else m.to(torch.complex128)
    if op == "RX":
        m = [[torch.complex(c, o), torch.complex(o, -s)], [torch.complex(o, -s), torch.complex(c, o)]]
    else:
        m = [[torch.complex(c, -s), torch.complex(o, o)], [torch.complex(o, o), torch.complex(c, s)]]
    return torch.stack([torch.stack(r, -1) for r in m], -2)


def _apply(m, q, v, n):
    """m [B or 1, 2, 2] on qubit q of v [B, 2^n], in place."""
    w = v.view(v.shape[0], 1 << (n - 1 - q), 2, 1 << q)
    m = m.reshape(m.shape[0], 4, 1, 1)
    a, b = w[:, :, 0], w[:, :, 1]
    x = a * m[:, 0] + b * m[:, 1]
    y = a * m[:, 2] + b * m[:, 3]
    a.copy_(x)
    b.copy_(y)


def _cnot(c, t, v, n):
    hi, lo = max(c, t), min(c, t)
    w = v.view(v.shape[0], 1 << (n - 1 - hi), 2, 1 << (hi - lo - 1), 2, 1 << lo)
    p, q = (w[:, :, 1, :, 0], w[:, :, 1, :, 1]) if c == hi else (w[:, :, 0, :, 1], w[:, :, 1, :, 1])
    x = p.clone()
    p.copy_(q)
    q.copy_(x)


def _times_h(s, v):
    """H v: per set of flipped qubits, the diagonal of its terms, then the flip."""
    j = torch.arange(1 << s.n, device=v.device)
    out, groups = torch.zeros_like(v), {}
    for row, c in zip(s.letters, s.coeffs):
        x = sum(1 << q for q in range(s.n) if row[q] in (1, 2))
        groups.setdefault(x, []).append((sum(1 << q for q in range(s.n) if row[q] in (2, 3)),
                                         c * 1j ** int((row == 2).sum())))
    for x, terms in groups.items():
        d = torch.zeros(1 << s.n, dtype=v.dtype, device=v.device)
        for z, c in terms:
            odd = j & z
            for k in (16, 8, 4, 2, 1):
                odd = odd ^ (odd >> k)
            d += (1 - 2 * (odd & 1)).to(v.dtype) * (c if v.is_complex() else c.real)
        out += (d * v)[:, j ^ x] if x else d * v
    return out


def _exact_one(case, seed):
    dev, s = "cuda" if torch.cuda.is_available() else "cpu", _Spec(case, seed)
    n, I = s.n, len(s.refs)
    real = all(g[0] in _REAL_OPS for g in s.gates) and not np.any((s.letters == 2).sum(1) % 2)
    kind = torch.float64 if real and case["call"] != "states" else torch.complex128
    real = kind == torch.float64
    theta = torch.as_tensor(s.theta, device=dev)
    inputs = None if s.inputs is None else torch.as_tensor(s.inputs, device=dev)

    def matrix(g):
        op, _, _, p, angle = g
        if op == "H":
            return torch.tensor([[[1.0, 1.0], [1.0, -1.0]]], dtype=kind, device=dev) / math.sqrt(2.0)
        if op == "ENC_RY_ASIN":
            return _matrix("RY", torch.asin(inputs[:, p]), real)
        if op == "ENC_RZ_ACOS_SQ":
            return _matrix("RZ", torch.acos(inputs[:, p] ** 2), real)
        return _matrix(op, theta[p:p + 1], real)

    psi = torch.zeros(I, 1 << n, dtype=kind, device=dev)
    psi[torch.arange(I, device=dev), torch.as_tensor(s.refs, device=dev)] = 1
    for g in s.gates:
        if g[0] == "CNOT":
            _cnot(g[2], g[1], psi, n)
        else:
            _apply(matrix(g), g[1], psi, n)
    if case["call"] == "states":
        return psi
    if case["family"] == "ddcl":
        P, Q = _ddcl_target(n, dev), psi[0].abs() ** 2
        M = (P + Q) / 2
        zero = torch.zeros_like(P)
        ratio = torch.where(Q > 0, torch.log(Q / M), zero)
        loss = 0.5 * (torch.where(P > 0, P * torch.log(P / M), zero) + Q * ratio).sum()
        lam, weight = psi * (0.5 * ratio), torch.ones(1, dtype=torch.float64, device=dev)
        E = torch.zeros(0, dtype=torch.float64, device=dev)
    else:
        lam = _times_h(s, psi)
        E = (psi.conj() * lam).sum(1).real if psi.is_complex() else (psi * lam).sum(1)
        if s.cost == "mse":
            y = torch.as_tensor(s.targets, device=dev)
            loss, weight = ((E - y) ** 2).mean(), 2 * (E - y) / I
        else:
            weight = torch.as_tensor(s.weights, device=dev)
            loss = (weight * E).sum()
    if case["call"] == "energies":
        return torch.cat([loss.reshape(1), E])
    grad = torch.zeros(s.n_params, dtype=torch.float64, device=dev)
    for g in reversed(s.gates):
        op, q, c, p, _ = g
        if op == "CNOT":
            _cnot(c, q, psi, n)
            _cnot(c, q, lam, n)
            continue
        if op in ("RX", "RY", "RZ"):
            w = psi.view(I, 1 << (n - 1 - q), 2, 1 << q)
            l = lam.view(I, 1 << (n - 1 - q), 2, 1 << q)
            a, b, u, v = w[:, :, 0], w[:, :, 1], l[:, :, 0].conj(), l[:, :, 1].conj()
            if op == "RY":
                d = v * a - u * b
                d = d.real if d.is_complex() else d
            else:
                d = (u * b + v * a).imag if op == "RX" else (u * a - v * b).imag
            grad[p] += (weight * d.sum((1, 2))).sum()
        m = matrix(g)
        m = m.transpose(1, 2).conj()
        _apply(m, q, psi, n)
        _apply(m, q, lam, n)
    return torch.cat([loss.reshape(1), E, grad])


def exact(case, seed):
    if _seconds(case) > 15:
        return None
    if case["family"] == "uneven":
        return [_exact_one(c, 1000 * seed + i) for i, c in enumerate(_uneven(case))]
    return _exact_one(case, seed)
