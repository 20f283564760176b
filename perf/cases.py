"""Performance cases: the work users have the state-vector simulator do.

Each listed case is one family of calls at one size; ``draw`` gives other
sizes of the same families.  Circuits are seeded and synthetic, of the shapes
the paper evaluates (grid random circuits, quantum multipliers) and of the
ones around it (random U3 + CZ circuits, variational training of a
hardware-efficient ansatz, batches of uneven circuits, read-out of a finished
state, gates applied one call at a time).  A state starts at |0...0> where a
circuit is run, and is a random dense vector (complex Gaussian amplitudes, as
a random circuit leaves them, each qubit tilted towards 0 or 1 as in a state
whose energy or <Z> is of interest) where it is read out.  Parameters and
gradients of a training step are float32, as an optimiser keeps them.
"""
import ctypes as C
import math
import random

import numpy as np
import torch

from paper_2106_13995_gb300 import _native as N
from paper_2106_13995_gb300 import circuit as B
from paper_2106_13995_gb300 import sim

PI = math.pi


# ---- cases ----------------------------------------------------------------
def listed():
    return [
        # a small state in double precision: reference runs and unit tests of
        # a circuit, where launches and latency count
        {"name": "u3cz 12q c128", "family": "u3cz", "n": 12, "layers": 20, "dtype": "c128"},
        # one mid-size random circuit, default options
        {"name": "u3cz 18q c64", "family": "u3cz", "n": 18, "layers": 40, "dtype": "c64"},
        # a grid circuit narrowed to an even width, default options (FP32)
        {"name": "grid 26q c64", "family": "grid", "n": 26, "cycles": 20, "dtype": "c64", "prec": "plain"},
        # the headline workload: the full lattice with split-BF16 blocks
        {"name": "grid 30q bf16x3", "family": "grid", "n": 30, "cycles": 20, "dtype": "c64", "prec": "bf16x3"},
        # a grid circuit in double precision at an odd width
        {"name": "grid 23q c128", "family": "grid", "n": 23, "cycles": 20, "dtype": "c128", "prec": "plain"},
        # reversible arithmetic on superposed inputs
        {"name": "multiplier 29q", "family": "mult", "nbits": 7},
        # gates applied by one call each, as interactive code does
        {"name": "gates 27q", "family": "gates", "n": 27, "dtype": "c64"},
        # one step of variational training
        {"name": "gradient 16q", "family": "grad", "n": 16, "layers": 6, "sets": 1},
        # the same over many parameter sets in one call
        {"name": "gradient 20q x64", "family": "grad", "n": 20, "layers": 10, "sets": 64},
        # many unrelated circuits of uneven widths in one call
        {"name": "uneven batch x48", "family": "batch", "count": 48, "nmin": 10, "nmax": 22, "depth": 40},
        # the energy of a transverse-field Ising chain on a finished state
        {"name": "ising energy 28q", "family": "energy", "n": 28, "dtype": "c64"},
        # read-out of a finished state: <Z> of every qubit, norm, shots
        {"name": "read-out 27q", "family": "readout", "n": 27, "shots": 4096, "dtype": "c64"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    f = rng.choice(["u3cz64", "u3cz128", "grid64", "gridbf", "grid128", "mult", "gates", "grad", "gradb", "batch",
                    "energy", "readout"])
    if f == "u3cz64":
        return {"family": "u3cz", "n": rng.randint(13, 22), "layers": rng.randint(8, 40), "dtype": "c64"}
    if f == "u3cz128":
        return {"family": "u3cz", "n": rng.randint(8, 16), "layers": rng.randint(8, 24), "dtype": "c128"}
    if f == "grid64":
        return {"family": "grid", "n": rng.randint(20, 28), "cycles": rng.randint(6, 20), "dtype": "c64",
                "prec": "plain"}
    if f == "gridbf":
        return {"family": "grid", "n": rng.randint(21, 30), "cycles": rng.randint(6, 20), "dtype": "c64",
                "prec": "bf16x3"}
    if f == "grid128":
        return {"family": "grid", "n": rng.randint(17, 24), "cycles": rng.randint(6, 20), "dtype": "c128",
                "prec": "plain"}
    if f == "mult":
        return {"family": "mult", "nbits": rng.randint(4, 7), "spread": rng.randint(2, 4)}
    if f == "gates":
        return {"family": "gates", "n": rng.randint(12, 28), "dtype": rng.choice(["c64", "c64", "c128"])}
    if f == "grad":
        return {"family": "grad", "n": rng.randint(8, 21), "layers": rng.randint(2, 10), "sets": 1}
    if f == "gradb":
        return {"family": "grad", "n": rng.randint(12, 20), "layers": rng.randint(2, 10), "sets": _log_int(rng, 4, 64)}
    if f == "batch":
        return {"family": "batch", "count": _log_int(rng, 4, 48), "nmin": rng.randint(8, 12),
                "nmax": rng.randint(16, 22), "depth": rng.randint(8, 40)}
    if f == "energy":
        return {"family": "energy", "n": rng.randint(16, 29), "dtype": rng.choice(["c64", "c64", "c128"])}
    return {"family": "readout", "n": rng.randint(16, 28), "shots": _log_int(rng, 100, 100000),
            "dtype": rng.choice(["c64", "c64", "c128"])}


# ---- circuits (seeded descriptions; (name, targets, controls, angles)) -----
def _u3cz(n, layers, rng):
    ops = []
    for _ in range(layers):
        for q in range(n):
            ops.append(("U3", (q,), (), tuple(rng.uniform(0, 2 * PI) for _ in range(3))))
        p = list(range(n))
        rng.shuffle(p)
        for i in range(n // 2):
            ops.append(("CZ", (p[2 * i], p[2 * i + 1]), (), ()))
    return ops


def _grid(n, cycles, rng):
    """A 5 x 6 lattice narrowed to n qubits: sqrt(X), sqrt(Y) or sqrt(W) on
    every qubit, never the previous one again, then fSim(pi/2, pi/6) on one
    of the four coupler sets; gates on removed qubits are left out."""
    rows, cols = 5, 6
    gone = set(rng.sample(range(rows * cols), rows * cols - n))
    at = {q: i for i, q in enumerate(q for q in range(rows * cols) if q not in gone)}
    sets = {"A": [], "B": [], "C": [], "D": []}
    for r in range(rows):
        for c in range(cols):
            q = r * cols + c
            if c + 1 < cols:
                sets["A" if c % 2 == 0 else "B"].append((q, q + 1))
            if r + 1 < rows:
                sets["C" if r % 2 == 0 else "D"].append((q, q + cols))
    prev = {}
    ops = []
    for cyc in range(cycles):
        for q in range(rows * cols):
            prev[q] = rng.choice([g for g in ("SX", "SY", "SW") if g != prev.get(q)])
            if q in at:
                ops.append((prev[q], (at[q],), (), ()))
        for a, b in sets["ABCDCDAB"[cyc % 8]]:
            if a in at and b in at:
                ops.append(("FSIM", (at[a], at[b]), (), (PI / 2, PI / 6)))
    return ops


def _multiplier(nbits, spread, rng):
    """p <- a * b by shift-and-add of controlled ripple-carry adders, on
    superposed inputs: H on every bit of a and all but `spread` bits of b
    (those are set at random)."""
    a, b = list(range(nbits)), list(range(nbits, 2 * nbits))
    p, carry = list(range(2 * nbits, 4 * nbits)), 4 * nbits
    fixed = set(rng.sample(b, min(spread, nbits)))
    ops = []
    for q in a + b:
        if q not in fixed:
            ops.append(("H", (q,), (), ()))
        elif rng.random() < 0.5:
            ops.append(("X", (q,), (), ()))
    for i in range(nbits):
        y, z, chain = p[i:i + nbits], p[i + nbits], [carry] + a[:-1]

        def cx(ctl, t):
            return ("X", (t,), (b[i],) + ctl, ())
        for j in range(nbits):
            ops += [cx((a[j],), y[j]), cx((a[j],), chain[j]), cx((chain[j], y[j]), a[j])]
        ops.append(cx((a[-1],), z))
        for j in reversed(range(nbits)):
            ops += [cx((chain[j], y[j]), a[j]), cx((a[j],), chain[j]), cx((chain[j],), y[j])]
    return ops


def _hea(n, layers):
    """RY and RZ on every qubit, each angle a parameter, then a CNOT ladder."""
    ops = []
    for k in range(layers):
        for q in range(n):
            ops.append(("RY", (q,), (), ((k * n + q) * 2,)))
            ops.append(("RZ", (q,), (), ((k * n + q) * 2 + 1,)))
        for q in range(n - 1):
            ops.append(("X", (q + 1,), (q,), ()))
    return ops


def _gate_calls(n, rng):
    """One-call-per-gate work: a U3 on every third qubit, CNOT and CZ between
    random qubits, a Toffoli and dense 2- and 3-qubit unitaries."""
    u3 = [("U3", (q,), (), tuple(rng.uniform(0, 2 * PI) for _ in range(3))) for q in range(rng.randrange(3), n, 3)]
    q = rng.sample(range(n), 8)
    return u3 + [("X", (q[0],), (q[1],), ()), ("PHASE", (q[2],), (q[3],), (PI,)), ("X", (q[4],), (q[5], q[6]), ()),
                 ("U3", (q[7],), (), (0.3, 0.1, rng.uniform(0, 2 * PI))),
                 ("MATRIX", tuple(q[0:2]), (), (rng.randrange(1 << 30),)),
                 ("MATRIX", tuple(q[2:5]), (), (rng.randrange(1 << 30),))]


def _unitary(k, seed):
    g = np.random.default_rng(seed)
    z = g.standard_normal((1 << k, 1 << k)) + 1j * g.standard_normal((1 << k, 1 << k))
    u, r = np.linalg.qr(z)
    return u * (np.diag(r) / np.abs(np.diag(r)))[None, :]


def _matrix(name, ang):
    """The gate's matrix in complex128 (bit j of an index is target j)."""
    if name == "MATRIX":
        return None
    s = 1 / math.sqrt(2)
    if name == "H":
        return np.array([[s, s], [s, -s]], dtype=complex)
    if name == "X":
        return np.array([[0, 1], [1, 0]], dtype=complex)
    if name in ("SX", "SY", "SW"):
        x, y = np.array([[0, 1], [1, 0]], dtype=complex), np.array([[0, -1j], [1j, 0]])
        p = {"SX": x, "SY": y, "SW": (x + y) * s}[name]
        return (1 + 1j) / 2 * (np.eye(2) - 1j * p)
    if name == "U3":
        t, f, l = ang
        c, d = math.cos(t / 2), math.sin(t / 2)
        return np.array([[c, -np.exp(1j * l) * d], [np.exp(1j * f) * d, np.exp(1j * (f + l)) * c]])
    if name == "PHASE":
        return np.diag([1, np.exp(1j * ang[0])])
    if name == "CZ":
        return np.diag([1, 1, 1, -1]).astype(complex)
    assert name == "FSIM"
    c, d = math.cos(ang[0]), math.sin(ang[0])
    m = np.diag([1, c, c, np.exp(-1j * ang[1])]).astype(complex)
    m[1, 2] = m[2, 1] = -1j * d
    return m


def _ising(n, h=0.5):
    return [(0, 3 << i, 1.0) for i in range(n - 1)] + [(1 << i, 0, h) for i in range(n)]


def _ops_of(case, seed):
    rng = random.Random(seed)
    f = case["family"]
    if f == "u3cz":
        return case["n"], _u3cz(case["n"], case["layers"], rng)
    if f == "grid":
        return case["n"], _grid(case["n"], case["cycles"], rng)
    if f == "mult":
        return 4 * case["nbits"] + 1, _multiplier(case["nbits"], case.get("spread", 2), rng)
    assert f == "gates"
    return case["n"], _gate_calls(case["n"], rng)


def _batch_ops(case, seed):
    rng = random.Random(seed)
    widths = random.Random(case["count"] * 1000 + case["nmax"])   # the same widths for every seed
    return [(n, _u3cz(n, case["depth"], rng))
            for n in (widths.randint(case["nmin"], case["nmax"]) for _ in range(case["count"]))]


def _circuit(n, ops, n_params=0):
    c = B.Circuit(n)
    par = [c.parameter() for _ in range(n_params)]
    for name, t, ctl, ang in ops:
        c.append(name, t, [par[ang[0]]] if n_params and ang else ang, ctl)
    return sim.marshal(c)


def _dense_state(n, dtype, seed):
    s = sim.StateVector(n, dtype)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    s.amps.normal_(generator=g)
    tilt = np.random.default_rng(seed).uniform(0.2, PI / 2 - 0.2, n)
    for lo in range(0, n, 8):   # the qubits' weights, eight at a time
        w = torch.ones(1, dtype=s.amps.dtype, device="cuda")
        for t in tilt[lo:lo + 8]:
            w = torch.outer(torch.tensor([math.cos(t), math.sin(t)], dtype=w.dtype, device="cuda"), w).view(-1)
        s.amps.view(-1, w.numel(), 2 << lo).mul_(w.view(1, -1, 1))
    s.amps.mul_(1.0 / math.sqrt(2.0))
    return s


# ---- a user's state and one pass -------------------------------------------
def prepare(case, seed):
    f = case["family"]
    if f in ("u3cz", "grid", "mult"):
        n, ops = _ops_of(case, seed)
        prec = {"plain": N.SV_PREC_PLAIN, "bf16x3": N.SV_PREC_TC_BF16X3}[case.get("prec", "plain")]
        opts = sim.options(prec=prec) if "prec" in case else None
        return {"f": "circuit", "s": sim.StateVector(n, case.get("dtype", "c64")), "c": _circuit(n, ops), "o": opts}
    if f == "gates":
        n, ops = _ops_of(case, seed)
        calls = [(_unitary(len(t), a[0]) if m == "MATRIX" else _matrix(m, a), t, c) for m, t, c, a in ops]
        return {"f": f, "s": _dense_state(n, case["dtype"], seed), "calls": calls}
    if f == "grad":
        n, sets = case["n"], case["sets"]
        np_ = 2 * n * case["layers"]
        return {"f": f, "psi": [sim.StateVector(n, "c64") for _ in range(sets)],
                "lam": [sim.StateVector(n, "c64") for _ in range(sets)],
                "c": _circuit(n, _hea(n, case["layers"]), np_), "terms": _ising(n),
                "p": torch.from_numpy(_params(case, seed)), "o": sim.options(mode=N.SV_MODE_TILED_GRAPH)}
    if f == "batch":
        cs = _batch_ops(case, seed)
        ss = [sim.StateVector(n, "c64") for n, _ in cs]
        ms = [_circuit(n, ops) for n, ops in cs]
        return {"f": f, "s": ss, "m": ms, "h": (C.c_void_p * len(ss))(*[s.h.value for s in ss]),
                "cs": (C.POINTER(N.SvCircuit) * len(ms))(*[C.pointer(m.c) for m in ms]),
                "o": sim.options(mode=N.SV_MODE_TILED_GRAPH)}
    s = _dense_state(case["n"], case["dtype"], seed)
    return {"f": f, "s": s, "terms": _ising(case["n"]), "shots": case.get("shots", 0), "seed": seed}


def _params(case, seed):
    # small angles: the near-identity start that keeps a deep ansatz trainable
    p = np.random.default_rng(seed).uniform(-0.3, 0.3, size=(case["sets"], 2 * case["n"] * case["layers"]))
    return p.astype(np.float32)


def run(st):
    f = st["f"]
    if f == "circuit":
        return st["s"].set_basis(0).apply_circuit(st["c"], opts=st["o"]).amps
    if f == "gates":
        for u, t, c in st["calls"]:
            st["s"].apply_gate(u, t, c)
        return st["s"].amps
    if f == "grad":
        if len(st["psi"]) == 1:
            th = st["p"][0].detach().requires_grad_(True)
            e = sim.SvExpectation.apply(th, st["psi"][0], st["lam"][0], st["c"], st["terms"], 0)
            e.backward()
            return {"energy": e.detach(), "grad": th.grad}
        for s in st["psi"]:
            s.set_basis(0)
        e, g = sim.adjoint_grad_batch(st["psi"], st["lam"], st["c"], st["p"].numpy(), st["terms"], st["o"])
        return {"energy": torch.from_numpy(e).float(), "grad": torch.from_numpy(g).float()}
    if f == "batch":
        for s in st["s"]:
            s.set_basis(0)
        N.check(N.lib().sv_apply_circuit_batch(st["h"], len(st["s"]), st["cs"], None, C.byref(st["o"])))
        return [s.amps for s in st["s"]]
    if f == "energy":
        return st["s"].expect(st["terms"])
    return {"z": st["s"].z_all(), "norm": st["s"].norm2(), "shots": st["s"].sample(st["shots"], st["seed"])}


# ---- the work that cannot be left out --------------------------------------
def _flops(n, ops):
    """Gate by gate: 14 flops for an amplitude that a 2 x 2 matrix makes, 6
    for a phase, none for one that only moves; 8 * 2^k - 2 for a dense
    k-qubit matrix; an amplitude that no control lets through costs nothing."""
    tot = 0.0
    for name, t, ctl, ang in ops:
        per = {"CZ": 0.0, "X": 0.0, "PHASE": 3.0, "FSIM": 1.5, "RZ": 6.0}.get(name, 14.0)
        if name == "MATRIX":
            per = 8.0 * (1 << len(t)) - 2
        tot += per * 2.0 ** (n - len(ctl))
    return tot


def work(case):
    f = case["family"]
    amp = 16 if case.get("dtype") == "c128" else 8
    if f == "grad":
        n = case["n"]
        # the forward sweep on one vector, the backward one on two, and a
        # probe (8 flops an amplitude) for each parameter
        fl = 3 * _flops(n, _hea(n, case["layers"])) + 8.0 * 2 ** n * 2 * n * case["layers"]
        return {"bytes": case["sets"] * (amp * 2 ** n + 32.0 * n * case["layers"]), "flops": case["sets"] * fl}
    if f == "batch":
        cs = _batch_ops(case, 0)
        return {"bytes": sum(amp * 2 ** n for n, _ in cs), "flops": sum(_flops(n, o) for n, o in cs)}
    if f in ("energy", "readout"):
        n = case["n"]
        return {"bytes": amp * 2.0 ** n, "flops": 2.0 ** n * (6 * n if f == "energy" else 3 + n)}
    n, ops = _ops_of(case, 0)
    return {"bytes": (2 if f == "gates" else 1) * amp * 2.0 ** n, "flops": _flops(n, ops)}


# ---- the same in 64 bits ----------------------------------------------------
def _axes(psi, n, qs):
    """psi (..., 2^n) seen with the axes of the qubits `qs` (bit order) first."""
    lead = psi.dim() - 1
    v = psi.view(*psi.shape[:-1], *([2] * n))
    return v, [lead + n - 1 - q for q in qs]


def _apply(psi, n, u, t, ctl=()):
    """In-place: u (2^k x 2^k, or a batch of 2 x 2 matrices over psi's rows)
    on targets t where every control is 1."""
    v, ax = _axes(psi, n, tuple(ctl) + tuple(t))
    for i, c in enumerate(ctl):
        v = v.select(ax[i], 1)
        ax = [a - 1 if a > ax[i] else a for a in ax]
    ax = ax[len(ctl):]
    k = len(t)
    part = []
    for y in range(1 << k):
        w = v
        for j in sorted(range(k), key=lambda j: -ax[j]):
            w = w.select(ax[j], (y >> j) & 1)
        part.append(w)
    if torch.is_tensor(u):
        m = [[u[:, r, c].view(-1, *([1] * (part[0].dim() - 1))) for c in range(2)] for r in range(2)]
        zero = [[False] * 2] * 2
    else:
        m = [[complex(x) for x in row] for row in u]
        zero = [[x == 0 for x in row] for row in m]
    new = []
    for r in range(1 << k):
        if not torch.is_tensor(u) and m[r][r] == 1 and sum(zero[r]) == (1 << k) - 1:
            new.append(None)
            continue
        acc = None
        for c in range(1 << k):
            if not zero[r][c]:
                x = part[c] * m[r][c]
                acc = x if acc is None else acc.add_(x)
        new.append(acc)
    for p, x in zip(part, new):
        if x is not None:
            p.copy_(x)


def _zero_state(n, rows=None):
    psi = torch.zeros((1 << n,) if rows is None else (rows, 1 << n), dtype=torch.complex128, device="cuda")
    psi[..., 0] = 1
    return psi


def _run64(n, ops, psi=None):
    psi = _zero_state(n) if psi is None else psi
    for name, t, ctl, ang in ops:
        _apply(psi, n, _unitary(len(t), ang[0]) if name == "MATRIX" else _matrix(name, ang), t, ctl)
    return torch.view_as_real(psi).reshape(-1)


def _rot(name, th):
    """RY or RZ matrices of a vector of angles (rows x 2 x 2)."""
    th = torch.as_tensor(th, dtype=torch.float64, device="cuda") / 2
    c, s = torch.cos(th).to(torch.complex128), torch.sin(th).to(torch.complex128)
    if name == "RY":
        return torch.stack([torch.stack([c, -s], -1), torch.stack([s, c], -1)], -2)
    z = torch.zeros_like(c)
    return torch.stack([torch.stack([c - 1j * s, z], -1), torch.stack([z, c + 1j * s], -1)], -2)


def _grad64(case, seed):
    n, sets = case["n"], case["sets"]
    p = _params(case, seed).astype(np.float64)
    ops = _hea(n, case["layers"])
    psi = _zero_state(n, sets)
    x = _matrix("X", ())
    for name, t, ctl, ang in ops:
        _apply(psi, n, x if name == "X" else _rot(name, p[:, ang[0]]), t, ctl)
    lam = torch.zeros_like(psi)
    idx = torch.arange(1 << n, device="cuda")
    diag = torch.zeros(1 << n, dtype=torch.float64, device="cuda")
    for xm, zm, cf in _ising(n):
        if xm == 0:
            i = zm.bit_length() - 2
            diag += cf * (1 - 2 * (((idx >> i) ^ (idx >> (i + 1))) & 1)).to(torch.float64)
    lam += psi * diag
    for xm, zm, cf in _ising(n):
        if xm:
            lam += cf * psi[:, idx ^ xm]
    del idx
    e = torch.sum(lam.conj() * psi, -1).real
    grad = torch.zeros(sets, p.shape[1], dtype=torch.float64, device="cuda")
    for name, t, ctl, ang in reversed(ops):
        if name == "X":
            _apply(psi, n, x, t, ctl)
            _apply(lam, n, x, t, ctl)
            continue
        v = psi.view(sets, -1, 2, 1 << t[0])
        w = lam.view(sets, -1, 2, 1 << t[0])
        a0, a1, b0, b1 = v[:, :, 0], v[:, :, 1], w[:, :, 0], w[:, :, 1]
        if name == "RY":
            g = torch.sum((b1.conj() * a0 - b0.conj() * a1).real, (1, 2))
        else:
            g = torch.sum((b0.conj() * a0 - b1.conj() * a1).imag, (1, 2))
        grad[:, ang[0]] = g
        r = _rot(name, -p[:, ang[0]])
        _apply(psi, n, r, t)
        _apply(lam, n, r, t)
    if sets == 1:
        return {"energy": e[0], "grad": grad[0]}
    return {"energy": e, "grad": grad}


def exact(case, seed):
    f = case["family"]
    if f in ("u3cz", "grid", "mult", "gates"):
        n, ops = _ops_of(case, seed)
        if n > 28 or len(ops) * 2.0 ** n > 800 * 2.0 ** 27:   # over 20 seconds
            return None
        psi = None
        if f == "gates":
            a = _dense_state(n, case["dtype"], seed).amps.double()
            psi = torch.view_as_complex(a.view(-1, 2)).clone()
        return _run64(n, ops, psi)
    if f == "grad":
        return _grad64(case, seed)
    if f == "batch":
        return [_run64(n, ops) for n, ops in _batch_ops(case, seed)]
    n = case["n"]
    a = _dense_state(n, case["dtype"], seed).amps
    if f == "energy":
        c = a.view(-1, 2)
        pr = sum(_prob64(c[:, k]) for k in range(2))
        tot = 0.0
        for i in range(n - 1):
            v = pr.view(-1, 2, 2, 1 << i)
            tot += float((v[:, 0, 0].sum() + v[:, 1, 1].sum() - v[:, 0, 1].sum() - v[:, 1, 0].sum()))
        del pr
        for i in range(n):
            v = c.view(-1, 2, 1 << i, 2)
            s = sum(float(torch.sum(p.double() * q.double())) for p, q in
                    ((v[j::8, 0], v[j::8, 1]) for j in range(8)))
            tot += 0.5 * 2 * s
        return tot
    pr = sum(_prob64(a.view(-1, 2)[:, k]) for k in range(2))
    tot = float(pr.sum())
    z = np.array([float(tot - 2 * pr.view(-1, 2, 1 << q)[:, 1].sum()) for q in range(n)])
    return {"z": z, "norm": tot, "shots": None}


def _prob64(x):
    return x.double().square_()
