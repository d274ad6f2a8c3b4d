"""The work that is timed: circuits as a program that uses the library runs them,
through the public entry points of ``paper_1908_07187_gb300.qk``.

A case is a dict of plain values; its ``kind`` says which entry points carry it:

* ``circuit``  one context, a gate list in bulk (``apply_gates``), SWAPs, a
  measurement, and the state viewed (on the host for small states, as a device
  tensor for large ones): the layered and QFT circuits of the configurations;
* ``dense``    user-defined dense matrix gates on arbitrary qubits;
* ``request``  one serving request: layers, a controlled modular multiplication and
  mid-circuit measurements, each followed by a gate conditioned on its bit;
* ``kitaev``   order finding with one recycled control qubit (fused stages);
* ``shor``     order finding with a control register (modular exponentiation);
* ``batch``    many small independent circuits in one batch, all states read back.

Every circuit is laid out here as a list of plain tuples from numpy's PCG64, keyed
by the seed; ``prepare`` turns it into the arrays that a program keeps, ``exact``
computes it in complex128 with torch alone.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1908_07187_gb300 import qk


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def _circuit(n, prec, style, gates, qft, measure, view):
    return {"kind": "circuit", "n": n, "prec": prec, "style": style, "gates": gates, "qft": qft, "measure": measure,
            "view": view}


def listed():
    return [
        # the smallest call: a 10-qubit circuit worked on interactively (run, look at the state, measure)
        {"name": "small_10q", **_circuit(10, "c64", "layered", 120, True, 10, "host")},
        # the 12-qubit complex128 configuration: H on all, 200 gates of U3 / CNOT-chain layers, QFT, measure all
        {"name": "plain_12q_c128", **_circuit(12, "c128", "cnot", 200, True, 12, "host")},
        # a mid-size state that fits L2: layers and QFT, the state handed on as a device tensor
        {"name": "layered_21q", **_circuit(21, "c64", "layered", 500, True, 0, "device")},
        # the headline configuration: 30 qubits, 500 layer gates, QFT, a measurement
        {"name": "layered_30q", **_circuit(30, "c64", "layered", 500, True, 8, "device")},
        # the same kind of circuit in complex128, as one checks a complex64 result
        {"name": "layered_23q_c128", **_circuit(23, "c128", "layered", 300, True, 3, "device")},
        # random two-qubit unitaries in a brickwork (as in quantum-volume circuits), given as matrices
        {"name": "pairs_22q", "kind": "dense", "n": 22, "prec": "c64", "k_min": 2, "k_max": 2, "controls": 0,
         "count": 63},
        # larger blocks given as matrices, on qubits anywhere, some of them controlled
        {"name": "blocks_24q", "kind": "dense", "n": 24, "prec": "c64", "k_min": 3, "k_max": 6, "controls": 1,
         "count": 12},
        # one serving request with a large state: mid-circuit measurements and conditioned gates
        {"name": "request_26q", "kind": "request", "n": 26, "layers": 23, "w": 13, "measures": 3},
        # order finding for a 20-bit N with one recycled control qubit (21 qubits, 40 stages)
        {"name": "kitaev_20b", "kind": "kitaev", "b": 20},
        # order finding with a control register for a 9-bit N (27 qubits)
        {"name": "shor_9b", "kind": "shor", "b": 9},
        # the small requests of a serving loop, collected into one batch (8..13 qubits)
        {"name": "batch_requests", "kind": "batch", "of": "requests", "count": 256, "n_min": 8, "n_max": 13,
         "d_min": 5, "d_max": 40},
        # many layer circuits of 10..20 qubits and 50..300 layers
        {"name": "batch_layers", "kind": "batch", "of": "layers", "count": 60, "n_min": 10, "n_max": 20,
         "d_min": 50, "d_max": 300},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["circuit", "circuit", "circuit", "dense", "dense", "request", "kitaev", "shor", "batch"])
    if kind == "circuit":
        prec = rng.choice(["c64", "c64", "c128"])
        n = rng.randint(4, 28 if prec == "c64" else 23)
        return _circuit(n, prec, rng.choice(["layered", "cnot", "mixed"]),
                        _log_int(rng, 30, 500 if prec == "c64" or n < 20 else 250), rng.random() < 0.7,
                        rng.randint(0, n), "host" if n <= 14 else "device")
    if kind == "dense":
        k_max = rng.randint(1, 6)
        prec = rng.choice(["c64", "c64", "c128"])
        return {"kind": "dense", "n": rng.randint(7, 24 if prec == "c64" else 20), "prec": prec,
                "k_min": rng.randint(1, k_max), "k_max": k_max, "controls": rng.randint(0, 1),
                "count": rng.randint(4, 24)}
    if kind == "request":
        return {"kind": "request", "n": _log_int(rng, 8, 26), "layers": rng.randint(5, 40), "w": rng.randint(10, 16),
                "measures": rng.randint(1, 4)}
    if kind == "kitaev":
        return {"kind": "kitaev", "b": rng.randint(12, 20)}
    if kind == "shor":
        return {"kind": "shor", "b": rng.randint(4, 9)}
    if rng.random() < 0.5:
        lo = rng.randint(4, 12)
        return {"kind": "batch", "of": "requests", "count": _log_int(rng, 2, 400), "n_min": lo,
                "n_max": rng.randint(lo, 13), "d_min": 5, "d_max": rng.randint(10, 40)}
    lo = rng.randint(8, 18)
    return {"kind": "batch", "of": "layers", "count": _log_int(rng, 2, 60), "n_min": lo, "n_max": rng.randint(lo, 20),
            "d_min": 10, "d_max": rng.randint(20, 200)}


# ---------------------------------------------------------------------------
# circuits as lists of tuples
#   ("g", gate, target, controls, cond, params)    built-in 1-target gate
#   ("swap", a, b)
#   ("mat", u, targets, controls)                  dense matrix, first target = MSB
#   ("mul", targets, controls, c, N)               x -> c x mod N, first target = MSB
#   ("modexp", targets, controls, multipliers, N)
#   ("measure", qubits, uniforms, cbits)
#   ("stage", control, targets, c, N, phase_cbits, uniform, cbit)
# ---------------------------------------------------------------------------

# Two generators lay out a circuit: `s`, keyed by the case alone, the gates' kinds
# and places and the sizes; `r`, keyed by the seed, every angle, matrix, modulus and
# uniform.

def _rng(seed, *more):
    return np.random.Generator(np.random.PCG64([int(seed) & 0xFFFFFFFF, *[int(x) for x in more]]))


def _u3(r, q, cond=()):
    return ("g", "u3", q, (), cond, tuple(float(x) for x in r.uniform(0.0, 2.0 * math.pi, 3)))


def _cz(a, b):
    return ("g", "z", b, (a,), (), ())


def _qft(qubits):
    """H, then controlled phases pi / 2^(i+1), qubit by qubit; SWAPs end for end."""
    ops, q = [], list(qubits)
    for c in range(len(q)):
        ops.append(("g", "h", q[c], (), (), ()))
        ops += [("g", "p", q[c], (q[d],), (), (math.pi / float(1 << (i + 1)),))
                for i, d in enumerate(range(c + 1, len(q)))]
    return ops + [("swap", q[i], q[-1 - i]) for i in range(len(q) // 2)]


def _gates(s, r, n, style, count):
    """Exactly `count` gates of a style's repeating layers."""
    ops, layer = [], 0
    while len(ops) < count:
        if style == "layered":      # U3 on all / CZ on even pairs / CZ on odd pairs
            new = [_u3(r, q) for q in range(n)] if layer % 3 == 0 else [_cz(q, q + 1)
                                                                        for q in range(layer % 3 - 1, n - 1, 2)]
        elif style == "cnot":       # U3 on all / CNOT chain
            new = [_u3(r, q) for q in range(n)] if layer % 2 == 0 else [("g", "x", q + 1, (q,), (), ())
                                                                        for q in range(n - 1)]
        else:                       # built-in gates at random, up to two controls
            new = []
            for _ in range(n):
                gate = ("x", "y", "z", "h", "s", "sdg", "t", "tdg", "u3", "p", "rz")[int(s.integers(11))]
                qs = [int(x) for x in s.permutation(n)[:1 + min(n - 1, (0, 0, 1, 1, 2)[int(s.integers(5))])]]
                par = tuple(float(x) for x in r.uniform(0.0, 2.0 * math.pi, {"u3": 3, "p": 1, "rz": 1}.get(gate, 0)))
                new.append(("g", gate, qs[0], tuple(qs[1:]), (), par))
        ops += new
        layer += 1
    return ops[:count]


def _unitary(r, d):
    z = r.standard_normal((d, d)) + 1j * r.standard_normal((d, d))
    q, t = np.linalg.qr(z)
    return q * (np.diag(t) / np.abs(np.diag(t)))


def _odd_composite(r, b):
    """A seeded odd b-bit composite that is no prime power, and a base coprime to it."""
    while True:
        N = (1 << (b - 1)) | int(r.integers(1 << (b - 1))) | 1
        if len(_prime_factors(N)) < 2:
            continue
        while True:
            a = 2 + int(r.integers(N - 3))
            if math.gcd(a, N) == 1:
                return N, a


def _prime_factors(m):
    out, p = set(), 2
    while p * p <= m:
        while m % p == 0:
            out.add(p)
            m //= p
        p += 1
    return out | ({m} if m > 1 else set())


def _request(s, r, n, layers, w, measures):
    """Layers cycling U3-all / CZ-even / CZ-odd, one controlled multiplication on a
    w-qubit register where it fits, `measures` measurements with a conditioned U3."""
    at = int(s.integers(layers)) if n >= w + 1 else -1
    when = sorted(int(s.integers(layers)) for _ in range(measures))
    ops, k = [], 0
    for layer in range(layers):
        ops += [_u3(r, q) for q in range(n)] if layer % 3 == 0 else [_cz(q, q + 1)
                                                                     for q in range(layer % 3 - 1, n - 1, 2)]
        if layer == at:
            N, a = _odd_composite(r, w)
            ops.append(("mul", tuple(range(1, w + 1)), (0,), pow(a, 1 << int(r.integers(2 * w)), N), N))
        while k < measures and when[k] == layer:
            q = int(s.integers(n))
            t = (q + 1 + int(s.integers(n - 1))) % n
            ops.append(("measure", (q,), (float(r.uniform()),), (k,)))
            ops.append(_u3(r, t, (k,)))
            k += 1
    return ops


def _layers(r, n, depth):
    """U3 on every qubit, then CZ on the even or odd neighbour pairs, `depth` times."""
    ang = r.uniform(0.0, 2.0 * math.pi, (depth, n, 3))
    ops = []
    for L in range(depth):
        ops += [("g", "u3", q, (), (), tuple(float(x) for x in ang[L, q])) for q in range(n)]
        ops += [_cz(q, q + 1) for q in range(L % 2, n - 1, 2)]
    return ops


def _build(case, seed):
    """(n_qubits, n_cbits, ops) of a one-context case."""
    kind = case["kind"]
    if kind == "circuit":
        n, m = case["n"], case["measure"]
        s, r = _rng(1, n, case["gates"]), _rng(seed, 1, n, case["gates"])
        ops = [("g", "h", q, (), (), ()) for q in range(n)] if case["style"] == "cnot" else []
        ops += _gates(s, r, n, case["style"], case["gates"])
        if case["qft"]:
            ops += _qft(range(n))
        if m:
            ops.append(("measure", tuple(range(m)), tuple(float(x) for x in r.uniform(size=m)), tuple(range(m))))
        return n, m, ops
    if kind == "dense":
        n = case["n"]
        s, r = _rng(2, n, case["count"], case["k_max"]), _rng(seed, 2, n, case["count"])
        ops = [_u3(r, q) for q in range(n)]
        for j in range(case["count"]):
            k = int(s.integers(case["k_min"], case["k_max"] + 1))
            nc = min(n - k, int(s.integers(case["controls"] + 1)) if j % 2 else 0)
            if case["k_min"] == case["k_max"] == 2:    # a brickwork of neighbours
                p = (2 * j + (2 * j // (n - 1)) % 2) % (n - 1)
                qs = [p, p + 1]
            else:
                qs = [int(x) for x in s.permutation(n)[:k + nc]]
            ops.append(("mat", _unitary(r, 1 << k), tuple(qs[:k]), tuple(qs[k:])))
        return n, 0, ops
    if kind == "request":
        n, m = case["n"], case["measures"]
        return n, m, _request(_rng(3, n, case["layers"]), _rng(seed, 3, n), n, case["layers"], case["w"], m)
    if kind == "kitaev":
        b = case["b"]
        r = _rng(seed, 4, b)
        N, a = _odd_composite(r, b)
        reg = tuple(range(1, b + 1))
        ops = [("g", "x", b, (), (), ())]
        for e in range(2 * b):
            ops.append(("stage", 0, reg, pow(a, 1 << (2 * b - 1 - e), N), N, tuple(range(e - 1, -1, -1)),
                        float(r.uniform()), e))
        return b + 1, 2 * b, ops
    if kind == "shor":
        b = case["b"]
        r = _rng(seed, 5, b)
        N, a = _odd_composite(r, b)
        t = (N * N - 1).bit_length()
        ctl, reg = tuple(range(t)), tuple(range(t, t + b))
        ops = [("g", "x", t + b - 1, (), (), ())] + [("g", "h", q, (), (), ()) for q in ctl]
        ops.append(("modexp", reg, tuple(t - 1 - c for c in range(t)), tuple(pow(a, 1 << c, N) for c in range(t)), N))
        ops.append(("measure", reg, tuple(float(x) for x in r.uniform(size=b)), tuple(range(b))))
        return t + b, b, ops + _qft(ctl)
    raise ValueError(kind)


def _build_batch(case, seed):
    out = []
    for i in range(case["count"]):
        s, r = _rng(6, i), _rng(seed, 6, i)
        n = int(s.integers(case["n_min"], case["n_max"] + 1))
        depth = int(s.integers(case["d_min"], case["d_max"] + 1))
        if case["of"] == "layers":
            out.append((n, 0, _layers(r, n, depth)))
        else:
            m = 1 + int(s.integers(4))
            out.append((n, m, _request(s, r, n, depth, 6 + int(s.integers(6)), m)))
    return out


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------

def _gate_array(ops):
    out = np.zeros(len(ops), dtype=qk.GATE_OP_DTYPE)
    for e, (_, gate, target, controls, cond, params) in zip(out, ops):
        e["gate_id"], e["target"] = qk.GATE[gate], target
        e["nc"], e["ncc"], e["np"] = len(controls), len(cond), len(params)
        e["controls"][:len(controls)] = controls
        e["cond"][:len(cond)] = cond
        e["params"][:len(params)] = params
    return out


def _runs(ops):
    """The ops with every stretch of built-in gates as one gate array."""
    out, run = [], []
    for op in ops:
        if op[0] == "g":
            run.append(op)
            continue
        if run:
            out.append(("gates", _gate_array(run)))
            run = []
        out.append(op)
    return out + ([("gates", _gate_array(run))] if run else [])


def prepare(case, seed):
    if case["kind"] == "batch":
        return {"kind": "batch", "batch": qk.Batch(), "layers": case["of"] == "layers",
                "circuits": [(n, m, _runs(ops)) for n, m, ops in _build_batch(case, seed)]}
    n, m, ops = _build(case, seed)
    ctx = qk.Context(case.get("prec", "c64"))
    ctx.add_qubits(n)
    if m:
        ctx.add_cbits(m)
    calls = []
    for op in _runs(ops):
        if op[0] == "mat":
            op = ("gate", ctx.define_gate_matrix(op[1]), op[2], op[3])
        elif op[0] == "mul":
            op = ("gate", ctx.define_gate_perm_mulmod(len(op[1]), op[3], op[4]), op[1], op[2])
        elif op[0] == "stage":
            op = ("stage", op[1], ctx.define_gate_perm_mulmod(len(op[2]), op[3], op[4]), *op[2:3], *op[5:])
        calls.append(op)
    return {"kind": case["kind"], "ctx": ctx, "calls": calls, "bits": m, "host": case.get("view") == "host"}


def _run_batch(state):
    b = state["batch"]
    b.clear()
    for n, m, calls in state["circuits"]:
        b.add_circuit(n, m)
        for op in calls:
            if op[0] == "gates":
                b.apply_gates(op[1])
            elif op[0] == "mul":
                b.apply_mulmod(op[1], op[2], op[3], op[4])
            else:
                b.measure(op[1], op[2], op[3])
    b.run(store_states=True)
    if state["layers"]:
        return [b.read(i)[1] for i in range(len(state["circuits"]))]
    return {"bits": b.read_all_cbits(), "states": np.concatenate([b.read(i)[1] for i in range(len(state["circuits"]))])}


def run(state):
    if state["kind"] == "batch":
        return _run_batch(state)
    ctx, seen = state["ctx"], None
    ctx.reset()
    for op in state["calls"]:
        kind = op[0]
        if kind == "gates":
            ctx.apply_gates(op[1])
        elif kind == "swap":
            ctx.apply_gate("swap", op[1:])
        elif kind == "gate":
            ctx.apply_gate(op[1], op[2], op[3])
        elif kind == "stage":
            ctx.apply_kitaev_stage(op[1], op[2], op[3], op[4], op[5], op[6])
        elif kind == "modexp":
            ctx.apply_modexp(op[1], op[2], op[3], op[4])
        elif state["host"]:        # look at the state, then measure
            seen = ctx.get_state()
            ctx.measure(op[1], op[2], op[3], wait=False)
        else:
            ctx.measure(op[1], op[2], op[3], wait=False)
    if state["host"] and seen is None:
        seen = ctx.get_state()
    if not state["host"]:
        seen = ctx.torch_view()
        seen.owner = ctx           # the view reads the context's memory: keep it as long as the view
    out = {"state": seen}
    if state["bits"]:
        out["bits"] = ctx.read_cbits()
    return out


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

_DIAGONAL = ("z", "s", "sdg", "t", "tdg", "p", "rz")


def _op_flops(n, op):
    """Arithmetic of one op on 2^n amplitudes: 16 per amplitude pair for a 2x2 gate,
    6 per amplitude multiplied by a phase, 8 * 2^k per amplitude of a dense block."""
    amps = float(1 << n)
    if op[0] == "g":
        part = amps / (1 << len(op[3]))
        if op[1] in _DIAGONAL:
            return 0.0 if op[1] == "z" else 6.0 * part * (1.0 if op[1] == "rz" else 0.5)
        return 0.0 if op[1] in ("x", "y") else 8.0 * part
    if op[0] == "mat":
        return 8.0 * len(op[1]) * amps / (1 << len(op[3]))
    if op[0] == "measure":
        return 4.0 * amps
    if op[0] == "stage":
        return 15.0 * amps
    return 0.0


def work(case):
    if case["kind"] == "batch":
        circuits = _build_batch(case, 0)
        return {"bytes": float(sum(8 << n for n, _, _ in circuits) + sum(80 * len(ops) for _, _, ops in circuits)),
                "flops": float(sum(_op_flops(n, op) for n, _, ops in circuits for op in ops))}
    n, _, ops = _build(case, 0)
    amp = 16 if case.get("prec") == "c128" else 8
    # the state starts as |0...0>, so it is written once at the least; a measurement
    # reads it once more, and so does a permutation or a stage (which needs the
    # amplitudes of other elements before any can be written)
    passes = 1 + sum(2 for op in ops if op[0] in ("mul", "modexp", "stage")) + sum(1 for op in ops if op[0] == "measure")
    return {"bytes": float(passes * (amp << n)), "flops": float(sum(_op_flops(n, op) for op in ops))}


# ---------------------------------------------------------------------------
# the same in complex128, with torch alone
# ---------------------------------------------------------------------------

def _at(psi, n, bits):
    """The amplitudes whose qubits have the given values, as a view of psi."""
    shape, index, top = [], [], n
    for q in sorted(bits, reverse=True):
        shape += [1 << (top - q - 1), 2]
        index += [slice(None), bits[q]]
        top = q
    return psi.view(shape + [1 << top])[tuple(index)]


def _matrix2(gate, p):
    e = lambda x: complex(math.cos(x), math.sin(x))  # noqa: E731
    h = math.sqrt(0.5)
    if gate == "u3":
        c, s = math.cos(p[0] / 2), math.sin(p[0] / 2)
        return c, -e(p[2]) * s, e(p[1]) * s, e(p[1] + p[2]) * c
    return {"x": (0, 1, 1, 0), "y": (0, -1j, 1j, 0), "z": (1, 0, 0, -1), "h": (h, h, h, -h), "s": (1, 0, 0, 1j),
            "sdg": (1, 0, 0, -1j), "t": (1, 0, 0, e(math.pi / 4)), "tdg": (1, 0, 0, e(-math.pi / 4)),
            "p": (1, 0, 0, e(p[0]) if p else 1), "rz": (e(-p[0] / 2) if p else 1, 0, 0, e(p[0] / 2) if p else 1)}[gate]


def _apply2(psi, n, m, q, controls):
    fixed = {c: 1 for c in controls}
    if m[1] == 0 and m[2] == 0:
        for v, f in ((0, m[0]), (1, m[3])):
            if f != 1:
                _at(psi, n, {**fixed, q: v}).mul_(f)
        return
    a, b = _at(psi, n, {**fixed, q: 0}), _at(psi, n, {**fixed, q: 1})
    y = m[2] * a
    y += m[3] * b
    a.mul_(m[0]).add_(b, alpha=m[1])
    b.copy_(y)


def _apply_matrix(psi, n, u, targets, controls):
    k = len(targets)
    free = [q for q in range(n - 1, -1, -1) if q not in targets and q not in controls]
    dims = [n - 1 - q for q in list(controls) + list(targets) + free]
    v = psi.view([2] * n).permute(dims)[(1,) * len(controls)]
    w = torch.as_tensor(u, dtype=psi.dtype, device=psi.device) @ v.reshape(1 << k, -1)
    v.copy_(w.view(v.shape))


def _register(n, targets, device):
    """Every index's register value (first target = MSB)."""
    i = torch.arange(1 << n, device=device)
    y = torch.zeros_like(i)
    for q in targets:
        y = (y << 1) | ((i >> q) & 1)
    return y


def _permuted(psi, n, targets, y, x):
    """psi gathered from where the register value y (of every index) is replaced by x."""
    src, d = torch.arange(1 << n, device=psi.device), y ^ x
    for j, q in enumerate(targets):
        src ^= ((d >> (len(targets) - 1 - j)) & 1) << q
    return psi[src]


def _mulmod(psi, n, targets, controls, c, N):
    y = _register(n, targets, psi.device)
    x = torch.where(y < N, (y * pow(c, -1, N)) % N, y)
    i = torch.arange(1 << n, device=psi.device)
    for q in controls:
        x = torch.where(((i >> q) & 1) == 1, x, y)
    return _permuted(psi, n, targets, y, x)


def _measure(psi, n, q, u):
    s0, s1 = (float(torch.view_as_real(_at(psi, n, {q: v})).square().sum()) for v in (0, 1))
    m = int(u >= s0 / (s0 + s1))
    _at(psi, n, {q: 1 - m}).zero_()
    psi.mul_(1.0 / math.sqrt(s1 if m else s0))
    return m


def _simulate(n, n_bits, ops, stop_at_measure=False):
    """(state before the final measurement if asked for, state, bits)."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    psi = torch.zeros(1 << n, dtype=torch.complex128, device=dev)
    psi[0] = 1.0
    bits, seen = [0] * n_bits, None
    for op in ops:
        kind = op[0]
        if kind == "g":
            if all(bits[c] for c in op[4]):
                _apply2(psi, n, _matrix2(op[1], op[5]), op[2], op[3])
        elif kind == "swap":
            a, b = _at(psi, n, {op[1]: 0, op[2]: 1}), _at(psi, n, {op[1]: 1, op[2]: 0})
            t = a.clone()
            a.copy_(b)
            b.copy_(t)
        elif kind == "mat":
            _apply_matrix(psi, n, op[1], op[2], op[3])
        elif kind == "mul":
            psi = _mulmod(psi, n, *op[1:])
        elif kind == "modexp":
            _, reg, ctl, mult, N = op
            i = torch.arange(1 << n, device=dev)
            m = torch.ones_like(i)
            for q, c in zip(ctl, mult):
                m = torch.where(((i >> q) & 1) == 1, m * pow(c, -1, N) % N, m)
            y = _register(n, reg, dev)
            psi = _permuted(psi, n, reg, y, torch.where(y < N, m * y % N, y))
        elif kind == "stage":
            _, ctl, reg, c, N, phase, u, dest = op
            _apply2(psi, n, _matrix2("h", ()), ctl, ())
            psi = _mulmod(psi, n, reg, (ctl,), c, N)
            theta = -2.0 * math.pi * sum(bits[b] / 2.0 ** (j + 2) for j, b in enumerate(phase))
            _apply2(psi, n, _matrix2("p", (theta,)), ctl, ())
            _apply2(psi, n, _matrix2("h", ()), ctl, ())
            bits[dest] = _measure(psi, n, ctl, u)
            if bits[dest]:
                _apply2(psi, n, _matrix2("x", ()), ctl, ())
        else:
            if stop_at_measure:
                seen = psi.clone()
            for q, u, d in zip(*op[1:]):
                bits[d] = _measure(psi, n, q, u)
    return (psi if seen is None else seen), psi, bits


EXACT_QUBITS = 27   # above: too long in 64 bits


def exact(case, seed):
    if case["kind"] == "batch":
        states, bits = [], []
        for n, m, ops in _build_batch(case, seed):
            _, psi, b = _simulate(n, m, ops)
            states.append(psi.cpu().numpy())
            bits += b
        return states if case["of"] == "layers" else {"bits": None, "states": np.concatenate(states)}
    n, m, ops = _build(case, seed)
    if n > EXACT_QUBITS:
        return None
    seen, psi, _ = _simulate(n, m, ops, case.get("view") == "host")
    out = {"state": seen if case.get("view") == "host" else psi}
    return {**out, "bits": None} if m else out
