"""Measuring many qubits in rounds: outcomes, cbits and the collapsed state against
a plain qubit-by-qubit computation in FP64, for lists that end at, below and above a
round, on the lowest qubits (told apart by lane), the highest and mixed, from states
smaller than a row up."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def reference(psi, qubits, us):
    psi = psi.astype(np.complex128)
    i = np.arange(len(psi))
    out, margin = [], 1.0
    for q, u in zip(qubits, us):
        p = np.abs(psi) ** 2
        bit = ((i >> q) & 1) == 1
        s0, s1 = p[~bit].sum(), p[bit].sum()
        m = int(u >= s0 / (s0 + s1))
        margin = min(margin, abs(u - s0 / (s0 + s1)))
        out.append(m)
        psi = np.where(bit == (m == 1), psi, 0) / np.sqrt(s1 if m else s0)
    return out, psi, margin


@pytest.mark.parametrize("prec", ["c64", "c128"])
@pytest.mark.parametrize("n,qubits", [
    (1, [0]), (2, [1, 0]), (4, [3, 0, 2, 1]), (5, [4]), (6, [0, 1, 2, 3, 4, 5]), (7, [6, 2, 0]),
    (9, list(range(9))), (10, list(range(10))[::-1]), (12, list(range(4, 12))), (13, [12, 0, 11, 1, 10, 2, 9, 3, 8]),
    (14, [13]), (14, [5]), (16, list(range(16))), (17, list(range(9, 17)) + [0, 7]), (18, [4, 5, 6, 17])])
def test_rounds_match_one_by_one(n, qubits, prec):
    from paper_1908_07187_gb300 import qk

    rng = np.random.Generator(np.random.PCG64([n, len(qubits), qubits[0]]))
    psi = rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)
    psi /= np.linalg.norm(psi)
    psi = psi.astype(np.complex64 if prec == "c64" else np.complex128)
    with qk.Context(prec) as ctx:
        ctx.add_qubits(n)
        ctx.add_cbits(len(qubits))
        for trial in range(3):
            us = [float(x) for x in rng.uniform(size=len(qubits))]
            bits, want, margin = reference(psi, qubits, us)
            if margin < 1e-6:           # a uniform on the edge of P0 decides nothing
                continue
            ctx.set_state(psi)
            got = ctx.measure(qubits, us, list(range(len(qubits))))
            assert got == int("".join(map(str, bits)), 2)
            assert list(ctx.read_cbits()) == bits
            # 1 / sqrt(P) from compensated sums: a few units of the working precision
            assert np.max(np.abs(ctx.get_state() - want)) <= (4e-7 if prec == "c64" else 1e-14)
