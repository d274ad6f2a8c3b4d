"""One-qubit matrices that a wide unitarity tolerance lets in, among ordinary gates: the
fused passes (both tile kinds, and the widths' edges) take them as they are, as one pass per
gate does.  Bounds: a unit of the working precision per gate (40 gates), relative to the
largest amplitude."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu
SIZES = [("c128", 3), ("c128", 9), ("c128", 13), ("c64", 2), ("c64", 9), ("c64", 12), ("c64", 13), ("c64", 15)]
TOL = {"c64": 40 * 2.0 ** -24, "c128": 40 * 2.0 ** -53}


def both_modes(n, prec, ops):
    """ops: (matrix, target, controls) in order; fused against plain."""
    from paper_1908_07187_gb300 import qk

    psi = workloads.random_state(n, 70 + n)
    got = []
    for mode in ("fused", "plain"):
        with qk.Context(prec, mode) as ctx:
            ctx.add_qubits(n)
            ctx.set_state(psi)
            for m, q, ctl in ops:
                ctx.apply_gate(ctx.define_gate_matrix(m, tol=1e9), (q,), ctl)
            got.append(ctx.get_state())
    assert np.all(np.isfinite(got[0]))
    assert np.max(np.abs(got[0] - got[1])) <= TOL[prec] * np.max(np.abs(got[1]))


def among_gates(n, seed, special, often=3, most=40):
    """40 gates, every third on average special(r), some controlled, with diagonal terms
    between neighbours that wait over the gates."""
    r = np.random.Generator(np.random.PCG64([n, seed]))
    ops, used = [], 0
    for _ in range(40):
        q, d = (int(x) for x in r.permutation(n)[:2])
        m, _ = np.linalg.qr(r.standard_normal((2, 2)) + 1j * r.standard_normal((2, 2)))
        if used < most and r.integers(often) == 0:
            m = special(r)
            used += 1
        ops.append((m, q, (d,) if r.random() < 0.3 else ()))
        if r.random() < 0.5:
            ops.append((np.diag([1, -1 if r.random() < 0.5 else np.exp(1j * r.uniform(0, 6))]), d, (q,)))
    return ops


@pytest.mark.parametrize("prec,n", SIZES)
@pytest.mark.parametrize("lower", [False, True])
def test_triangular(n, prec, lower):
    def special(r):
        m = np.diag(np.exp(1j * r.uniform(0, 6, 2)))
        m[(1, 0) if lower else (0, 1)] = 0.3 * (r.standard_normal() + 1j * r.standard_normal())
        return m
    both_modes(n, prec, among_gates(n, 1 + lower, special))


@pytest.mark.parametrize("prec,n", SIZES)
def test_diagonal_of_any_magnitude(n, prec):
    def special(r):
        return np.diag(r.uniform(0.3, 1.8, 2) * np.exp(1j * r.uniform(0, 6, 2)))
    both_modes(n, prec, among_gates(n, 3, special))


SINGULAR = {
    "diagonal": lambda r: np.diag([1.0, 0.0] if r.random() < 0.5 else [0.0, 1.0]),
    "projector": lambda r: np.outer(v := r.standard_normal(2) + 1j * r.standard_normal(2), v.conj()) / np.vdot(v, v),
    "column": lambda r: np.linalg.qr(r.standard_normal((2, 2)))[0] * ([1, 0] if r.random() < 0.5 else [0, 1]),
    "nilpotent": lambda r: np.array([[0, 1], [0, 0]] if r.random() < 0.5 else [[0, 0], [1, 0]]),
    "rows": lambda r: np.linalg.qr(r.standard_normal((2, 2)))[0] * [[1], [2.0 ** -30]],
}


@pytest.mark.parametrize("prec,n", SIZES)
@pytest.mark.parametrize("kind", list(SINGULAR))
def test_singular_and_far_from_unitary(n, prec, kind):
    """Three of them among the gates, or the state would soon be empty."""
    both_modes(n, prec, among_gates(n, 4, SINGULAR[kind], often=6, most=3))


@pytest.mark.parametrize("prec,n", [s for s in SIZES if s[0] == "c128" or s[1] == 2])   # 2^(63 n) fits the type
def test_magnitudes_that_pile_up(n, prec):
    """Each qubit scaled by 2^-9 on one value many times, turned by gates between, and back."""
    ops, h = [], np.array([[1, 1], [1, -1]]) / np.sqrt(2)
    for q in range(n):
        ops += [(np.diag([1, 2.0 ** -9]), q, ())] * 6
        ops += [(h, q, ()), (np.diag([1, 2.0 ** -9]), q, ()), (h, q, ())]
    for q in range(n):
        ops += [(np.diag([1, 2.0 ** 9]), q, ())] * 7
    both_modes(n, prec, ops)


@pytest.mark.parametrize("n", [13, 15])
def test_small_matrices_that_are_multiplied(n):
    """Gates on one qubit that become one before the passes, each scaled by 2^-27."""
    h = 2.0 ** -27 * np.array([[1, 1], [1j, -1j]]) / np.sqrt(2)
    ops = [(h, 3, ()), (h, 3, ()), (np.array([[0.6, 0.8], [0.8, -0.6]]), 4, (3,)), (h, 3, ())]
    both_modes(n, "c64", ops)


def test_direction_between_the_entries():
    """Register tiles turn a gate by one angle; a matrix whose off-diagonal entries ask for
    angles 9e-8 apart gets the one between, so either entry is off by half of that.  The mean
    over 400 gates, rounding (2^-25 each) averaged down to 2e-9."""
    from paper_1908_07187_gb300 import qk

    n, d, off = 13, 9e-8, []
    r = np.random.Generator(np.random.PCG64(8))
    with qk.Context("c64") as ctx:
        ctx.add_qubits(n)
        for _ in range(400):
            c = np.cos(r.uniform(0.1, 0.7))          # the larger entries on the diagonal
            a, b = np.exp(1j * r.uniform(0, 6, 2))
            s = np.sqrt(1 - c * c)
            m = np.array([[c, -b * s], [a * s * np.exp(1j * d), a * b * c]])
            ctx.reset()
            ctx.apply_gate(ctx.define_gate_matrix(m, tol=1e-6), (6,))
            off.append(np.imag(ctx.get_state()[1 << 6] / m[1, 0]))
    assert abs(np.mean(off)) <= d / 2 + 4e-9


@pytest.mark.parametrize("prec,n", SIZES)
@pytest.mark.parametrize("noise", [1e-3, 1e-7, "float32"])
def test_nearly_unitary(n, prec, noise):
    def special(r):
        u = np.linalg.qr(r.standard_normal((2, 2)) + 1j * r.standard_normal((2, 2)))[0]
        if noise == "float32":
            return u.astype(np.complex64).astype(np.complex128)
        return u + noise * (r.standard_normal((2, 2)) + 1j * r.standard_normal((2, 2)))
    both_modes(n, prec, among_gates(n, 5, special))
