"""The tiled modular-exponentiation gather against controlled multiplications worked
out index by index: a permutation, so bit-exact, at the edges of its rule (register
on the lowest, middle and highest qubits, in both orders, from one qubit to the
widest that is tiled and one beyond)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def expected(psi, n, reg, ctrls, mults, N):
    i = np.arange(1 << n, dtype=np.int64)
    y = np.zeros_like(i)
    for q in reg:
        y = (y << 1) | ((i >> q) & 1)
    m = np.full_like(i, 1 % N)
    for q, v in zip(ctrls, mults):
        m = np.where((i >> q) & 1, m * pow(v, -1, N) % N, m)
    x = np.where(y < N, m * y % N, y)
    src = i.copy()
    for a, q in enumerate(reg):
        src = (src & ~(1 << q)) | (((x >> (len(reg) - 1 - a)) & 1) << q)
    return psi[src]


@pytest.mark.parametrize("prec", ["c64", "c128"])
@pytest.mark.parametrize("n,p0,w", [(3, 0, 2), (6, 5, 1), (9, 0, 4), (10, 3, 4), (11, 7, 4), (14, 0, 9), (14, 5, 9),
                                    (15, 1, 11), (15, 3, 12), (16, 2, 13), (16, 1, 14), (16, 0, 14), (17, 13, 3),
                                    (17, 9, 8)])
@pytest.mark.parametrize("first_is_low", [False, True])
def test_tiled_gather_bit_exact(n, p0, w, first_is_low, prec):
    from paper_1908_07187_gb300 import qk

    rng = np.random.Generator(np.random.PCG64([n, p0, w]))
    N = max(2, (1 << w) - int(rng.integers(1 << max(0, w - 2))))
    units = [v for v in range(1, N) if np.gcd(v, N) == 1]
    reg = list(range(p0, p0 + w))
    reg = reg if first_is_low else reg[::-1]
    ctrls = [int(q) for q in rng.permutation([q for q in range(n) if q not in reg])]
    mults = [int(units[int(rng.integers(len(units)))]) for _ in ctrls]
    psi = (rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)).astype(
        np.complex64 if prec == "c64" else np.complex128)
    with qk.Context(prec) as ctx:
        ctx.add_qubits(n)
        ctx.set_state(psi)
        ctx.apply_modexp(reg, ctrls, mults, N)
        assert np.array_equal(ctx.get_state(), expected(psi, n, reg, ctrls, mults, N))
