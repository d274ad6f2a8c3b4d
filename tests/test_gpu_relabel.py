"""The qubit-relabelling gather (tiles of up to ten bits): every amplitude moves to
its place bit for bit, below, at and above the tile width, in both precisions."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["c64", "c128"])
@pytest.mark.parametrize("n", [1, 2, 4, 5, 6, 8, 9, 10, 11, 14, 17])
def test_swaps_move_every_amplitude(n, prec):
    from paper_1908_07187_gb300 import qk

    rng = np.random.Generator(np.random.PCG64([n, 77]))
    orders = [rng.permutation(n) for _ in range(3)] + [np.arange(n)[::-1]]
    psi = (rng.standard_normal(1 << n) + 1j * rng.standard_normal(1 << n)).astype(
        np.complex64 if prec == "c64" else np.complex128)
    i = np.arange(1 << n)
    with qk.Context(prec) as ctx:
        ctx.add_qubits(n)
        for order in orders:
            ctx.set_state(psi)
            at = list(range(n))               # at[q]: where the amplitude bit of qubit q came from
            for q in range(n):                # selection sort into `order` by SWAPs
                p = at.index(int(order[q]))
                if p != q:
                    ctx.apply_gate("swap", (q, p))
                    at[q], at[p] = at[p], at[q]
            src = np.zeros_like(i)
            for q in range(n):
                src |= ((i >> q) & 1) << at[q]
            assert np.array_equal(ctx.get_state(), psi[src])
