"""A Kitaev stage whose two branches nearly cancel: with the identity as the permutation and a
phase close to half a turn the kept amplitudes are 1 + e^{i theta} times the old ones.  Each is
formed by FMAs onto the old amplitude, so it is off by two units of the working precision (the
sum and the scaling) and not by units of the amplitudes that cancel.  What all of them share, a
factor from the rounded phase and the norm, is divided out: the norm comes from 2^13 terms whose
errors of 2^-24 / |1 + e^{i theta}| average out below one unit.  4 units in all."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [14, 18, 20, 23])
@pytest.mark.parametrize("bits", [8, 9, 10])
def test_kept_branch_keeps_its_digits(n, bits):
    from paper_1908_07187_gb300 import qk

    r = np.random.Generator(np.random.PCG64([n, bits]))
    half = (np.exp(1j * r.uniform(0, 2 * np.pi, 1 << (n - 1))) * 2.0 ** (-(n - 1) / 2)).astype(np.complex64)
    psi = np.zeros(1 << n, dtype=np.complex64)
    psi[::2] = half
    with qk.Context("c64") as ctx:
        ctx.add_qubits(n)
        ctx.add_cbits(bits + 1)
        ctx.write_cbits(0, [1] * bits)              # theta = -pi (1 - 2^-bits)
        ctx.set_state(psi)
        ident = ctx.define_gate_perm_table(list(range(16)))
        ctx.apply_kitaev_stage(0, ident, (4, 3, 2, 1), tuple(range(bits)), 0.0, bits)
        got = ctx.get_state()
        assert ctx.read_cbits()[bits] == 0
    assert not np.any(got[1::2])
    ratio = got[::2].astype(np.complex128) / half.astype(np.complex128)
    assert np.max(np.abs(ratio / ratio.mean() - 1)) <= 4 * 2.0 ** -24
