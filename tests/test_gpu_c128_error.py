"""Rounding error of fused complex128 circuits.  A fused gate rounds an amplitude at most four
times (two FMAs of a turn, two of an update), as the 2x2 product of the plain path does, and
what stays pending on the host is kept in twice the precision; so over circuits of a few hundred
gates the fused error against extended precision is within 1.5 of the plain one."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def layers(n, gates, r):
    out, layer = [], 0
    while len(out) < gates:
        if layer % 3 == 0:
            for q in range(n):
                c, s = np.cos(r.uniform(0, np.pi)), 0.0
                s = np.sqrt(1 - c * c)
                a, b = np.exp(1j * r.uniform(0, 2 * np.pi, 2))
                out.append((np.array([[c, -b * s], [a * s, a * b * c]]), q, None))
        else:
            out += [(np.diag([1.0, -1.0 if r.random() < 0.5 else np.exp(1j * r.uniform(0, 6))]), q + 1, q)
                    for q in range(layer % 3 - 1, n - 1, 2)]
        layer += 1
    return out


def exact(n, ops):
    psi = np.zeros(1 << n, dtype=np.clongdouble)
    psi[0] = 1
    i = np.arange(1 << n)
    for m, q, ctl in ops:
        lo = i[((i >> q) & 1 == 0) & ((i >> ctl) & 1 == 1 if ctl is not None else True)]
        a, b = psi[lo].copy(), psi[lo | 1 << q].copy()
        m = m.astype(np.clongdouble)
        psi[lo], psi[lo | 1 << q] = m[0, 0] * a + m[0, 1] * b, m[1, 0] * a + m[1, 1] * b
    return psi


@pytest.mark.parametrize("n", [5, 9, 12])
def test_error_is_that_of_plain_gates(n):
    from paper_1908_07187_gb300 import qk

    err = {"fused": 0.0, "plain": 0.0}
    for seed in range(8):
        ops = layers(n, 290, np.random.Generator(np.random.PCG64([n, seed])))
        ref = exact(n, ops)
        for mode in err:
            with qk.Context("c128", mode) as ctx:
                ctx.add_qubits(n)
                for m, q, ctl in ops:
                    ctx.apply_gate(ctx.define_gate_matrix(m), (q,), () if ctl is None else (ctl,))
                d = ctx.get_state().astype(np.clongdouble) - ref
            err[mode] += float(np.sqrt(np.sum(d.real ** 2 + d.imag ** 2))) / 8
    assert err["fused"] <= 1.5 * err["plain"], err
