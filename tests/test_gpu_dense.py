"""Dense gates of 2..6 qubits on CUDA cores, alone and grouped into passes, against the
oracle: every k with targets on the lowest, highest and mixed qubits, controls inside
and outside a tile, conditions, states smaller than a tile, runs longer than a pass
holds.  complex64: 1e-6 per element of a normalised state after the run (a few rounding
errors of 2^-24 per 64-term product); complex128: 1e-13."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu
TOL = {"c64": 1e-6, "c128": 1e-13}


def haar(r, d):
    q, t = np.linalg.qr(r.standard_normal((d, d)) + 1j * r.standard_normal((d, d)))
    return q * (np.diag(t) / np.abs(np.diag(t)))


def run(n, prec, mode, gates, cbits=()):
    from paper_1908_07187_gb300 import qk

    psi = workloads.random_state(n, 40 + n)
    with qk.Context(prec, mode, tensor_cores=False) as ctx:
        ctx.add_qubits(n)
        if cbits:
            ctx.add_cbits(len(cbits))
            ctx.write_cbits(0, cbits)
        ctx.set_state(psi)
        for u, t, c, cond in gates:
            if u is None:
                ctx.apply_gate("u3", t, c, cond, (0.3, 1.2, -0.7))
            else:
                ctx.apply_gate(ctx.define_gate_matrix(u), t, c, cond)
        got = ctx.get_state()
    ref = oracle.OracleState(n, psi=psi)
    for u, t, c, cond in gates:
        if all(cbits[k] for k in cond):
            ref.apply_matrix(oracle.u3(0.3, 1.2, -0.7) if u is None else u, t, c)
    assert np.max(np.abs(got - ref.psi)) <= TOL[prec], (n, prec, mode)


@pytest.mark.parametrize("prec", ["c64", "c128"])
@pytest.mark.parametrize("k", [2, 3, 4, 5, 6])
@pytest.mark.parametrize("n", [6, 8, 9, 10, 13, 16])
def test_one_gate(n, k, prec):
    r = np.random.Generator(np.random.PCG64([n, k]))
    for targets in (list(range(k)), list(range(n - k, n))[::-1], [int(q) for q in r.permutation(n)[:k]]):
        free = [q for q in range(n) if q not in targets]
        for nc in {0, min(1, len(free)), min(3, len(free))}:
            ctl = [int(q) for q in r.permutation(free)[:nc]] if nc else []
            run(n, prec, "plain", [(haar(r, 1 << k), targets, ctl, ())])


@pytest.mark.parametrize("prec", ["c64", "c128"])
@pytest.mark.parametrize("n", [7, 12, 15, 18])
def test_runs_of_gates(n, prec):
    r = np.random.Generator(np.random.PCG64([n, 9]))
    gates = []
    for j in range(70):
        k = int(r.integers(2, 7)) if j % 3 else 2
        qs = [int(q) for q in r.permutation(n)[:min(n, k + int(r.integers(3)))]]
        cond = (int(r.integers(6)),) if r.random() < 0.3 else ()
        gates.append((haar(r, 1 << k), qs[:k], qs[k:], cond))
        if j % 10 == 9:
            gates.append((None, qs[:1], qs[1:2], ()))
    run(n, prec, "fused", gates, [1, 0, 1, 1, 1, 0])


@pytest.mark.parametrize("n", [13, 20, 23])
def test_brickwork_of_pairs(n):
    r = np.random.Generator(np.random.PCG64([n, 10]))
    gates = [(haar(r, 4), (q, q + 1), (), ()) for layer in range(4) for q in range(layer % 2, n - 1, 2)]
    run(n, "c64", "fused", gates)
