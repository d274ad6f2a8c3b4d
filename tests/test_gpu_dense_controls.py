"""Dense gates with several controls, alone and in runs, against the oracle: many controls
leave few tiles (the tile is cut for what is enumerated), and a run of such gates goes in a
pass each where that moves less of the state, which the launches count shows."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu
TOL = {"c64": 1e-6, "c128": 1e-13}     # as for any run of dense gates


def haar(r, d):
    q, t = np.linalg.qr(r.standard_normal((d, d)) + 1j * r.standard_normal((d, d)))
    return q * (np.diag(t) / np.abs(np.diag(t)))


@pytest.mark.parametrize("prec", ["c64", "c128"])
@pytest.mark.parametrize("n,k,nc,count", [
    (8, 2, 6, 3), (12, 6, 6, 2), (16, 2, 14, 4), (16, 3, 4, 5), (18, 4, 4, 1), (18, 5, 2, 3), (19, 2, 16, 2),
    (20, 2, 4, 8), (20, 4, 4, 4), (20, 6, 3, 2), (21, 2, 1, 6), (21, 3, 2, 6)])
def test_runs_of_controlled_gates(n, k, nc, count, prec):
    from paper_1908_07187_gb300 import qk

    r = np.random.Generator(np.random.PCG64([n, k, nc]))
    psi = workloads.random_state(n, 30 + n)
    ref = oracle.OracleState(n, psi=psi)
    with qk.Context(prec, tensor_cores=False) as ctx:
        ctx.add_qubits(n)
        ctx.add_cbits(6)
        ctx.write_cbits(0, [1, 0, 1, 1, 1, 0])
        ctx.set_state(psi)
        for j in range(count):
            qs = [int(q) for q in r.permutation(n)[:k + max(0, nc - j % 2)]]
            u = haar(r, 1 << k)
            cond = (j,) if j < 6 and j % 3 == 1 else ()
            ctx.apply_gate(ctx.define_gate_matrix(u), qs[:k], qs[k:], cond)
            if not cond or [1, 0, 1, 1, 1, 0][j]:
                ref.apply_matrix(u, qs[:k], qs[k:])
        got = ctx.get_state()
    assert np.max(np.abs(got - ref.psi)) <= TOL[prec]


@pytest.mark.parametrize("nc,launches", [(4, 6), (0, 1)])
def test_passes_over_what_the_controls_leave(nc, launches):
    from paper_1908_07187_gb300 import qk

    n, r = 24, np.random.Generator(np.random.PCG64(nc))
    with qk.Context("c64") as ctx:
        ctx.add_qubits(n)
        gates = [ctx.define_gate_matrix(haar(r, 4)) for _ in range(6)]
        ctx.reset_counters()
        for j, g in enumerate(gates):
            ctx.apply_gate(g, (j, j + 1), tuple(range(12, 12 + nc)))
        ctx.flush()
        assert ctx.counters()["launches"] == launches
