"""Queues of a few ops on states that run in shared-memory tiles: ops that concern a small part
of a large state move only that part, longer queues go in passes, and the results are those of
one pass per gate on either side of the line."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu
TOL = {"c64": 1e-6, "c128": 1e-14}
FEW = [
    [("z", (9,), (1,))],
    [("t", (9,), ())],
    [("x", (9,), (1, 11))],
    [("h", (9,), (1, 2, 10, 11, 8))],
    [("z", (9,), (1,)), ("z", (3,), (2,))],
]
MORE = [
    [("h", (9,), ())],
    [("x", (9,), (1,)), ("x", (3,), (2,))],
    [("z", (9,), (1,))] * 3,
    [("x", (q,), (q + 1, (q + 5) % 12)) for q in range(6)],
    [("h", (q,), ()) for q in range(12)],
]


@pytest.mark.parametrize("prec,n", [("c64", 12), ("c128", 12), ("c128", 17), ("c128", 20), ("c128", 22)])
@pytest.mark.parametrize("gates", FEW + MORE)
@pytest.mark.parametrize("cond", [(), (0,), (1,)])
def test_same_state_as_gate_by_gate(n, prec, gates, cond):
    from paper_1908_07187_gb300 import qk

    psi = workloads.random_state(n, 90 + n)
    got = []
    for mode in ("fused", "plain"):
        with qk.Context(prec, mode) as ctx:
            ctx.add_qubits(n)
            ctx.add_cbits(2)
            ctx.write_cbits(0, [1, 0])
            ctx.set_state(psi)
            for g, t, c in gates:
                ctx.apply_gate(g, t, c, cond)
            got.append(ctx.get_state())
    assert np.max(np.abs(got[0] - got[1])) <= TOL[prec]


@pytest.mark.parametrize("gates,eighths", list(zip(FEW, [2, 4, 2, 0.25, 4])))
@pytest.mark.parametrize("n", [22, 24])
def test_small_parts_of_large_states(n, gates, eighths):
    """eighths: the most of the state that the queue may move."""
    from paper_1908_07187_gb300 import qk

    with qk.Context("c128") as ctx:
        ctx.add_qubits(n)
        ctx.reset_counters()
        for g, t, c in gates:
            ctx.apply_gate(g, t, c)
        ctx.flush()
        assert ctx.counters()["algorithmic_bytes"] <= 2 * 16 * 2 ** n * eighths / 8
