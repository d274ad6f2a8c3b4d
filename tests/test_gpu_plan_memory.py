"""The planner's host storage: what a thread keeps between plans does not grow with the longest
queue it has seen."""
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def resident():
    with open("/proc/self/statm") as f:
        return int(f.read().split()[1]) * os.sysconf("SC_PAGE_SIZE")


def test_a_long_queue_leaves_nothing_behind():
    from paper_1908_07187_gb300 import qk

    n, count = 13, 60000
    r = np.random.Generator(np.random.PCG64(1))
    ops = np.zeros(count, dtype=qk.GATE_OP_DTYPE)
    ops["gate_id"], ops["nc"], ops["np"] = qk.GATE["u3"], 1, 3
    ops["target"] = r.integers(0, n, count)
    ops["controls"][:, 0] = (ops["target"] + r.integers(1, n, count)) % n
    ops["params"] = r.uniform(0, 6, (count, 3))

    def run(gates, pending):
        with qk.Context("c64", max_pending=pending) as ctx:
            ctx.add_qubits(n)
            ctx.apply_gates(gates)
            ctx.sync()

    run(ops[:4000], 0)
    before = resident()
    run(ops, 1 << 20)                                # each gate becomes up to four: 44 MB of ops
    assert resident() - before < 24 << 20
