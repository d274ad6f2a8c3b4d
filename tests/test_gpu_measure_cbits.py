"""Several measured qubits copied into one cbit: the last of the list stays, within a round
of eight and across rounds."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["c64", "c128"])
@pytest.mark.parametrize("nq", [2, 3, 8, 9, 12])
def test_last_outcome_stays(nq, prec):
    from paper_1908_07187_gb300 import qk

    r = np.random.Generator(np.random.PCG64(nq))
    with qk.Context(prec) as ctx:
        ctx.add_qubits(nq)
        ctx.add_cbits(3)
        for trial in range(40):
            dest = [int(x) for x in r.integers(0, 3, nq)]
            bits = [int(x) for x in r.integers(0, 2, nq)]
            ctx.reset()
            ctx.write_cbits(0, [1, 0, 1])
            for q in range(nq):
                if bits[q]:
                    ctx.apply_gate("x", (q,))
            ctx.measure(list(range(nq)), [0.5] * nq, dest, wait=False)
            want = [1, 0, 1]
            for q in range(nq):
                want[dest[q]] = bits[q]
            assert list(ctx.read_cbits()) == want
