"""What a batch hands out after a run is that run's circuits, also when circuits are added
after it: the run's circuits read as before, in any order and with both totals grown far
beyond the run's, and an added one is refused until it has run."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def circuit(n, seed, ncb=0):
    r = np.random.Generator(np.random.PCG64([n, seed]))
    ops = [workloads.Op("u3", (q,), params=tuple(float(x) for x in r.uniform(0, 6.28, 3))) for q in range(n)]
    ops += [workloads.Op("z", (q + 1,), controls=(q,)) for q in range(n - 1)]
    if ncb:
        ops.append(workloads.Op("measure", tuple(range(ncb)), uniforms=tuple(float(x) for x in r.uniform(size=ncb)),
                                cbits=tuple(range(ncb))))
    return n, ncb, ops


def alone(qk, circ):
    b = qk.Batch()
    b.add_ops(*circ)
    b.run()
    bits, psi = b.read(0)
    b.close()
    return list(bits), psi


@pytest.mark.parametrize("before", [0, 1, 2, 3])
def test_circuits_added_after_a_run(before):
    """before: how many of the run's circuits are read before more are added."""
    from paper_1908_07187_gb300 import qk

    first = [circuit(4, 1, 2), circuit(6, 2), circuit(3, 3, 1), circuit(14, 4)]
    added = [circuit(13, 5, 4), circuit(13, 6, 4), circuit(15, 7)]
    want = [alone(qk, c) for c in first]
    b = qk.Batch()
    for c in first:
        b.add_ops(*c)
    with pytest.raises(qk.QKError) as e:             # nothing has run
        b.read(0)
    assert e.value.status == qk.QK_ESTATE
    b.run()
    for i in range(before):
        assert np.array_equal(b.read(i)[1], want[i][1])
    for c in added:
        b.add_ops(*c)
    for i in [0, 4, 1, 6, 2, 5, 3, 0, 1]:
        if i < len(first):
            bits, psi = b.read(i)
            assert list(bits) == want[i][0] and np.array_equal(psi, want[i][1]), i
            continue
        with pytest.raises(qk.QKError) as e:
            b.read(i)
        assert e.value.status == qk.QK_ESTATE
    with pytest.raises(qk.QKError) as e:             # its cbits include the added circuits'
        b.read_all_cbits()
    assert e.value.status == qk.QK_ESTATE
    b.run()
    for i, c in enumerate(first + added):
        bits, psi = b.read(i)
        ref = alone(qk, c)
        assert list(bits) == ref[0] and np.array_equal(psi, ref[1]), i
    assert list(b.read_all_cbits()) == sum((alone(qk, c)[0] for c in first + added), [])
    b.clear()
    b.add_ops(*first[0])
    with pytest.raises(qk.QKError) as e:
        b.read(0)
    assert e.value.status == qk.QK_ESTATE
    b.close()


def test_large_circuits_have_cbits_of_0():
    from paper_1908_07187_gb300 import qk

    b = qk.Batch()
    for _ in range(8):                               # cbits of 1 in the buffer
        b.add_ops(4, 4, [workloads.Op("x", (q,)) for q in range(4)] + [
            workloads.Op("measure", (0, 1, 2, 3), uniforms=(0.5,) * 4, cbits=(0, 1, 2, 3))])
    b.run()
    assert list(b.read_all_cbits()) == [1] * 32
    b.clear()
    for i in range(8):
        b.add_ops(14 if i % 2 else 3, 4, [workloads.Op("x", (0,))])
    b.run()
    assert list(b.read_all_cbits()) == [0] * 32
    assert all(list(b.read(i)[0]) == [0] * 4 for i in range(8))
    b.close()
