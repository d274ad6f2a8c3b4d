"""Reading many circuits of a batch: reads in order take following circuits along, in windows
that grow; every order, with and without states, small and large circuits mixed, gives each
circuit's own result, and reading two circuits of a large batch does not bring all of it over."""
import os

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def fill(b, count, seed):
    """Circuits of 1..13 qubits with some of 14 between, each in a basis state of its own; the
    small ones measure it into their cbits."""
    r = np.random.Generator(np.random.PCG64([count, seed]))
    want = []
    for i in range(count):
        n = 14 if i % 11 == 5 else int(r.integers(1, 14))
        x = int(r.integers(1 << n))
        m = 0 if n > 13 else int(r.integers(0, n + 1))
        ops = [workloads.Op("x", (q,)) for q in range(n) if (x >> q) & 1]
        if m:
            ops.append(workloads.Op("measure", tuple(range(m)), uniforms=(0.5,) * m, cbits=tuple(range(m))))
        b.add_ops(n, m, ops)
        want.append((n, x, [(x >> q) & 1 for q in range(m)]))
    b.run()
    return want


def check(b, want, i, state=True):
    n, x, bits = want[i]
    got, psi = b.read(i, state=state)
    assert list(got) == bits, i
    if state:
        assert psi.shape == (1 << n,) and abs(psi[x]) == 1 and np.count_nonzero(psi) == 1, i


@pytest.mark.parametrize("count", [2, 3, 6, 23, 300])
def test_every_order(count):
    from paper_1908_07187_gb300 import qk

    b = qk.Batch()
    for seed in range(2):
        b.clear()
        want = fill(b, count, seed)
        r = np.random.Generator(np.random.PCG64(count))
        orders = [range(count), range(0, count, 2), range(0, count, 3), range(count - 1, -1, -1),
                  [int(i) for i in r.permutation(count)], list(range(count // 2, count)) + list(range(count // 2))]
        for k, order in enumerate(orders):
            for i in order:
                check(b, want, i)
        for i in range(count):                       # cbits alone, then with states
            check(b, want, i, state=False)
        for i in range(count):
            check(b, want, i, state=i % 3 != 1)
    b.close()


def resident():
    with open("/proc/self/statm") as f:
        return int(f.read().split()[1]) * os.sysconf("SC_PAGE_SIZE")


def test_two_reads_do_not_copy_the_batch():
    from paper_1908_07187_gb300 import qk

    b = qk.Batch()
    for _ in range(900):                             # 59 MB of states
        b.add_ops(13, 0, [workloads.Op("x", (3,))])
    b.run()
    b.read(0)
    before = resident()
    for i in (1, 2, 600):
        assert b.read(i)[1][8] == 1
    assert resident() - before < 16 << 20
    b.close()


def test_runs_that_store_no_small_states():
    """Large circuits' states are always kept; reading them in order, with cbits, takes no
    states of small circuits along from a run that stored none."""
    from paper_1908_07187_gb300 import qk

    b = qk.Batch()
    for i in range(60):
        n = 14 if i % 2 else 13
        b.add_ops(n, 2, [workloads.Op("x", (i % n,))])
    b.run(store_states=False)
    for i in range(60):
        bits, psi = b.read(i, state=i % 2 == 1)
        assert list(bits) == [0, 0]
        if i % 2:
            assert abs(psi[1 << (i % 14)]) == 1 and np.count_nonzero(psi) == 1
        else:
            with pytest.raises(qk.QKError) as e:
                b.read(i)
            assert e.value.status == qk.QK_EINVAL
    b.close()
