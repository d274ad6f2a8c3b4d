"""Reading a batch's circuits: the second read of a run copies every small circuit's
state and cbits to the host at once, later reads come from that copy.  Small circuits of
several sizes and large ones in one batch (the launches go round side streams), read in
any order, more than once, by several threads, after a second run and after clear; each
result equals the same circuit's in a batch of its own (the same kernels: bit-exact)."""
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

SIZES = (3, 12, 14, 7, 13, 7, 15, 9, 3)


def circuits(seed):
    out = []
    for i, n in enumerate(SIZES):
        r = np.random.Generator(np.random.PCG64([seed, i]))
        ops = []
        for _ in range(3):
            ops += [workloads.Op("u3", (q,), params=tuple(float(x) for x in r.uniform(0, 6.28, 3))) for q in range(n)]
            ops += [workloads.Op("z", (q + 1,), controls=(q,)) for q in range(n - 1)]
        ncb = 0
        if n <= 13 and i % 2 == 0:
            ncb = 2
            ops.append(workloads.Op("measure", (0, 1), uniforms=(float(r.uniform()), float(r.uniform())), cbits=(0, 1)))
        out.append((n, ncb, ops))
    return out


def alone(qk, circ):
    b = qk.Batch()
    b.add_ops(*circ)
    b.run()
    bits, psi = b.read(0)
    b.close()
    return list(bits), psi


def fill(b, circs):
    b.clear()
    for c in circs:
        b.add_ops(*c)
    b.run()


def test_reads_in_any_order_and_after_new_runs():
    from paper_1908_07187_gb300 import qk

    first, second = circuits(1), circuits(2)
    want = [[alone(qk, c) for c in cs] for cs in (first, second)]
    b = qk.Batch()
    for run, cs in enumerate((first, second, first[:4], second)):
        fill(b, cs)
        order = [int(i) for i in np.random.Generator(np.random.PCG64(run)).permutation(len(cs))]
        for i in order + order[::-1]:
            bits, psi = b.read(i)
            ref = want[run % 2 if run != 2 else 0][i]
            assert list(bits) == ref[0] and np.array_equal(psi, ref[1]), (run, i)
        if run == 0:
            b.run()                                  # the same program again
            assert np.array_equal(b.read(4)[1], want[0][4][1])
    b.close()


def test_reads_from_several_threads():
    from paper_1908_07187_gb300 import qk

    cs = circuits(3)
    want = [alone(qk, c) for c in cs]
    b = qk.Batch()
    fill(b, cs)
    with ThreadPoolExecutor(8) as pool:
        got = list(pool.map(b.read, list(range(len(cs))) * 4))
    for k, (bits, psi) in enumerate(got):
        assert list(bits) == want[k % len(cs)][0] and np.array_equal(psi, want[k % len(cs)][1])
    b.close()
