"""Contexts and batches driven from several threads at once, one thread each, whose launches
ask for different amounts of shared memory of the same kernels: every call succeeds and every
round of a thread gives the same state as the first."""
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def haar(r, d):
    q, t = np.linalg.qr(r.standard_normal((d, d)) + 1j * r.standard_normal((d, d)))
    return q * (np.diag(t) / np.abs(np.diag(t)))


def dense(qk, i):
    """Runs of 5-qubit gates on CUDA cores: one to four matrices in shared memory."""
    n, r = 20, np.random.Generator(np.random.PCG64(i))
    with qk.Context("c64", tensor_cores=False) as ctx:
        ctx.add_qubits(n)
        gates = [ctx.define_gate_matrix(haar(r, 32)) for _ in range(1 + i % 4)]
        first = None
        for k in range(400):
            ctx.reset()
            for j, g in enumerate(gates):
                ctx.apply_gate(g, (j, 8, 9, 10, 11))
            ctx.flush()
            if k % 100 == 0:
                psi = ctx.get_state()
                first = psi if first is None else first
                assert np.array_equal(psi, first)


def tiles(qk, i):
    """complex128 passes over tiles in shared memory, of different numbers of ops."""
    n = 21 + i % 2
    with qk.Context("c128") as ctx:
        ctx.add_qubits(n)
        first = None
        for k in range(60):
            ctx.reset()
            for _ in range(1 + 3 * (i % 4)):
                for q in range(8):
                    ctx.apply_gate("u3", (q,), params=(0.3 + q, 0.2, 0.1))
                    ctx.apply_gate("x", ((q + 1) % 8,), (q,))
            ctx.flush()
            if k % 20 == 0:
                psi = ctx.get_state()
                first = psi if first is None else first
                assert np.array_equal(psi, first)


def modexp(qk, i):
    """Tiled modular exponentiation: 64 and 128 KiB tiles."""
    w, t = (9, 8) if i % 2 else (12, 6)
    N = (1 << w) - 3
    with qk.Context("c64") as ctx:
        ctx.add_qubits(w + t)
        first = None
        for k in range(400):
            ctx.reset()
            for q in range(t):
                ctx.apply_gate("h", (q,))
            ctx.apply_gate("x", (t + w - 1,))
            ctx.apply_modexp(tuple(range(t, t + w)), tuple(range(t)), [pow(2, 1 << c, N) for c in range(t)], N)
            ctx.flush()
            if k % 100 == 0:
                psi = ctx.get_state()
                first = psi if first is None else first
                assert np.array_equal(psi, first)


def batch(qk, i):
    n = (13, 12, 11, 8)[i % 4]
    b = qk.Batch()
    first = None
    for k in range(60):
        b.clear()
        ops = [workloads.Op("h", (q,)) for q in range(n)] + [
            workloads.Op("mulmod", tuple(range(1, n)), (0,), params=(2, 0, (1 << (n - 1)) - 1))]
        for _ in range(4):
            b.add_ops(n, 0, ops)
        b.run()
        psi = b.read(k % 4)[1]
        first = psi if first is None else first
        assert np.array_equal(psi, first)
    b.close()


@pytest.mark.parametrize("work", [dense, tiles, modexp, batch])
def test_threads_with_different_launch_sizes(work):
    from paper_1908_07187_gb300 import qk

    with ThreadPoolExecutor(8) as pool:
        for f in [pool.submit(work, qk, i) for i in range(8)]:
            f.result()
