"""Tiles that hold only zeros are left as they are by a fused pass: states with one
nonzero amplitude anywhere, states that are zero but for the last tile, negative zeros,
a tile whose only content is not a number, and the first passes from |0...0>.  Against
the oracle (complex64 1e-5, complex128 1e-13 of the largest amplitude: 150 gates)."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu

TOL = {"c64": 1e-5, "c128": 1e-13}


def ops_for(n, seed):
    r = np.random.Generator(np.random.PCG64([n, seed]))
    ops = []
    for step in range(150):
        # gates gather on a few qubits at a time, so that passes differ and support grows slowly
        lo = int(r.integers(n)) if step % 25 == 0 else lo
        q = (lo + int(r.integers(4))) % n
        d = (q + 1 + int(r.integers(n - 1))) % n
        if r.random() < 0.6:
            ops.append(workloads.Op("u3", (q,), params=tuple(float(x) for x in r.uniform(0, 6.28, 3))))
        else:
            ops.append(workloads.Op(("x", "z", "y")[int(r.integers(3))], (q,), controls=(d,)))
    return ops


def run(n, prec, psi, ops):
    from paper_1908_07187_gb300 import qk

    with qk.Context(prec) as ctx:
        ctx.add_qubits(n)
        if psi is not None:
            ctx.set_state(psi)
        qk.run_ops(ctx, ops)
        return ctx.get_state()


@pytest.mark.parametrize("start", ["reset", "one", "last", "negative"])
@pytest.mark.parametrize("n,prec", [(13, "c64"), (17, "c64"), (20, "c64"), (11, "c64"), (9, "c128"), (14, "c128"),
                                    (18, "c128")])
def test_sparse_states(n, prec, start):
    r = np.random.Generator(np.random.PCG64([n, 4]))
    psi = np.zeros(1 << n, dtype=np.complex64 if prec == "c64" else np.complex128)
    if start == "negative":
        psi = -psi
    if start in ("one", "negative"):
        psi[int(r.integers(1 << n))] = 1.0
    elif start == "last":
        psi[-64:] = workloads.random_state(6, 3)
    else:
        psi[0] = 1.0
    ops = ops_for(n, 6)
    got = run(n, prec, None if start == "reset" else psi, ops)
    ref = oracle.OracleState(n, 0, psi)
    for op in ops:
        ref.apply_op(op)
    assert np.max(np.abs(got - ref.psi)) <= TOL[prec] * np.max(np.abs(ref.psi))


@pytest.mark.parametrize("n,prec", [(16, "c64"), (11, "c64"), (14, "c128")])
def test_not_a_number_is_not_zero(n, prec):
    psi = np.zeros(1 << n, dtype=np.complex64 if prec == "c64" else np.complex128)
    psi[0] = 1.0
    psi[-1] = np.nan
    got = run(n, prec, psi, [workloads.Op("h", (0,))])
    assert np.isnan(got[-1]) and np.isnan(got[-2])
    assert np.max(np.abs(got[:2] - np.sqrt(0.5))) <= 1e-6
