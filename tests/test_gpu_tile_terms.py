"""Diagonal terms of the fused tile pass: each waits in the planner until a gate acts on
one of its qubits and is applied there as a sign, a phase from thread and tile bits or
a register-pair factor.  Circuits chosen so that every placement occurs, with qubits
stored flipped (X), terms left over at the end, controlled and conditioned gates in
between, and terms that wait over several passes; against the oracle, at 1e-5 of the
largest amplitude of a normalised random state (a few hundred gates at 2^-24)."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu


def ops_for(n, style, seed):
    r = np.random.Generator(np.random.PCG64([n, seed]))
    ang = lambda: float(r.uniform(0, 6.28))  # noqa: E731
    ops = []
    for step in range(260 if n < 16 else 160):
        q, d, e = (int(x) for x in r.permutation(n)[:3])
        pick = float(r.random())
        if pick < 0.45:
            if style == "cz":
                ops.append(workloads.Op("z", (q,), controls=(d,)))
            elif style == "phase":
                ops.append(workloads.Op("p", (q,), controls=(d,), params=(ang(),)))
            else:
                ops.append(workloads.Op("rz", (q,), controls=(d,) if pick < 0.3 else (d, e), params=(ang(),)))
        elif pick < 0.8:
            k = ("u3", "h", "x", "y")[int(r.integers(4))]
            ops.append(workloads.Op(k, (q,), params=(ang(), ang(), ang()) if k == "u3" else ()))
        elif pick < 0.9:
            ops.append(workloads.Op("x", (q,), controls=(d,)))
        else:
            ops.append(workloads.Op("u3", (q,), controls=(d,) if pick < 0.95 else (), params=(ang(), ang(), ang()),
                                    cond=(int(r.integers(6)),) if style == "rz" else ()))
    for q in range(n - 1):                     # terms that nothing calls for
        ops.append(workloads.Op("p", (q,), controls=(q + 1,), params=(ang(),)))
        ops.append(workloads.Op("z", (q,), controls=((q + 5) % n,)))
    return ops


@pytest.mark.parametrize("style", ["cz", "phase", "rz"])
@pytest.mark.parametrize("n", [13, 14, 15, 17, 20])
def test_every_placement(n, style):
    from paper_1908_07187_gb300 import qk

    bits = [1, 0, 1, 1, 0, 1]
    ops = ops_for(n, style, 3)
    psi = workloads.random_state(n, 8)
    with qk.Context("c64") as ctx:
        ctx.add_qubits(n)
        ctx.add_cbits(6)
        ctx.write_cbits(0, bits)
        ctx.set_state(psi)
        qk.run_ops(ctx, ops)
        got = ctx.get_state()
    ref = oracle.OracleState(n, 6, psi)
    for op in ops:
        if all(bits[c] for c in op.cond):
            ref.apply_op(workloads.Op(op.kind, op.targets, op.controls, op.params))
    assert np.max(np.abs(got - ref.psi)) <= 1e-5 * np.max(np.abs(ref.psi))
