"""The fused queue rewritten for tile passes: gates that follow one another on a qubit
become one, controlled gates become gates on the target around phases.  Every built-in
gate with 0 to 3 controls and conditions, runs that cancel, angles at which a controlled
gate is a multiple of 1 or nearly so, and circuits that only permute, which stay exact.
Against the oracle, at 1e-5 of the largest amplitude (200 gates at 2^-24)."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu

KINDS = ("x", "y", "z", "h", "s", "sdg", "t", "tdg", "u3", "p", "rz")
ANGLES = (0.0, 1e-9, 1e-7, np.pi, np.pi - 1e-8, 2 * np.pi, 0.7, 2.9, 5.1)


def ops_for(n, style, seed):
    r = np.random.Generator(np.random.PCG64([n, seed]))
    ops = []
    while len(ops) < 200:
        qs = [int(x) for x in r.permutation(n)]
        nc = int(r.integers(4)) if style != "runs" else int(r.integers(2))
        kind = KINDS[int(r.integers(len(KINDS)))]
        np_ = {"u3": 3, "p": 1, "rz": 1}.get(kind, 0)
        par = tuple(float(ANGLES[int(r.integers(len(ANGLES)))] if style == "angles" else r.uniform(0, 6.28))
                    for _ in range(np_))
        cond = (int(r.integers(4)),) if r.random() < 0.1 else ()
        op = workloads.Op(kind, (qs[0],), controls=tuple(qs[1:1 + nc]), params=par, cond=cond)
        ops += [op] * (int(r.integers(1, 4)) if style == "runs" else 1)   # x x, h h, cx cx, ...
        if style == "runs":
            ops.append(workloads.Op("h", (qs[0],)))
    return ops


# 21 and 22 qubits: either side of the kernel's two register budgets
@pytest.mark.parametrize("n,style", [(n, style) for n in (13, 14, 16) for style in ("controls", "angles", "runs")]
                         + [(21, "controls"), (22, "controls")])
def test_against_oracle(n, style):
    from paper_1908_07187_gb300 import qk

    bits = [1, 0, 1, 1]
    ops = ops_for(n, style, 5)
    psi = workloads.random_state(n, 9)
    with qk.Context("c64") as ctx:
        ctx.add_qubits(n)
        ctx.add_cbits(4)
        ctx.write_cbits(0, bits)
        ctx.set_state(psi)
        qk.run_ops(ctx, ops)
        got = ctx.get_state()
    ref = oracle.OracleState(n, 4, psi)
    for op in ops:
        if all(bits[c] for c in op.cond):
            ref.apply_op(workloads.Op(op.kind, op.targets, op.controls, op.params))
    assert np.max(np.abs(got - ref.psi)) <= 1e-5 * np.max(np.abs(ref.psi))


@pytest.mark.parametrize("n", [13, 15])
def test_permutations_stay_exact(n):
    from paper_1908_07187_gb300 import qk

    r = np.random.Generator(np.random.PCG64(n))
    at, ops = 0, []
    for _ in range(150):
        qs = [int(x) for x in r.permutation(n)[:1 + int(r.integers(3))]]
        ops.append(workloads.Op("x", (qs[0],), controls=tuple(qs[1:])))
        if all((at >> q) & 1 for q in qs[1:]):
            at ^= 1 << qs[0]
    with qk.Context("c64") as ctx:
        ctx.add_qubits(n)
        qk.run_ops(ctx, ops)
        got = ctx.get_state()
    want = np.zeros(1 << n, dtype=np.complex64)
    want[at] = 1.0
    assert np.array_equal(got, want)


@pytest.mark.parametrize("n", [13, 14])
def test_more_phases_than_table_slots(n):
    """Every gate with phase terms from other qubits: more of them in a pass than the
    kernel's tables have slots."""
    from paper_1908_07187_gb300 import qk

    r = np.random.Generator(np.random.PCG64(n))
    ops = []
    for _ in range(9):
        for q in range(n):
            for d in (3, 5, 8):
                ops.append(workloads.Op("p", (q,), controls=((q + d) % n,), params=(float(r.uniform(0, 6.28)),)))
            ops.append(workloads.Op("u3", (q,), params=tuple(float(x) for x in r.uniform(0, 6.28, 3))))
    psi = workloads.random_state(n, 2)
    with qk.Context("c64") as ctx:
        ctx.add_qubits(n)
        ctx.set_state(psi)
        qk.run_ops(ctx, ops)
        got = ctx.get_state()
    ref = oracle.OracleState(n, 0, psi)
    for op in ops:
        ref.apply_op(op)
    assert np.max(np.abs(got - ref.psi)) <= 1e-5 * np.max(np.abs(ref.psi))
