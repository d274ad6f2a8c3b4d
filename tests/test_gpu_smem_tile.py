"""The pass over shared-memory tiles (complex128, and complex64 below 13 qubits) against
the one-pass-per-gate path and the oracle: every op kind, every tile width and the
widths' edges, terms that wait over several passes, conditions, and matrices that are
only nearly unitary.  1e-12 is the complex128 target; complex64 is held to 1e-5 (a few
hundred gates at 2^-24 each)."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu
TOL = {"c64": 1e-5, "c128": 1e-12}
SIZES = [("c128", n) for n in (1, 2, 3, 6, 7, 8, 9, 10, 13, 16, 17, 18, 20, 21)] + [
    ("c64", n) for n in (1, 2, 3, 5, 8, 9, 10, 11, 12, 13)]


def mixed_ops(n, seed, gates, conds=False):
    r = np.random.Generator(np.random.PCG64([n, seed]))
    names = ["x", "y", "z", "h", "s", "sdg", "t", "tdg", "u3", "p", "rz"]
    ops = []
    for _ in range(gates):
        k = names[int(r.integers(len(names)))]
        qs = [int(q) for q in r.permutation(n)[:1 + int(min(n - 1, r.integers(4)))]]
        cond = (int(r.integers(6)),) if conds and r.random() < 0.4 else ()
        ops.append(workloads.Op(k, (qs[0],), controls=tuple(qs[1:]), cond=cond, params=tuple(
            float(x) for x in r.uniform(0, 6.2, {"u3": 3, "p": 1, "rz": 1}.get(k, 0)))))
    return ops


@pytest.mark.parametrize("prec,n", SIZES)
def test_mixed_circuits(n, prec):
    from paper_1908_07187_gb300 import qk

    ops = mixed_ops(n, 1, 220 if n < 18 else 120) + workloads.qft_ops(range(n))
    psi = workloads.random_state(n, 5)
    got = []
    for mode in ("fused", "plain"):
        with qk.Context(prec, mode) as ctx:
            ctx.add_qubits(n)
            ctx.set_state(psi)
            qk.run_ops(ctx, ops)
            got.append(ctx.get_state())
    assert np.max(np.abs(got[0] - got[1])) <= TOL[prec]
    if n <= 16:
        ref = oracle.OracleState(n, psi=psi)
        for op in ops:
            ref.apply_op(op)
        assert np.max(np.abs(got[0] - ref.psi)) <= TOL[prec]


@pytest.mark.parametrize("prec", ["c64", "c128"])
@pytest.mark.parametrize("n", [2, 8, 12, 17])
def test_conditions_more_than_one_pass_holds(n, prec):
    from paper_1908_07187_gb300 import qk

    ops = mixed_ops(n, 2, 150, conds=True)
    psi = workloads.random_state(n, 6)
    got = []
    for mode in ("fused", "plain"):
        with qk.Context(prec, mode) as ctx:
            ctx.add_qubits(n)
            ctx.add_cbits(6)
            ctx.set_state(psi)
            ctx.write_cbits(0, [1, 0, 1, 1, 0, 1])
            qk.run_ops(ctx, ops)
            got.append(ctx.get_state())
    assert np.max(np.abs(got[0] - got[1])) <= TOL[prec]


@pytest.mark.parametrize("prec,n", [("c128", 5), ("c128", 14), ("c64", 5), ("c64", 11)])
def test_loose_matrices_are_taken_as_they_are(n, prec):
    """One-qubit matrices that a wide tolerance lets in, plain and diagonal."""
    from paper_1908_07187_gb300 import qk

    r = np.random.Generator(np.random.PCG64(n))
    psi = workloads.random_state(n, 7)
    got = []
    for mode in ("fused", "plain"):
        r = np.random.Generator(np.random.PCG64(n))
        with qk.Context(prec, mode) as ctx:
            ctx.add_qubits(n)
            ctx.set_state(psi)
            for j in range(20):
                u, _ = np.linalg.qr(r.standard_normal((2, 2)) + 1j * r.standard_normal((2, 2)))
                u = u + 1e-3 * r.standard_normal((2, 2))
                if j % 4 == 3:
                    u = np.diag([1.002, 0.997j])
                q = [int(x) for x in r.permutation(n)[:2]]
                ctx.apply_gate(ctx.define_gate_matrix(u, tol=0.1), (q[0],), (q[1],) if j % 3 == 2 else ())
                ctx.apply_gate("z", (q[1],), (q[0],))
            got.append(ctx.get_state())
    assert np.max(np.abs(got[0] - got[1])) <= TOL[prec]
