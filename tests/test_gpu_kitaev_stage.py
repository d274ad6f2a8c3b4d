"""The one-launch Kitaev stage against the six separate calls, over the sizes where a
thread holds 1, 2, 4 and 8 amplitudes, one block and all of them, and the first size
that is left to the two-kernel form; bits equal, amplitudes to the working precision
after four stages."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,n", [("c64", n) for n in (2, 3, 6, 10, 17, 18, 19, 20, 21, 22, 23)] + [
    ("c128", n) for n in (2, 7, 18, 19, 20, 21)])
def test_stage_equals_its_calls(n, prec):
    from paper_1908_07187_gb300 import qk

    r = np.random.Generator(np.random.PCG64([n, 4]))
    control = int(r.integers(n))
    free = [q for q in range(n) if q != control]
    reg = [int(q) for q in r.permutation(free)[:max(1, n - 1 - int(r.integers(2)))]]
    if n > 16:
        reg = [q for q in free[::-1]][:16]          # consecutive but for the control
    f = [int(x) for x in r.permutation(1 << min(len(reg), 12))]
    half = workloads.random_state(n - 1, 60 + n)
    psi = np.zeros(1 << n, dtype=np.complex128)
    i = np.arange(1 << (n - 1))
    lo = i & ((1 << control) - 1)
    psi[((i - lo) << 1) | lo] = half                # the control is |0>
    got = []
    for fused in (True, False):
        with qk.Context(prec) as ctx:
            ctx.add_qubits(n)
            ctx.add_cbits(4)
            ctx.set_state(psi)
            gid = ctx.define_gate_perm_table(f) if len(reg) <= 12 else ctx.define_gate_perm_mulmod(16, 40503, 65521)
            for e in range(4):
                u = (0.37, 0.81, 0.12, 0.55)[e]
                ph = list(range(e - 1, -1, -1))
                if fused:
                    ctx.apply_kitaev_stage(control, gid, reg, ph, u, e)
                    continue
                ctx.apply_gate("h", (control,))
                ctx.apply_gate(gid, reg, (control,))
                ctx.apply_rphase_cbits(control, ph)
                ctx.apply_gate("h", (control,))
                ctx.measure((control,), (u,), (e,), wait=False)
                ctx.apply_gate("x", (control,), (), (e,))
            ctx.sync()
            got.append((list(ctx.read_cbits()), ctx.get_state()))
    assert got[0][0] == got[1][0]
    scale = np.max(np.abs(got[1][1]))
    assert np.max(np.abs(got[0][1] - got[1][1])) <= (3e-6 if prec == "c64" else 1e-14) * scale
