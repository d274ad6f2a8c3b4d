"""Runs that follow one another without a wait, each with more circuits than the last, behind
other work on the batch's stream: every run uploads its own program."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def test_runs_without_waiting():
    import torch

    from paper_1908_07187_gb300 import qk

    r = np.random.Generator(np.random.PCG64(5))
    stream = torch.cuda.Stream()
    busy = torch.empty(1 << 28, device="cuda")
    for trial in range(4):
        b, want = qk.Batch(stream=stream.cuda_stream), []
        with torch.cuda.stream(stream):
            for _ in range(30):                      # about 10 ms in front of the first upload
                busy.mul_(1.0)
        for k in range(4):
            for _ in range(5 + 7 * k):
                n = int(r.integers(2, 13))
                x = int(r.integers(1 << n))
                b.add_ops(n, 0, [workloads.Op("x", (q,)) for q in range(n) if (x >> q) & 1])
                want.append(x)
            b.run()
        for i, x in enumerate(want):
            psi = b.read(i)[1]
            assert abs(psi[x]) == 1 and np.count_nonzero(psi) == 1
        b.close()
