"""A batch of fixed membership finds back to its default partition: z-chunk 0
after other settings gives the same bits and the untuned speed (equal shares of
the columns, here several times as fast as chunks of 64 planes).

Bound: 10 %, more than the runs differ by."""

import numpy as np
import pytest

from paper_1510_05061_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_default_partition_returns():
    import torch

    from paper_1510_05061_gb300 import hydro as hy

    per = (inputs.BC_PERIODIC,) * 3
    items = []
    for i, n in enumerate((17, 32, 60)):
        prob = inputs.Problem(ndim=3, n=(n, n, n), bc_lo=per, bc_hi=per, precision=inputs.FP32)
        items.append((prob, np.ones(prob.shape) + 0.2 * np.random.default_rng(i).random(prob.shape)))
    a, b = hy.Batch(items), hy.Batch(items)

    def us(batch):
        out = []
        for _ in range(7):
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            torch.cuda.synchronize()
            e0.record(batch.stream)
            batch.step(20)
            e1.record(batch.stream)
            e1.synchronize()
            out.append(e0.elapsed_time(e1) / 20 * 1e3)
        return sorted(out)[3]

    us(a)
    untuned = us(a)
    us(b)
    b.configure(7, 64)
    chunks = us(b)
    best = min((b.configure(v, 0), us(b))[1] for v in (2, 7))
    assert best <= 1.1 * untuned < chunks, (best, untuned, chunks)
    a.step(280)   # as many steps as b
    for i in range(len(items)):
        assert a.nstep(i) == b.nstep(i)
        assert np.array_equal(a.get_state(i), b.get_state(i)), i
