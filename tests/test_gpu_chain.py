"""Steps that follow one another in the stream are not slower than steps
launched one by one: the next step's CTAs must not be placed before this
step's have left, or a grid that leaves slots open is spread unevenly.

Bound: the lone step's time contains the launch and the events, a few us of 30
to 70; 8 % above it is more than the runs differ by, and the uneven spread cost
15 to 25 %."""

import pytest

from paper_1510_05061_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hy():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1510_05061_gb300 import build, hydro

    build.build()
    hydro.load()
    return hydro


@pytest.mark.parametrize("n,variant,zchunk", [(96, 0, 12), (80, 0, 8), (128, 0, 32)])
def test_following_steps_keep_their_spread(hy, n, variant, zchunk):
    import torch

    prob, W = inputs.rayleigh_taylor(n, precision=inputs.FP32)
    sim = hy.Simulation(prob, W)
    sim.configure(variant, zchunk)

    def ms(steps):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        torch.cuda.synchronize()
        a.record()
        sim.run_steps(steps)
        b.record()
        b.synchronize()
        return a.elapsed_time(b) / steps

    ms(200)
    lone = sorted(ms(1) for _ in range(41))[20]
    chained = sorted(ms(40) for _ in range(11))[5]
    sim.close()
    assert chained <= 1.08 * lone, (chained, lone)
