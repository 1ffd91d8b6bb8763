"""The default launch shape (tile and balanced z partition chosen from the
grid) gives the bits of a fixed tile on z-chunks, on both sides of the sizes
where the choice changes."""

import numpy as np
import pytest

from paper_1510_05061_gb300 import inputs

pytestmark = pytest.mark.gpu

SHAPES = [(2, 2, 2), (16, 16, 16), (17, 5, 40), (33, 31, 9), (200, 8, 3), (64, 40, 33)]


@pytest.fixture(scope="module")
def hy():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1510_05061_gb300 import build, hydro

    build.build()
    hydro.load()
    return hydro


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("precision", [inputs.FP64, inputs.FP32])
@pytest.mark.parametrize("scheme,recon", [(inputs.HANCOCK, inputs.PLM), (inputs.SSPRK2, inputs.PLM),
                                          (inputs.SSPRK2, inputs.PPM)])
def test_default_equals_fixed_tile(hy, shape, precision, scheme, recon):
    if recon == inputs.PPM and min(shape) < 3:
        pytest.skip("PPM needs three cells per axis")
    prob = inputs.Problem(ndim=3, n=shape, bc_lo=(1, 2, 0), bc_hi=(1, 2, 0), grav=(0.1, -0.2, -0.3),
                          precision=precision, scheme=scheme, recon=recon)
    rng = np.random.default_rng(5)
    W = rng.uniform(-0.2, 0.2, prob.shape)
    W[0] += 1.0
    W[4] += 1.5
    outs = []
    for fixed in (False, True):
        sim = hy.Simulation(prob, W)
        if fixed:
            sim.configure(2, 4)
        sim.run_steps(3)
        outs.append((sim.get_state(), sim.t))
        sim.configure(1, 0)   # 0: the default partition again
        sim.run_steps(2)
        outs[-1] += (sim.get_state(),)
        sim.close()
    assert np.array_equal(outs[0][0], outs[1][0]) and outs[0][1] == outs[1][1]
    assert np.array_equal(outs[0][2], outs[1][2])
