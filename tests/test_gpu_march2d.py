"""The marched 2D step (column strips, taken on large grids) gives the bits of
the tiled step (what a batch runs), for grids that end inside, at and just
past a strip, with every boundary; its Runge-Kutta stages match the oracle."""

import numpy as np
import pytest

from paper_1510_05061_gb300 import inputs

pytestmark = pytest.mark.gpu

BCS = [(inputs.BC_PERIODIC, inputs.BC_REFLECT), (inputs.BC_REFLECT, inputs.BC_PERIODIC),
       (inputs.BC_OUTFLOW, inputs.BC_OUTFLOW)]


@pytest.fixture(scope="module")
def hy():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1510_05061_gb300 import build, hydro

    build.build()
    hydro.load()
    return hydro


def data(nx, ny, precision, bc, scheme=inputs.HANCOCK):
    prob = inputs.Problem(ndim=2, n=(nx, ny, 1), bc_lo=(bc[0], bc[1], 0), bc_hi=(bc[0], bc[1], 0),
                          grav=(0.3, -0.5, 0.0), precision=precision, scheme=scheme)
    rng = np.random.default_rng(nx * 7 + ny)
    W = rng.uniform(-0.3, 0.3, prob.shape)
    W[0] += 1.0
    W[3] += 1.5
    return prob, W


@pytest.mark.parametrize("bc", BCS)
@pytest.mark.parametrize("precision,shape", [(inputs.FP64, (744, 801)), (inputs.FP64, (745, 740)), (inputs.FP64, (1001, 600)),
                                             (inputs.FP32, (124, 19001)), (inputs.FP32, (125, 24000)),
                                             (inputs.FP32, (1514, 1111)), (inputs.FP32, (1300, 1501))])
def test_strips_equal_tiles_bitwise(hy, bc, precision, shape):
    prob, W = data(*shape, precision, bc)
    sim = hy.Simulation(prob, W)
    sim.run_steps(3)
    batch = hy.Batch([(prob, W)])
    batch.step(3)
    assert np.array_equal(sim.get_state(), batch.get_state(0))
    assert sim.t == batch.t(0)
    sim.close()
    batch.close()


@pytest.mark.parametrize("bc", BCS)
def test_stages_match_oracle(hy, orc, bc):
    prob, W = data(870, 610, inputs.FP64, bc, inputs.SSPRK2)
    sim = hy.Simulation(prob, W)
    sim.run_steps(2)
    o = orc.Oracle(prob)
    U, t, _, _ = o.run(o.state_from_prim(W), max_steps=2)
    G = sim.conserved()
    for q in range(4):
        assert np.abs(G[q] - U[q]).sum() <= 1e-10 * np.abs(U[q]).sum()
    assert abs(sim.t - t) <= 1e-13 * t
    sim.close()
