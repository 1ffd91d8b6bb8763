"""The marched 2D step at shapes that take it, as the choice itself says
(csrc/plan.h): strips of 128 threads in both precisions and of 256 in FP32,
grids that end at, just before and one column past a strip; the MUSCL-Hancock
step has the bits of the tiled step (what a batch runs), the Runge-Kutta stages
match the oracle."""

import numpy as np
import pytest

from paper_1510_05061_gb300 import inputs

from test_gpu_march2d import BCS, data, hy  # noqa: F401  (fixture)
from test_gpu_parity import assert_parity
from test_plan2d import needs_gxx, plans

pytestmark = [pytest.mark.gpu, needs_gxx]

F64, F32 = inputs.FP64, inputs.FP32
SHAPES = [(F64, 744, 801, 128), (F64, 745, 1300, 128), (F64, 1001, 600, 128), (F32, 1365, 2239, 128), (F32, 505, 3000, 128),
          (F32, 124, 19001, 128), (F32, 249, 2600, 256), (F32, 252, 2600, 256), (F32, 2017, 700, 256), (F32, 1488, 1500, 256)]
# sums of some 30 terms per cell and stage, values of order one: 1e-10 of FP64 as
# elsewhere; FP32 two steps of 60 roundings of 6e-8, which mostly cancel: 1e-5
TOL = {F64: 1e-10, F32: 1e-5}


def marched(nx, ny, precision, threads, tmp_path):
    got = plans([(nx, ny, int(precision == F32), 0)], str(tmp_path))
    assert got[0][0] == threads, got


@pytest.mark.parametrize("precision,nx,ny,threads", SHAPES)
@pytest.mark.parametrize("bc", BCS)
def test_strips_have_the_tiles_bits(hy, tmp_path, precision, nx, ny, threads, bc):  # noqa: F811
    marched(nx, ny, precision, threads, tmp_path)
    prob, W = data(nx, ny, precision, bc)
    sim = hy.Simulation(prob, W)
    sim.run_steps(3)
    batch = hy.Batch([(prob, W)])
    batch.step(3)
    assert np.array_equal(sim.get_state(), batch.get_state(0))
    assert sim.t == batch.t(0)
    sim.close()
    batch.close()


@pytest.mark.parametrize("precision,nx,ny,threads", [SHAPES[1], SHAPES[4], SHAPES[6], SHAPES[8]])
@pytest.mark.parametrize("bc", BCS)
def test_stages_match_the_oracle(hy, orc, tmp_path, precision, nx, ny, threads, bc):  # noqa: F811
    marched(nx, ny, precision, threads, tmp_path)
    prob, W = data(nx, ny, precision, bc, inputs.SSPRK2)
    sim = hy.Simulation(prob, W)
    sim.run_steps(2)
    o = orc.Oracle(prob.replace(precision=F64))
    U, t, _, _ = o.run(o.state_from_prim(W), max_steps=2)
    assert_parity(np.asarray(sim.conserved()), U, TOL[precision], f"{nx}x{ny}")
    assert abs(sim.t - t) <= (1e-13 if precision == F64 else 1e-5) * t
    sim.close()
