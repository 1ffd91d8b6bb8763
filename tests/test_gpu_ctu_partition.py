"""GPU: the 3D corner transport upwind step where its z partition and thread
lists can go wrong: one-piece chunks, the balanced grid, more tiles than
resident CTAs, the fewest planes, ragged tiles and walls, in both precisions,
against the FP64 oracle."""

import numpy as np
import pytest

from paper_1510_05061_gb300 import inputs
from paper_1510_05061_gb300.inputs import BC_OUTFLOW, BC_PERIODIC, BC_REFLECT

from test_gpu_ctu import ctu, hy, orc  # noqa: F401  (fixtures)
from test_gpu_parity import assert_parity, smooth_random

pytestmark = pytest.mark.gpu


# one piece per CTA, one and several planes; balanced; more tiles than CTAs; two planes
@pytest.mark.parametrize("n", [(16, 16, 16), (40, 37, 41), (100, 60, 50), (210, 205, 5), (17, 33, 2)])
@pytest.mark.parametrize("bc", [BC_PERIODIC, BC_REFLECT, BC_OUTFLOW])
def test_partition_against_the_oracle(hy, orc, n, bc):  # noqa: F811
    walls = (bc,) * 3
    prob = ctu(inputs.Problem(ndim=3, n=n, bc_lo=walls, bc_hi=walls, grav=(0.1, -0.2, -0.3)))
    W = smooth_random(prob, 5)
    o = orc.Oracle(prob)
    V, _, _, _ = o.run(o.state_from_prim(W), max_steps=2)
    V = o.total(V)
    for precision, tol in ((inputs.FP64, 1e-10), (inputs.FP32, 1e-5)):
        # FP32: some 20 roundings of 6e-8 per cell and step on values of order one
        sim = hy.Simulation(prob.replace(precision=precision), W)
        sim.run_steps(2)
        assert_parity(np.asarray(sim.conserved()), V, tol, f"{n} {precision}")
