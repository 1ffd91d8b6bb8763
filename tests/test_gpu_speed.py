"""The step's maximum signal speed, taken from the cells an FP32 estimate
cannot rule out, equals the one of a full evaluation of the new state, for
speeds that rise or fall along the march, single spikes, near-vacuum and
units outside FP32's range.

Tolerance: the two kernels order the same FP64 operations differently, a few
roundings of 2^-53 each: 1e-14."""

import numpy as np
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


def fields(kind, prob, rng):
    W = rng.uniform(-0.01, 0.01, prob.shape)
    z = np.linspace(0.0, 1.0, prob.n[2])[:, None, None]
    W[0] += 1.0
    W[4] += 1.0
    if kind == "rising":
        W[4] += 5.0 * z
    elif kind == "falling":
        W[4] += 5.0 * (1.0 - z)
    elif kind == "spike":
        W[4, prob.n[2] // 2 + 1, 3, 5] = 40.0
    elif kind == "vacuum":
        W[0] *= np.exp(-14.0 * z)
        W[4] *= np.exp(-14.0 * z)
    elif kind == "stream":
        W[3] += 30.0 * z
    return W


@pytest.mark.parametrize("scheme", [inputs.HANCOCK, inputs.SSPRK2])
@pytest.mark.parametrize("kind", ["rising", "falling", "spike", "vacuum", "stream"])
@pytest.mark.parametrize("rho_unit,speed_unit", [(1.0, 1.0), (1e30, 1e-6), (1e-45, 1e9)])
def test_max_speed_is_exact(hy, kind, scheme, rho_unit, speed_unit):
    prob = inputs.Problem(ndim=3, n=(37, 21, 30), bc_lo=(1, 2, 0), bc_hi=(1, 2, 0), scheme=scheme)
    W = fields(kind, prob, np.random.default_rng(11))
    W[0] *= rho_unit
    W[1:4] *= speed_unit
    W[4] *= rho_unit * speed_unit ** 2
    sim = hy.Simulation(prob, W)
    for _ in range(3):
        sim.run_steps(1)
        s, state = sim.max_speed, sim.get_state()
        assert np.isfinite(state).all()
        t, n = sim.t, sim.nstep
        sim.set_state(state, t, n)
        assert abs(s / sim.max_speed - 1.0) <= 1e-14
    sim.close()


@pytest.mark.parametrize("nz", [24, 60])
def test_max_speed_with_background(hy, nz):
    prob, W = inputs.filament_column(nz=nz, nxy=16, hse_subtract=1)
    sim = hy.Simulation(prob, W)
    for _ in range(4):
        sim.run_steps(1)
        s, state, t, n = sim.max_speed, sim.get_state(), sim.t, sim.nstep
        sim.set_state(state, t, n)
        assert abs(s / sim.max_speed - 1.0) <= 1e-14
    sim.close()
