"""The FP64 steps do not depend on the units: a solve in units that differ by
powers of two gives the same bits, scaled, from the smallest cgs densities to
cells of a megaparsec, and reports a negative pressure at the same step.
(Powers of two change no mantissa, so nothing rounds differently.)"""

import numpy as np
import pytest

from paper_1510_05061_gb300 import inputs

pytestmark = pytest.mark.gpu

# log2 of the units of density, velocity and length
UNITS = [(-66, 0, 0), (-75, 0, 0), (-93, 0, 0), (-123, 0, 0), (-90, 27, 74), (-93, 27, 77), (-96, 23, 81),
         (-100, 23, 81), (-100, 23, 91), (0, 0, 125), (0, 0, 146), (0, -30, 0), (0, -45, 10), (0, 40, 0), (400, 20, -60),
         (-400, -20, 60), (90, -3, -100)]
# 2D: wide enough for the marched strips; 3D: ragged against the tiles
CASES = [(3, inputs.HANCOCK, inputs.PLM, 0), (3, inputs.SSPRK2, inputs.PLM, 0), (3, inputs.SSPRK2, inputs.PPM, 0),
         (3, inputs.CTU, inputs.PLM, 0), (3, inputs.HANCOCK, inputs.PLM, 1), (3, inputs.CTU, inputs.PLM, 1),
         (2, inputs.HANCOCK, inputs.PLM, 0), (2, inputs.SSPRK2, inputs.PLM, 0)]


@pytest.fixture(scope="module")
def hy():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1510_05061_gb300 import build, hydro

    build.build()
    hydro.load()
    return hydro


def problem(ndim, scheme, recon, hse, mach, cfl):
    """Crossing waves 20 cells long, velocities up to `mach` times the sound
    speed, in units of one; hse: on an exponential background."""
    n = (37, 21, 40) if ndim == 3 else (3000, 300, 1)
    prob = inputs.Problem(ndim=ndim, n=n, hi=(n[0] / 16, n[1] / 16, n[2] / 16 if ndim == 3 else 1.0), bc_lo=(1, 1, 1 - hse),
                          bc_hi=(1, 1, 1 - hse), gamma=5 / 3, cfl=cfl, scheme=scheme, recon=recon,
                          grav=(0.0, 0.0, -0.25 if hse else 0.0))
    axes = [2 * np.pi * (np.arange(n[d]) + 0.5).reshape([(1, 1, -1), (1, -1, 1), (-1, 1, 1)][d]) / 20 for d in range(ndim)]
    W = np.zeros(prob.shape)
    W[0], W[-1] = 1.0, 0.6
    for d in range(ndim):
        W[0] += 0.05 * np.cos(2 * axes[d] + d)
        W[-1] *= 1.0 + 0.2 * np.cos(axes[d] + 2 * d)
        W[1 + d] = mach / ndim * np.sin(axes[d])
    if hse:
        zc, zf = (np.arange(n[2] + 4) - 1.5) / 16, (np.arange(n[2] + 5) - 2.0) / 16
        rho, p = (lambda z: np.exp(-z / 2.4)), (lambda z: 0.6 * np.exp(-z / 2.4))
        prob = prob.replace(hse_subtract=1, bg_rho_c=rho(zc), bg_p_c=p(zc), bg_rho_f=rho(zf), bg_p_f=p(zf))
        W[0] *= rho(zc[2:-2])[:, None, None]
        W[-1] *= p(zc[2:-2])[:, None, None] / 0.6
    return prob, W


def scaled(prob, W, units):
    r, v, x = (2.0 ** u for u in units)
    kw = {k: getattr(prob, k) * (r if "rho" in k else r * v * v) for k in ("bg_rho_c", "bg_p_c", "bg_rho_f", "bg_p_f")
          if getattr(prob, k) is not None}
    return (prob.replace(hi=tuple(h * x for h in prob.hi), grav=tuple(g * v * v / x for g in prob.grav), **kw),
            W * np.array([r] + [v] * prob.ndim + [r * v * v]).reshape(-1, 1, 1, 1))


def solve(hy, prob, W, steps):
    """The state, the time and largest speed after each step, and whether the
    solve stopped."""
    sim = hy.Simulation(prob, W)
    seen, stopped = [], False
    try:
        for _ in range(steps):
            sim.run_steps(1)
            seen.append((sim.t, sim.max_speed))
    except hy.HydroError:
        stopped = True
    state = sim.get_state()
    sim.close()
    return state, seen, stopped


@pytest.mark.parametrize("mach,cfl", [(3.5, 0.8), (0.5, 0.8), (20.0, 3.0)])
@pytest.mark.parametrize("ndim,scheme,recon,hse", CASES)
def test_bits_do_not_depend_on_the_units(hy, ndim, scheme, recon, hse, mach, cfl):
    prob, W = problem(ndim, scheme, recon, hse, mach, cfl)
    base, seen, stopped = solve(hy, prob, W, 5)
    assert stopped == (cfl > 1.0)   # the large steps end in a negative pressure,
    # which a second Runge-Kutta stage and an open boundary below the background's
    # own pressure turn into NaN
    assert np.isfinite(base).all() or (stopped and (scheme == inputs.SSPRK2 or hse))
    for r, v, x in UNITS:
        state, seen_u, stopped_u = solve(hy, *scaled(prob, W, (r, v, x)), 5)
        scale = np.array([r] + [r + v] * ndim + [r + 2 * v]).reshape(-1, 1, 1, 1)
        assert stopped_u == stopped, (r, v, x)
        assert seen_u == [(np.ldexp(t, x - v), np.ldexp(s, v - x)) for t, s in seen], (r, v, x)
        assert np.array_equal(np.ldexp(state, -scale), base, equal_nan=True), (r, v, x)
