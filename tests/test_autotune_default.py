"""Host checks (no GPU) that tuning can only choose what is at least as fast as
the untuned solve: the default partition of every tile is among the timed
settings, and FP64 variants that are one kernel are timed once."""

import pytest

from paper_1510_05061_gb300 import autotune, hydro, inputs

from test_autotune_host import FakeSim, lib  # noqa: F401  (fixture)


class FakeBatch(FakeSim):
    def __init__(self, probs):
        super().__init__(probs[0])
        self.probs = probs

    def configure(self, v, z):
        if self.prob.precision == inputs.FP64 and v % 4 == 3:
            raise hydro.HydroError(hydro.HYDRO_ERR_INVALID_ARG, "hydro_batch_configure")
        super().configure(v, z)

    def step(self, n):
        pass


@pytest.mark.parametrize("batch", [False, True])
@pytest.mark.parametrize("precision", [inputs.FP64, inputs.FP32])
def test_default_is_a_candidate(lib, monkeypatch, precision, batch):  # noqa: F811
    prob, _ = inputs.rayleigh_taylor(8, nz=40, precision=precision)
    cost = lambda s, steps: 1.0 + 0.01 * s.v + (0.0 if s.z == 0 else 0.5)   # noqa: E731
    monkeypatch.setattr(autotune, "sim_signature", lambda s: "host-test")
    monkeypatch.setattr(autotune, "signature", lambda s: "host-test")
    monkeypatch.setattr(autotune, "time_sim_steps", cost)
    monkeypatch.setattr(autotune, "time_steps", cost)
    sim = FakeBatch([prob]) if batch else FakeSim(prob)
    choice = (autotune.tune_batch if batch else autotune.tune_simulation)(sim, use_cache=False)
    assert (choice["variant"], choice["zchunk"]) == (0, 0) and (sim.v, sim.z) == (0, 0)
    timed = {(r["variant"], r["zchunk"]) for r in choice["table"]}
    fp32 = precision == inputs.FP32
    assert {(v, 0) for v in (range(8) if fp32 else range(3))} <= timed
    assert fp32 or not any(4 <= v < 8 for v, _ in timed)
