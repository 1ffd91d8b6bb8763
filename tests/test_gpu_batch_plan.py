"""GPU: a batch in its default configuration (equal shares of all 3D columns)
gives the bits of the claimed chunks, for uneven and ragged boxes, and keeps
doing so when its membership changes."""

import ctypes as C

import numpy as np
import pytest

from paper_1510_05061_gb300 import inputs

pytestmark = pytest.mark.gpu

SIZES = {
    "one": [(16, 16, 16)],
    "flat": [(3, 70, 2), (33, 17, 5), (2, 2, 2)],
    "mixed": [(40, 24, 70), (17, 19, 23), (48, 30, 1), (33, 9, 41)],
}


def _items(sizes, precision, hse):
    out = []
    for i, n in enumerate(sizes):
        if hse:
            prob, W = inputs.rayleigh_taylor(n[0], seed=i, nz=n[2], hse_subtract=1)
        else:
            per = (inputs.BC_PERIODIC,) * 3
            prob = inputs.Problem(ndim=3 if n[2] > 1 else 2, n=n, bc_lo=per, bc_hi=per)
            W = np.ones(prob.shape) + 0.2 * np.random.default_rng(i).random(prob.shape)
        out.append((prob.replace(precision=precision), W))
    return out


@pytest.mark.parametrize("precision", [inputs.FP64, inputs.FP32])
@pytest.mark.parametrize("name,hse", [("one", 0), ("flat", 0), ("mixed", 0), ("rt", 1)])
def test_shares_give_the_chunks_bits(name, hse, precision):
    from paper_1510_05061_gb300 import hydro as hy

    sizes = SIZES.get(name, [(16, 16, 33), (24, 24, 20)])
    a, b = hy.Batch(_items(sizes, precision, hse)), hy.Batch(_items(sizes, precision, hse))
    b.configure(1, 9)
    a.step(5)
    b.step(5)
    for i in range(len(sizes)):
        assert np.array_equal(a.conserved(i), b.conserved(i)), i
        assert a.t(i) == b.t(i)
    if len(sizes) > 2:   # one instance leaves: the shares are cut again
        for x in (a, b):
            hy._check(hy.load().hydro_batch_remove(x.h, C.c_int(0)), "hydro_batch_remove")
            x.step(3)
        for i in range(1, len(sizes)):
            assert np.array_equal(a.conserved(i), b.conserved(i)), i
