"""The FP64 reciprocal and reciprocal square root refined on the integer pipe:
every binade, mantissas at the ends and middle of a binade, and the arguments
outside their normal range.

Tolerance: half an ulp for the rounding, plus what the second-order series
leaves out and the fixed-point truncations: with the seeds' 2^-20 (relative)
below 2^-56 together, i.e. 0.07 ulp of 2^-52; 0.6 ulp bounds the sum."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1510_05061_gb300 import build, hydro

    build.build()
    hydro.load()
    return torch, hydro


def run(env, which, x):
    torch, hy = env
    xd = torch.as_tensor(x, device="cuda")
    out = torch.empty_like(xd)
    hy.hydro_selftest_math(which, xd.data_ptr(), 0, out.data_ptr(), xd.numel(), torch.cuda.current_stream().cuda_stream)
    return out.cpu().numpy()


def samples(rng, lo, hi):
    """Doubles with exponent fields lo..hi: random mantissas and the ones
    next to the ends of a binade."""
    n = 1 << 17
    m = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    m[: n // 8] &= np.uint64(0xFFFF)
    m[n // 8: n // 4] |= np.uint64(((1 << 52) - 1) & ~0xFFFF)
    m[n // 4: n // 4 + 8] = 0
    m[n // 4 + 8: n // 4 + 16] = (1 << 52) - 1
    e = rng.integers(lo, hi + 1, n).astype(np.uint64)
    return ((e << np.uint64(52)) | m).view(np.float64)


def ulps(rel, y):
    """|relative error| in units of the last place of y."""
    return np.abs(rel) * np.abs(np.frexp(y)[0]) * 2.0 ** 53


@pytest.mark.parametrize("lo,hi", [(1020, 1026), (2, 2040)])
def test_reciprocal_accuracy(env, lo, hi):
    x = samples(np.random.default_rng(7), lo, hi)
    x[::3] *= -1
    y = run(env, 0, x)
    rel = np.longdouble(x) * np.longdouble(y) - 1
    assert ulps(rel, y).max() <= 0.6
    assert np.array_equal(run(env, 0, 2.0 ** np.arange(-1000, 1000.0)), 2.0 ** -np.arange(-1000, 1000.0))


@pytest.mark.parametrize("lo,hi", [(1020, 1026), (1, 2046)])
def test_reciprocal_square_root_accuracy(env, lo, hi):
    x = samples(np.random.default_rng(8), lo, hi)
    y = run(env, 2, x)
    rel = (np.longdouble(y) * np.longdouble(y) * np.longdouble(x) - 1) / 2
    assert ulps(rel, y).max() <= 0.6
    assert np.array_equal(run(env, 2, 4.0 ** np.arange(-500, 500.0)), 2.0 ** -np.arange(-500, 500.0))


def test_outside_the_normal_range(env):
    x = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 1e-310, -1e-310, 2.0 ** 1022 * 1.5, -(2.0 ** 1023)])
    y = run(env, 0, x)
    assert np.isnan(y[:7]).all() and (y[7:] == 0.0).all()
    x = np.array([0.0, np.inf, 1e-310, 5e-324, -1.0, np.nan, -np.inf])
    y = run(env, 2, x)
    assert y[0] == np.inf and y[1] == 0.0 and np.isnan(y[4:]).all()
    assert np.allclose(y[2:4], 1.0 / np.sqrt(x[2:4]), rtol=1e-15)


@pytest.mark.parametrize("spread", [0, 1, 2, 3, 4, 60])
def test_mc_slope_bits(env, spread):
    """The integer slope has the bits of the FP64 formula, for exponent
    differences on both sides of the shortcut, ties of the rounding and
    differences from 2^-900 to 2^900."""
    torch, hy = env
    rng = np.random.default_rng(20 + spread)
    n = 1 << 17
    e = rng.integers(120, 1920, n)
    d = rng.integers(-spread, spread + 1, n)
    m = rng.integers(0, 1 << 52, (2, n), dtype=np.uint64)
    m[:, : n // 4] &= np.uint64(0xFFFFFFFFFFF00)
    m[:, n // 4: n // 3] |= np.uint64(0xFFFFFFFFFFF00)
    m[1, n // 3: n // 2] = m[0, n // 3: n // 2] ^ rng.integers(0, 8, n // 2 - n // 3, dtype=np.uint64)
    x = ((e.astype(np.uint64) << np.uint64(52)) | m[0]).view(np.float64)
    y = (((e + d).astype(np.uint64) << np.uint64(52)) | m[1]).view(np.float64)
    s = rng.choice([-1.0, 1.0], n)
    x, y = x * s, y * s
    y[::9] *= -1
    y[::17] = 0.0
    xd, yd = (torch.as_tensor(v, device="cuda") for v in (x, y))
    out = torch.empty_like(xd)
    hy.hydro_selftest_math(3, xd.data_ptr(), yd.data_ptr(), out.data_ptr(), n, torch.cuda.current_stream().cuda_stream)
    a = np.minimum(np.minimum(2 * np.abs(x), 2 * np.abs(y)), 0.5 * np.abs(x + y))
    want = np.where((np.sign(x) * np.sign(y)) > 0, np.copysign(a, y), 0.0)
    assert np.array_equal(out.cpu().numpy(), want)
