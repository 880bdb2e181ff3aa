"""Positions through one step, bit for bit: the two half steps x + dt/2 u are FP64 sums of an FP32 product,
whatever the product (zero, subnormal, tiny, ordinary) and wherever the particle (a corner of the box or of
a cell).  Exact but for an FP32 subnormal, which may count as zero: 1e-37."""
import numpy as np
import pytest

from _sph import GpuRun, params, random_velocity_ic

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_08919_gb300 import binding, build

    build.build()
    return binding


def wrap(a):   # a value just below 0 rounds up to 1, which is 0
    a = np.where(a < 0.0, a + 1.0, a)
    return np.where(a >= 1.0, a - 1.0, a)


@pytest.mark.parametrize("u", [0.0, 1e-42, 3e-39, 1e-30, -1e-12, 0.31, -0.27])
def test_half_steps_are_exact(B, u):
    nx, dt = 32, 2.0 ** -14
    p = params(nx, apd=0)
    p["dt"] = dt
    ic = random_velocity_ic(nx, 5)
    ic["x"], ic["y"] = ic["x"] - ic["x"].min(), ic["y"] - ic["y"].min()   # lattice points on the corners
    ic["ux"][:], ic["uy"][:] = u, -0.5 * u
    run = GpuRun(B, p, ic)
    try:
        run.step(1)
        out = run.state()
    finally:
        run.close()
    hd = np.float32(0.5 * dt)
    for x, v, u0 in (("x", "ux", u), ("y", "uy", -0.5 * u)):
        want = wrap(ic[x] + np.float64(hd * np.float32(u0)))
        want = wrap(want + (hd * out[v].astype(np.float32)).astype(np.float64))
        assert np.abs(out[x] - want).max() <= 1e-37
