"""Spectrum, correlation and defects on the gridded fields at every grid size from the smallest to the largest: one
block or two kernels for the correlation (64 | 128 nodes a side), one or eight rows a block for the defects (128 | 256),
odd and even powers of two in the FFT.  The definitions of the oracle on the GPU's own grid; tolerances as in
test_gpu_diagnostics.py (1e-12, integers exact)."""
import numpy as np
import pytest

from _sph import GpuRun, params, random_velocity_ic, stable_dt

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_08919_gb300 import binding, build

    build.build()
    return binding


def test_every_grid_size(B):
    from oracle import diagnostics as D

    ic = random_velocity_ic(96, 12, u_scale=1e-2, rho_scale=1e-4)
    p = params(96, c0_min=0.05)
    p["dt"] = stable_dt(p)
    run = GpuRun(B, p, ic)
    try:
        run.step(4)
        for M in (8, 16, 32, 64, 128, 256, 512, 1024, 2048):
            g = B.ann_grid_fields(run.ctx, M)
            om = D.vorticity(g[0], g[1], p["L"])
            for origins in (True, False):
                C, _ = B.ann_vorticity_correlation(run.ctx, M, all_origins=origins)
                want = D.correlation(om, origins)
                tol = 1e-12 if origins else 1e-9 * np.abs(want).max()
                assert C.shape == want.shape and np.abs(C - want).max() <= tol, (M, origins)
            counts, m = B.ann_defects(run.ctx, M, with_map=True)
            mo, co = D.defects(g[2], g[3])
            assert np.array_equal(m, mo) and list(counts) == list(co), M
            E, (_, want) = B.ann_energy_spectrum(run.ctx, M), D.energy_spectrum(g[0], g[1], p["L"])
            assert np.abs(E - want).max() <= 1e-12 * want.sum(), M
    finally:
        run.close()
