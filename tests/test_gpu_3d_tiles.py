"""The 3D step's tiles against the FP64 3D oracle where the tiling can go wrong: boxes of three and four
cells a side (every cell in every halo), cells of 64 to 125 particles, more halo particles than a
block stages (the lists then name particles in global memory), and a box most of whose cells are
empty.  The measure and the bound (2e-5 normwise, identical neighbour counts) are those of
tests/test_gpu_3d.py: FP32 pair sums of ~250-420 terms with FP64 positions."""
import numpy as np
import pytest

import sph_inputs as si

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_08919_gb300 import binding, build

    build.build()
    return binding


def relerr(a, b):
    a, b = np.asarray(a, dtype=np.float64), np.asarray(b, dtype=np.float64)
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


# side, h / dx, box side over the lattice's side
CASES = {
    "3 cells a side, all halos the whole box": (14, 1.3, 1.0),
    "4 cells of 125": (20, 1.3, 1.0),
    "cells of 64 to 125": (22, 1.3, 1.0),
    "more halo particles than a block stages": (16, 1.55, 1.0),
    "seven of eight cells empty": (13, 1.3, 2.0),
}


@pytest.mark.parametrize("name", list(CASES))
def test_tiles_match_the_oracle(B, name):
    from oracle import oracle3d as O

    side, hd, stretch = CASES[name]
    ic = si.jittered_lattice3(side, seed=21, jitter=0.2, u_scale=0.2)
    n, L, h = ic["n"], stretch, hd / side   # the lattice fills the unit cube of a box of side L
    kw = dict(L=L, h=h, dt=1e-4, eta=0.2, A=0.05, B=0.3, zeta=0.3, c0_min=0.5)
    st = {k: ic[k] for k in ("x", "y", "z", "u", "q", "rho")}
    want, rec = O.step(O.make_params(**kw), st, 3, record=True)
    ctx = B.ann3_create(B.ann3_default_params(n=n, **kw))
    try:
        B.ann3_set_particles(ctx, *[ic[k] for k in ("x", "y", "z", "u", "q", "rho")])
        B.ann3_step(ctx, 3)
        got = {k: B.ann3_get_field(ctx, k, n) for k in B.FIELDS3}
    finally:
        B.ann3_destroy(ctx)
    x0 = np.stack([ic["x"], ic["y"], ic["z"]], axis=1)
    disp = lambda p: (p - x0) - L * np.round((p - x0) / L)   # noqa: E731
    errs = {"disp": relerr(disp(got["POS"]), disp(np.stack([want["x"], want["y"], want["z"]], axis=1))),
            "u": relerr(got["U"], want["u"]), "q": relerr(got["Q"], want["q"]),
            "rho-1": relerr(got["RHO"][:, 0] - 1.0, want["rho"] - 1.0), "a": relerr(got["A"], want["a"]),
            "sumW": relerr(got["SUMW"][:, 0], rec["sumW"]), "gradu": relerr(got["GRADU"], rec["gradu"]),
            "lapQ": relerr(got["LAPQ"], rec["lapQ"]), "qrate": relerr(got["QRATE"], rec["qrate"]),
            "p": relerr(got["P"][:, 0], rec["p"])}
    print(name, {k: f"{v:.2e}" for k, v in errs.items()})
    assert np.array_equal(got["NNBR"][:, 0].astype(np.int64), rec["nnbr"])
    assert max(errs.values()) < 2e-5, errs
