"""The surrogate's backward kernels at row counts that do not fill their 128-row tiles (169 rows: a whole tile
and 41 rows; 1,369; 20,449: more tiles than CTAs), against the oracle's hand-derived FP64 backward pass.  Bound as
in tests/test_gpu_surrogate.py: 6e-2 normwise per weight (BF16 activations and adjoints, 2^-9 each,
through four layers and back).  The weight gradients add their partial sums in a fixed order, so two
calls give the same bits; tendencies by particle and by component load the same graph."""
import numpy as np
import pytest

import sph_inputs as si
from _sph import gpu_params, params, relerr

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_08919_gb300 import binding, build

    build.build()
    return binding


@pytest.mark.parametrize("nx", [13, 37, 143])
def test_gradients_of_ragged_rows(B, orc, nx):
    from oracle import surrogate as S

    ic = si.jittered_lattice(nx, seed=41)
    r = si.uniform53(42, 2 * ic["n"]).reshape(2, -1) - 0.5
    ic["ux"], ic["uy"] = 0.02 * r[0], 0.02 * r[1]
    n, p = ic["n"], params(nx)
    us, ysq, ysu, k = 0.01, 0.02, 0.004, 8
    w = S.init_params(5)
    for key, s in (("b1", 0), ("b2", 1), ("b3", 2), ("bo", 3)):
        w[key] = 0.2 * (si.uniform53(60 + s, w[key].size) - 0.5)
    flat = np.concatenate([w[key].ravel() for key in S.ORDER]).astype(np.float32)
    split = lambda f: dict(zip(S.ORDER, (v.reshape(S.SHAPES[key]) for key, v in zip(S.ORDER, np.split(   # noqa: E731
        f.astype(np.float64), np.cumsum([int(np.prod(S.SHAPES[key])) for key in S.ORDER])[:-1])))))
    tend = (si.uniform53(24, 8 * n).reshape(-1, 8) - 0.5) * [3.0, 3.0, 10.0, 10.0, 50.0, 50.0, 2.0, 2.0]
    tend = tend.astype(np.float32)
    t = si.uniform53(23, 4 * n).reshape(-1, 4) - 0.5
    ctx, sg = B.ann_create(gpu_params(B, p, n)), B.ann_surrogate_create(n)
    try:
        B.ann_set_particles(ctx, ic["x"], ic["y"], ic["ux"], ic["uy"], ic["q11"], ic["q12"], ic["rho"])
        B.ann_surrogate_set_params(sg, flat)
        B.ann_surrogate_set_scales(sg, us, ysq, ysu, k)
        B.ann_surrogate_load(sg, ctx, tend)                           # n x 8: sorted on the device
        y = B.ann_surrogate_forward(sg, n)
        B.ann_surrogate_load(sg, ctx, np.ascontiguousarray(tend.T))   # component-major, as the C call takes it
        assert np.array_equal(y, B.ann_surrogate_forward(sg, n))
        loss, g = B.ann_surrogate_gradients(sg, t)
        loss2, g2 = B.ann_surrogate_gradients(sg, t)
    finally:
        B.ann_surrogate_destroy(sg)
        B.ann_destroy(ctx)
    w = split(flat)
    rp, cols = orc.neighbors(ic["x"], ic["y"], 1.0, p["h"], mode="cells")
    G = S.Graph(ic["x"], ic["y"], 1.0, p["h"], rp, cols)
    Gn = S.Graph(ic["x"], ic["y"], 1.0, p["h"], rp, cols, radius=2.0)
    x = S.features(G, ic["q11"], ic["q12"], ic["ux"], ic["uy"], tend.astype(np.float64), us, k * p["dt"],
                   p["Gamma"] * p["K"], ysq, ysu)
    yo, c = S.forward(w, Gn, x)
    go, got = S.backward(w, Gn, c, yo, t), split(g)
    errs = {key: relerr(got[key], go[key]) for key in S.ORDER}
    print(nx, {key: f"{v:.1e}" for key, v in errs.items()})
    assert max(errs.values()) <= 6e-2, errs
    first = slice(0, g.size - 4)   # bo's four sums go through atomics
    assert np.array_equal(g[first], g2[first]) and abs(loss - loss2) <= 1e-12 * abs(loss)
