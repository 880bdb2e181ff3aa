"""Ensembles of small members that fill the GPU together: a member of few tiles has several lanes per particle
(8 at 96^2, 4 at 113^2, 2 at 150^2), which one thread then takes in turn.  Every member still ends with the
bits of a solo run, whichever way its passes are launched, and the ensemble is not slowed down by lanes
that the full GPU has no use for."""
import time

import numpy as np
import pytest

from _sph import gpu_params, params, random_velocity_ic, stable_dt

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_08919_gb300 import binding, build

    build.build()
    return binding


VARIANTS = {"paper": {}, "q_old": dict(q_new_in_momentum=0), "elastic": dict(elastic=1, A=0.3, B=0.2, C=0.5),
            "conservative": dict(conservative=1), "elastic_conservative": dict(elastic=1, conservative=1, A=0.3, B=0.2, C=0.5)}
SIDES = (96,) * 6 + (113,) * 4 + (150,) * 4   # particles x lanes: 0.83M side by side, 45,000 to 74,000 a member


def _load(B, ctx, ic):
    B.ann_set_particles(ctx, ic["x"], ic["y"], ic["ux"], ic["uy"], ic["q11"], ic["q12"], ic["rho"])


@pytest.mark.parametrize("variant", list(VARIANTS))
def test_lanes_in_turn_give_the_bits_of_a_solo_run(B, variant):
    mem = []
    for k, side in enumerate(SIDES):
        p = params(side, c0_min=0.5, **VARIANTS[variant])
        p["dt"] = stable_dt(p)
        ic = random_velocity_ic(side, 60 + k, u_scale=0.5 if k % 2 else 1e-2, rho_scale=1e-4)
        if variant.startswith("elastic"):
            ic["q11"], ic["q12"] = 0.05 * ic["q11"], 0.05 * ic["q12"]
        mem.append((p, ic))
    ens = B.ann_ensemble_create([gpu_params(B, p, ic["n"]) for p, ic in mem])
    try:
        for k, (_, ic) in enumerate(mem):
            _load(B, B.ann_ensemble_member(ens, k), ic)
        B.ann_ensemble_set_groups(ens, len(mem))   # side by side: in turn
        B.ann_ensemble_step(ens, 9)
        B.ann_ensemble_set_groups(ens, 1)          # one after the other: lanes on threads of their own
        B.ann_ensemble_step(ens, 3)
        for k in (0, 5, 6, 9, 10, 13):
            p, ic = mem[k]
            ctx = B.ann_ensemble_member(ens, k)
            solo = B.ann_create(gpu_params(B, p, ic["n"]))
            try:
                _load(B, solo, ic)
                B.ann_step(solo, 12)
                for f in ("X", "Y", "UX", "UY", "Q11", "Q12", "DRHO", "AX", "AY", "SUMW", "NNBR"):
                    got, want = B.ann_get_field(ctx, f, ic["n"]), B.ann_get_field(solo, f, ic["n"])
                    assert np.array_equal(got, want), (k, f)
            finally:
                B.ann_destroy(solo)
    finally:
        B.ann_ensemble_destroy(ens)


def test_sixteen_small_members_cost_less_than_four_solo_steps(B):
    """16 x 96^2 side by side against one 96^2 box alone, which leaves most of the GPU idle: 3.4 times its step with
    the lanes in turn, 4.8 times with each member's lanes on threads of their own."""
    p = params(96)
    p["dt"] = stable_dt(p)
    ic = random_velocity_ic(96, 7, u_scale=1e-3)

    def best(step):
        step(20)
        t = []
        for _ in range(9):
            t0 = time.perf_counter()
            step(50)
            t.append(time.perf_counter() - t0)
        return min(t)

    solo = B.ann_create(gpu_params(B, p, ic["n"]))
    ens = B.ann_ensemble_create([gpu_params(B, p, ic["n"])] * 16)
    try:
        _load(B, solo, ic)
        for k in range(16):
            _load(B, B.ann_ensemble_member(ens, k), ic)
        B.ann_ensemble_set_groups(ens, 16)
        one, all16 = best(lambda n: B.ann_step(solo, n)), best(lambda n: B.ann_ensemble_step(ens, n))
    finally:
        B.ann_destroy(solo)
        B.ann_ensemble_destroy(ens)
    print(f"solo {one / 50 * 1e6:.1f} us a step, 16 members {all16 / 50 * 1e6:.1f} us")
    assert all16 < 4.0 * one, (one, all16)
