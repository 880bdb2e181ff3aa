"""Performance cases: the calls a user of this library makes, over the sizes they are made at.

A case is one pass through the public binding (``paper_2108_08919_gb300.binding``).  The kinds:

* ``step``       ``steps`` time steps of a 2D box held in a context, then the state read into device
                 tensors (the plain solver; the paper's set-up, with the options of the C-ABI);
* ``roundtrip``  the host holds the state in page-locked arrays: upload, one step, read back;
* ``ensemble``   many boxes of uneven size stepped by one graph launch per step (parameter sweeps);
* ``train``      a stored snapshot pair: graph and features loaded, the surrogate's forward and
                 backward pass (loss and all parameter gradients);
* ``cycle``      a stored snapshot put into a running context, one recorded plain step and one
                 surrogate jump over k = 8 steps (the surrogate's evaluation);
* ``step3``      ``steps`` time steps of the three-dimensional variant, then its fields read;
* ``analyse``    a stored snapshot loaded and analysed on an M x M grid: energy spectrum, vorticity
                 correlation and defects (the results section's statistics).

Inputs: jittered lattices (5 % of the spacing, 20 % in 3D) with a random director per particle, as
the configurations state, in a moving state: a box-scale cellular flow plus a random velocity per
particle, so that pressure, viscous and displacement terms all act.  ``exact`` restates the method in
FP64 torch (dense neighbour rows), without the library.
"""
import math

import numpy as np
import torch

from paper_2108_08919_gb300 import binding as B

DEV = "cuda"
STATE = B.STATE_FIELDS         # X, Y, UX, UY, Q11, Q12, DRHO: the state a program reads
U_SCALE = 0.02                 # velocities of the moving states
HOVER = 1.3                    # h / dx, as the configurations state
SG_K = 8                       # steps a surrogate jump spans
SG_SHAPES = (("W1", (128, 32)), ("b1", (128,)), ("P1", (32, 128)), ("W2", (128, 160)), ("b2", (128,)),
             ("P2", (32, 128)), ("W3", (128, 160)), ("b3", (128,)), ("Wo", (4, 128)), ("bo", (4,)))


def _step(name, side, steps, **kw):
    c = {"name": name, "kind": "step", "side": side, "steps": steps, "eta": 1.0, "dt_check": False,
         "conservative": False, "zeta": 0.08, "K": 0.02}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest configuration (64^2, 100 steps): launches and latency
        _step("step_64", 64, 100, zeta=0.05, K=0.04),
        # the 20,000-step configuration's size and long-run parameters (eta 0.03, checked dt 1e-4)
        _step("step_256", 256, 20, eta=0.03, dt_check=True, zeta=0.1),
        # an odd size in the mode that conserves momentum to round-off
        _step("step_333_conservative", 333, 20, conservative=True),
        # the headline configuration: 1024^2
        _step("step_1024", 1024, 10),
        # a box far beyond the L2, where the step reaches its steady rate
        _step("step_4096", 4096, 2),
        # a host program that owns the state between steps (the end-to-end path), 1024^2
        {"name": "roundtrip_1024", "kind": "roundtrip", "side": 1024},
        # a (zeta, K) sweep: uneven members between 128^2 and 512^2, as the ensemble configuration
        {"name": "ensemble_16", "kind": "ensemble", "members": 16, "lo": 128, "hi": 512, "steps": 10},
        # one training pair of the surrogate at its training size
        {"name": "train_256", "kind": "train", "side": 256},
        # one recorded step and one jump at the evaluation size
        {"name": "cycle_1024", "kind": "cycle", "side": 1024},
        # the 3D variant at its default size and at one where it fills the GPU
        {"name": "step3_32", "kind": "step3", "side": 32, "steps": 40},
        {"name": "step3_64", "kind": "step3", "side": 64, "steps": 24},
        # a 1024^2 snapshot analysed at the particles' own resolution
        {"name": "analyse_1024", "kind": "analyse", "side": 1024, "grid": 1024},
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "roundtrip", "ensemble", "train", "cycle", "step3", "step3", "analyse"])
    zeta, K = round(0.01 * 20.0 ** rng.random(), 4), round(rng.uniform(0.01, 0.08), 4)
    if kind == "step":
        side = _log(rng, 40, 3000)
        cons = rng.random() < 0.25
        c = _step("", side, max(2, min(100, int(2e7 / side ** 2))), zeta=zeta, K=K, conservative=cons)
    elif kind == "roundtrip":
        c = {"kind": kind, "side": _log(rng, 128, 1400)}
    elif kind == "ensemble":
        lo = rng.randrange(100, 200)
        c = {"kind": kind, "members": rng.randrange(4, 21), "lo": lo, "hi": rng.randrange(lo + 40, 480), "steps": 10}
    elif kind == "train":
        c = {"kind": kind, "side": _log(rng, 60, 700)}
    elif kind == "cycle":
        c = {"kind": kind, "side": _log(rng, 100, 1200)}
    elif kind == "step3":
        side = _log(rng, 14, 80)
        c = {"kind": kind, "side": side, "steps": max(5, min(60, int(4e6 / side ** 3)))}
    else:
        c = {"kind": kind, "side": _log(rng, 100, 1400), "grid": rng.choice([128, 256, 512, 1024])}
    c.pop("name", None)
    return c


# ------------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------------

def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + salt) & 0x7FFFFFFFFFFFFFFF)
    return g


def _inputs2(side, seed, salt=0):
    """A jittered lattice of side^2 particles in the unit box, random directors, a moving state."""
    n, dx = side * side, 1.0 / side
    r = torch.rand((6, n), dtype=torch.float64, device=DEV, generator=_gen(seed, 7919 * salt + side))
    i = torch.arange(n, device=DEV)
    x = ((i % side).double() + 0.5 + 0.1 * (r[0] - 0.5)) * dx
    y = ((i // side).double() + 0.5 + 0.1 * (r[1] - 0.5)) * dx
    th = 2.0 * math.pi * r[2]
    s = 1.0 + 2e-3 * (r[3] - 0.5)
    ux = U_SCALE * (torch.sin(2 * math.pi * y) + 2.0 * r[4] - 1.0)
    uy = U_SCALE * (torch.sin(2 * math.pi * x) + 2.0 * r[5] - 1.0)
    return {"X": x, "Y": y, "UX": ux, "UY": uy, "Q11": s * torch.cos(th), "Q12": s * torch.sin(th)}


def _inputs3(side, seed):
    """A jittered cubic lattice, uniaxial Q about random directions, a moving state (host arrays)."""
    n, dx = side ** 3, 1.0 / side
    r = torch.rand((8, n), dtype=torch.float64, device=DEV, generator=_gen(seed, side))
    i = torch.arange(n, device=DEV)
    pos = [(c.double() + 0.5 + 0.4 * (r[k] - 0.5)) * dx
           for k, c in enumerate((i % side, (i // side) % side, i // (side * side)))]
    cz, ph = 2.0 * r[3] - 1.0, 2.0 * math.pi * r[4]
    sz = torch.sqrt(1.0 - cz * cz)
    a, b = sz * torch.cos(ph), sz * torch.sin(ph)
    q = 0.5 * torch.stack([a * a - 1 / 3, a * b, a * cz, b * b - 1 / 3, b * cz], 1)
    u = 0.5 * U_SCALE * (torch.stack([torch.sin(2 * math.pi * pos[(k + 1) % 3]) for k in range(3)], 1)
                   + 2.0 * r[5:8].T - 1.0)
    return {"x": pos[0], "y": pos[1], "z": pos[2], "u": u, "q": q}


def _params2(case, side):
    """Keyword parameters of ann_default_params for a 2D case; unit box."""
    p = dict(n=side * side, h=HOVER / side, eta=case.get("eta", 1.0), zeta=case.get("zeta", 0.08),
             K=case.get("K", 0.02), dt_mode=1)
    if case.get("dt_check"):   # the long runs: dt = 1e-4 checked, sound speed floored by the active velocity
        p.update(dt_mode=2, c0_min=10.0 * math.sqrt(p["K"] * p["zeta"]) / 0.34)
    if case.get("conservative"):
        p.update(momentum_mode=B.MOMENTUM_CONSERVATIVE)
    return p


def _params3(side):
    return dict(n=side ** 3, h=HOVER / side, dt=1e-5, eta=1.0, A=0.05, B=0.3, zeta=0.3, c0_min=0.5)


def _members(case):
    """(side, parameters) of each ensemble member: sides spread over [lo, hi], zeta log-spread over
    [0.01, 0.2], K spread over [0.01, 0.08] in another order."""
    m = case["members"]
    out = []
    for k in range(m):
        f, g = k / max(m - 1, 1), (k * 5 % m) / m
        side = int(round(case["lo"] + (case["hi"] - case["lo"]) * ((k * 7 % m) / max(m - 1, 1))))
        out.append((side, _params2({"zeta": 0.01 * 20.0 ** f, "K": 0.01 + 0.07 * g}, side)))
    return out


def _weights(seed):
    """He-scaled weights with a live output layer, as during training (flat FP32)."""
    g = _gen(seed, 3)
    out = []
    for name, shape in SG_SHAPES:
        w = torch.randn(shape, dtype=torch.float64, device=DEV, generator=g)
        w = 0.01 * w if name.startswith("b") else w * math.sqrt(2.0 / shape[1]) * (0.5 if name == "Wo" else 1.0)
        out.append(w.reshape(-1))
    return torch.cat(out).float().cpu().numpy()


SG_US, SG_YSQ, SG_YSU = 0.02, 1e-3, 1e-4   # velocity scale, increment scales of Q and u
SG_YS_CYCLE = 2e-3   # both increment scales of a cycle: a tenth of the increments of its eight steps


def _snapshot_pair(case, seed):
    """A training pair: a state, its tendencies and the targets (host FP32, ID order).  The
    tendencies are drawn at the size that makes each an O(1) feature, as the scales are chosen to."""
    side = case["side"]
    n = side * side
    kdt = SG_K * B_dt(case, side)
    ic = _inputs2(side, seed)
    g = _gen(seed, 17)
    r = 2.0 * torch.rand((n, 12), dtype=torch.float64, device=DEV, generator=g) - 1.0
    K, Gamma = 0.02, 0.34
    size = torch.tensor([SG_YSU, SG_YSU, SG_YSQ, SG_YSQ, SG_YSQ / (Gamma * K), SG_YSQ / (Gamma * K), 1.0, 1.0],
                        dtype=torch.float64, device=DEV) / kdt
    st = {k: ic[k] if k in "XY" else ic[k].float() for k in ic}
    st["DRHO"] = torch.zeros(n, dtype=torch.float32, device=DEV)
    return st, (r[:, :8] * size).float(), r[:, 8:].float()


def B_dt(case, side):
    """The step of dt_mode "stable": min(1e-4, 0.125 h^2 / nu, 0.125 h^2 / (Gamma K))."""
    h, p = HOVER / side, _params2(case, side)
    return min(1e-4, 0.125 * h * h / p["eta"], 0.125 * h * h / (0.34 * p["K"]))


# ------------------------------------------------------------------------------------------------
# what a program keeps
# ------------------------------------------------------------------------------------------------

class _Held:
    """Library handles a program keeps, released with the object."""

    def __init__(self):
        self._free = []

    def keep(self, handle, free):
        self._free.append((handle, free))
        return handle

    def __del__(self):
        while self._free:
            handle, free = self._free.pop()
            free(handle)


def _context(h, prm, ic):
    ctx = h.keep(B.ann_create(B.ann_default_params(**prm)), B.ann_destroy)
    torch.cuda.synchronize()   # the inputs were made on torch's stream
    B.ann_set_particles(ctx, ic["X"], ic["Y"], ic["UX"], ic["UY"], ic["Q11"], ic["Q12"])
    return ctx


def _state_tensors(n):
    return {f: torch.empty(n, dtype=torch.float64 if f in "XY" else torch.float32, device=DEV) for f in STATE}


def prepare(case, seed):
    h = _Held()
    h.case, kind = case, case["kind"]
    if kind in ("step", "cycle"):
        side = case["side"]
        h.n = side * side
        ic = _inputs2(side, seed)
        h.ctx = _context(h, _params2(case, side), ic)
        h.out = _state_tensors(h.n)
        if kind == "cycle":
            h.state = {k: ic[k] if k in "XY" else ic[k].float() for k in ic}
            h.sg = h.keep(B.ann_surrogate_create(h.n), B.ann_surrogate_destroy)
            B.ann_surrogate_set_params(h.sg, _weights(seed))
            B.ann_surrogate_set_scales(h.sg, SG_US, SG_YS_CYCLE, SG_YS_CYCLE, SG_K)
            B.ann_set_record(h.ctx, True)
    elif kind == "roundtrip":
        side = case["side"]
        h.n = side * side
        ic = _inputs2(side, seed)
        h.ctx = _context(h, _params2(case, side), ic)
        h.host = {}
        for f in B.FULL_STATE:   # with the acceleration, which the next step needs back
            t = torch.zeros(h.n, dtype=torch.float64 if f in "XY" else torch.float32, pin_memory=True)
            if f in ic:
                t.copy_(ic[f])
            h.host[f] = t.numpy()
        torch.cuda.synchronize()
    elif kind == "ensemble":
        mem = _members(case)
        h.ens = h.keep(B.ann_ensemble_create([B.ann_default_params(**p) for _, p in mem]), B.ann_ensemble_destroy)
        B.ann_ensemble_set_groups(h.ens, min(16, len(mem)))
        total = sum(s * s for s, _ in mem)
        h.out = _state_tensors(total)
        h.members, at = [], 0
        for k, (side, _) in enumerate(mem):
            ic = _inputs2(side, seed, k + 1)
            torch.cuda.synchronize()
            c = B.ann_ensemble_member(h.ens, k)
            B.ann_set_particles(c, ic["X"], ic["Y"], ic["UX"], ic["UY"], ic["Q11"], ic["Q12"])
            n = side * side
            h.members.append((c, n, {f: t[at:at + n] for f, t in h.out.items()}))
            at += n
    elif kind == "train":
        side = case["side"]
        h.n = side * side
        h.ctx = h.keep(B.ann_create(B.ann_default_params(**_params2(case, side))), B.ann_destroy)
        h.sg = h.keep(B.ann_surrogate_create(h.n), B.ann_surrogate_destroy)
        B.ann_surrogate_set_params(h.sg, _weights(seed))
        B.ann_surrogate_set_scales(h.sg, SG_US, SG_YSQ, SG_YSU, SG_K)
        h.state, tend, target = _snapshot_pair(case, seed)
        h.tend, h.target = tend.cpu().numpy(), target.cpu().numpy()
    elif kind == "step3":
        side = case["side"]
        h.n = side ** 3
        ic = {k: v.cpu().numpy() for k, v in _inputs3(side, seed).items()}
        h.ctx = h.keep(B.ann3_create(B.ann3_default_params(**_params3(side))), B.ann3_destroy)
        B.ann3_set_particles(h.ctx, ic["x"], ic["y"], ic["z"], ic["u"], ic["q"])
    else:
        side = case["side"]
        h.n = side * side
        h.ctx = h.keep(B.ann_create(B.ann_default_params(**_params2(case, side))), B.ann_destroy)
        ic = _inputs2(side, seed)
        h.state = {k: ic[k] if k in "XY" else ic[k].float() for k in ic}
    torch.cuda.synchronize()
    return h


def run(h):
    case = h.case
    kind = case["kind"]
    if kind == "step":
        B.ann_step(h.ctx, case["steps"])
        return B.ann_get_state(h.ctx, h.n, h.out)
    if kind == "roundtrip":
        B.ann_update_state(h.ctx, h.host)
        B.ann_step(h.ctx, 1)
        return B.ann_get_state(h.ctx, h.n, h.host)
    if kind == "ensemble":
        B.ann_ensemble_step(h.ens, case["steps"])
        for c, n, views in h.members:
            B.ann_get_state(c, n, views)
        return h.out
    if kind == "train":
        B.ann_set_state(h.ctx, h.state)
        B.ann_surrogate_load(h.sg, h.ctx, h.tend)
        loss, grads = B.ann_surrogate_gradients(h.sg, h.target)
        return {"loss": np.float32(loss), "grads": grads}
    if kind == "cycle":
        B.ann_update_state(h.ctx, h.state)
        B.ann_step(h.ctx, 1)
        B.ann_surrogate_jump(h.sg, h.ctx)
        return B.ann_get_state(h.ctx, h.n, h.out)
    if kind == "step3":
        B.ann3_step(h.ctx, case["steps"])
        # u and Q are FP32 in the solver and only widened by the call: a program keeps them as FP32
        return {"pos": B.ann3_get_field(h.ctx, "POS", h.n),
                "u": B.ann3_get_field(h.ctx, "U", h.n).astype(np.float32),
                "q": B.ann3_get_field(h.ctx, "Q", h.n).astype(np.float32)}
    M = case["grid"]
    B.ann_set_state(h.ctx, h.state)
    E = B.ann_energy_spectrum(h.ctx, M)
    C, _ = B.ann_vorticity_correlation(h.ctx, M)
    counts, winding = B.ann_defects(h.ctx, M, with_map=True)
    return {"E": E, "C": C, "counts": counts, "map": winding}


# ------------------------------------------------------------------------------------------------
# work: inputs once, outputs once, and the pair arithmetic of the method
# ------------------------------------------------------------------------------------------------

def work(case):
    kind = case["kind"]
    if kind == "step3":
        n, s = case["side"] ** 3, case["steps"]
        # state 72 B in and out per step (FP64 positions, u, Q, density, a); ~250 neighbours of 360 flops
        return {"bytes": n * (144.0 * s + 44), "flops": n * s * 250 * 360.0}
    if kind == "ensemble":
        n, s = sum(side * side for side, _ in _members(case)), case["steps"]
    else:
        n, s = case["side"] ** 2, case.get("steps", 1)
    pair = 44 * 207.0   # 44 neighbours; volumes 27, gradients 70, density and div Q 48, momentum 62 flops each
    sg = 2.0 * (32 * 128 + 128 * 32 + 160 * 128 + 128 * 32 + 160 * 128 + 128 * 4)   # flops a row, forward
    if kind in ("step", "ensemble"):
        return {"bytes": n * (88.0 * s + 44), "flops": n * s * pair}
    if kind == "roundtrip":
        return {"bytes": n * 88.0, "flops": n * pair}
    if kind == "train":   # state 36 B, tendencies 32 B, targets 16 B in; gradients out
        return {"bytes": n * 84.0 + 4 * 54148, "flops": n * (3 * sg + 21 * 2 * 2 * (16 + 32 + 32))}
    if kind == "cycle":
        return {"bytes": n * (176.0 + 44), "flops": n * (pair + sg + 44 * 40.0 + 21 * 2 * (16 + 32 + 32))}
    M = case["grid"]
    return {"bytes": n * 32.0 + 9.0 * M * M, "flops": n * 44 * 27.0 + M * M * (44 * 32.0 + 20 * math.log2(M))}


# ------------------------------------------------------------------------------------------------
# exact: the method in FP64 torch
# ------------------------------------------------------------------------------------------------

CHUNK_PAIRS = 1 << 26


def _neighbours(pos, L, R, chunk_pairs=CHUNK_PAIRS):
    """Dense neighbour rows of particles in a periodic box: (n, K) int64 indices, -1 where absent, of
    every other particle closer than R (minimum image)."""
    d, n = len(pos), pos[0].numel()
    nc = int(math.floor(L / R))
    cell = [torch.clamp((p * (nc / L)).long(), 0, nc - 1) for p in pos]
    key = cell[0]
    for k in range(1, d):
        key = key + cell[k] * nc ** k
    order = torch.argsort(key)
    cnt = torch.bincount(key, minlength=nc ** d)
    start = torch.cumsum(cnt, 0) - cnt
    m = int(cnt.max())
    off = torch.cartesian_prod(*[torch.arange(-1, 2, device=DEV)] * d)
    rows = max(1, chunk_pairs // (off.shape[0] * m))
    lists, width = [], 0
    for a in range(0, n, rows):
        i = torch.arange(a, min(n, a + rows), device=DEV)
        c = sum(((cell[k][i][:, None] + off[None, :, k]) % nc) * nc ** k for k in range(d))
        slot = torch.arange(m, device=DEV)
        j = (start[c][:, :, None] + slot).reshape(i.numel(), -1)
        ok = (slot < cnt[c][:, :, None]).reshape(i.numel(), -1)
        j = order[torch.where(ok, j, torch.zeros_like(j))]
        r2 = torch.zeros(j.shape, dtype=torch.float64, device=DEV)
        for p in pos:
            e = p[i][:, None] - p[j]
            e = torch.where(e > 0.5 * L, e - L, torch.where(e < -0.5 * L, e + L, e))
            r2 = r2 + e * e
        ok &= (r2 < R * R) & (j != i[:, None])
        at = torch.cumsum(ok, 1) - 1
        w = int(ok.sum(1).max())
        row = torch.full((i.numel(), w + 1), -1, dtype=torch.int64, device=DEV)
        row.scatter_(1, torch.where(ok, at, torch.full_like(at, w)), j)
        lists.append(row[:, :w])
        width = max(width, w)
    return torch.cat([torch.nn.functional.pad(r, (0, width - r.shape[1]), value=-1) for r in lists])


class _Pairs:
    """Geometry of the neighbour rows of particles i0 .. i1: d = x_i - x_j, r, and the kernel."""

    def __init__(self, pos, nbr, i0, i1, L, h, ad):
        self.i = slice(i0, i1)
        j = nbr[i0:i1]
        self.on = j >= 0
        self.j = torch.where(self.on, j, torch.zeros_like(j))
        self.d = []
        for p in pos:
            e = p[i0:i1, None] - p[self.j]
            e = torch.where(e > 0.5 * L, e - L, torch.where(e < -0.5 * L, e + L, e))
            self.d.append(torch.where(self.on, e, torch.ones_like(e)))
        self.r = torch.sqrt(sum(e * e for e in self.d))
        b = self.r / h
        t3, t2, t1 = (torch.clamp(k - b, min=0.0) for k in (3.0, 2.0, 1.0))
        zero = torch.zeros_like(b)
        self.W = torch.where(self.on, ad * (t3 ** 5 - 6 * t2 ** 5 + 15 * t1 ** 5), zero)
        self.F = torch.where(self.on, ad / h * (-5 * t3 ** 4 + 30 * t2 ** 4 - 75 * t1 ** 4) / self.r, zero)

    def of(self, f):   # f_j
        return f[self.j]

    def diff(self, f):   # f_j - f_i
        return f[self.j] - f[self.i, None]


def _chunks(n, nbr):
    step = max(1, CHUNK_PAIRS // (4 * max(1, nbr.shape[1])))
    return [(a, min(n, a + step)) for a in range(0, n, step)]


def _wrap(x, L):
    x = torch.where(x < 0, x + L, x)
    return torch.where(x >= L, x - L, x)


def _inv2(a11, a12, a22):
    det = a11 * a22 - a12 * a12
    return a22 / det, -a12 / det, a11 / det


def _step2(p, S, rec=None):
    """One 2D step in FP64 (predictor, volumes, gradients and Q rate, density and pressure,
    momentum, displacement, corrector).  rec: receives the recorded tendencies."""
    L, h, dt, n = 1.0, p["h"], p["dt"], S["X"].numel()
    rho0, Gam, lam, C, gam, c = 1.0, 0.34, 0.7, 1.0, 7.0, 1.0 / 3.0
    nu, K, zeta = p["eta"], p["K"], p["zeta"]
    cons = p.get("momentum_mode", 0) == 1
    ad = 7.0 / (478.0 * math.pi * h * h)
    W0 = 66.0 * ad
    ux, uy = S["UX"] + 0.5 * dt * S["AX"], S["UY"] + 0.5 * dt * S["AY"]
    x, y = _wrap(S["X"] + 0.5 * dt * ux, L), _wrap(S["Y"] + 0.5 * dt * uy, L)
    q1, q2, dr = S["Q11"], S["Q12"], S["DRHO"]
    nbr = _neighbours((x, y), L, 3.0 * h)
    parts = _chunks(n, nbr)
    new = lambda: torch.empty(n, dtype=torch.float64, device=DEV)   # noqa: E731
    sumW = new()
    for a, b in parts:
        sumW[a:b] = W0 + _Pairs((x, y), nbr, a, b, L, h, ad).W.sum(1)
    V = 1.0 / sumW
    B11, B12, B22, kr, dh, Q1, Q2 = (new() for _ in range(7))
    m1s, m2s, l1s, l2s, dv, vo = (new() for _ in range(6)) if rec is not None else [None] * 6
    for a, b in parts:
        g = _Pairs((x, y), nbr, a, b, L, h, ad)
        dx, dy = g.d
        vf = g.of(V) * g.F
        gx, gy = vf * dx, vf * dy
        b11, b12, b22 = _inv2(-(gx * dx).sum(1), -(gx * dy).sum(1), -(gy * dy).sum(1))
        dux, duy = g.diff(ux), g.diff(uy)
        l00, l01, l10, l11 = (dux * gx).sum(1), (dux * gy).sum(1), (duy * gx).sum(1), (duy * gy).sum(1)
        D00, D01, D10, D11 = l00 * b11 + l01 * b12, l00 * b12 + l01 * b22, l10 * b11 + l11 * b12, l10 * b12 + l11 * b22
        div = D00 + D11
        w = vf / (g.r * g.r)
        lap = []
        for q in (q1, q2):
            e = -g.diff(q) * w
            lap.append(2.0 * (b11 * (e * dx * dx).sum(1) + 2.0 * b12 * (e * dx * dy).sum(1) + b22 * (e * dy * dy).sum(1)))
        s1, s2 = q1[a:b], q2[a:b]
        E12, om = 0.5 * (D01 + D10), 0.5 * (D10 - D01)
        QE = s1 * (D00 - D11) + 2.0 * s2 * E12
        hb = -C * 2.0 * (s1 * s1 + s2 * s2)
        H1, H2 = hb * s1 + K * lap[0], hb * s2 + K * lap[1]
        m1 = lam * div * s1 + c * lam * (D00 - D11) - 2.0 * om * s2 - 2.0 * lam * QE * s1 + Gam * H1
        m2 = lam * div * s2 + 2.0 * c * lam * E12 + 2.0 * om * s1 - 2.0 * lam * QE * s2 + Gam * H2
        B11[a:b], B12[a:b], B22[a:b] = b11, b12, b22
        kr[a:b] = -(1.0 + dr[a:b]) * div
        dh[a:b] = dr[a:b] + 0.5 * dt * kr[a:b]
        Q1[a:b], Q2[a:b] = s1 + dt * m1, s2 + dt * m2
        if rec is not None:
            m1s[a:b], m2s[a:b], l1s[a:b], l2s[a:b], dv[a:b], vo[a:b] = m1, m2, lap[0], lap[1], div, D10 - D01
    c0 = max(10.0 * float(torch.sqrt((ux * ux + uy * uy).max())), p.get("c0_min", 0.0))
    dhat, fx, fy = new(), new(), new()
    for a, b in parts:
        g = _Pairs((x, y), nbr, a, b, L, h, ad)
        dhat[a:b] = dh[a:b] + (g.diff(dh) * g.W).sum(1) / sumW[a:b]
        if not cons:
            vf = g.of(V) * g.F
            gx, gy = vf * g.d[0], vf * g.d[1]
            bx, by = B11[a:b, None] * gx + B12[a:b, None] * gy, B12[a:b, None] * gx + B22[a:b, None] * gy
            d1, d2 = g.diff(Q1), g.diff(Q2)
            fx[a:b] = -zeta * (d1 * bx + d2 * by).sum(1)
            fy[a:b] = -zeta * (d2 * bx - d1 * by).sum(1)
    rho = rho0 * (1.0 + dhat)
    pr = rho0 * c0 * c0 / gam * torch.expm1(gam * torch.log1p(dhat)) / (rho * rho)
    out = {k: new() for k in B.FULL_STATE}
    for a, b in parts:
        g = _Pairs((x, y), nbr, a, b, L, h, ad)
        dx, dy = g.d
        dux, duy = -g.diff(ux), -g.diff(uy)
        visc = 8.0 * nu * (dux * dx + duy * dy) / (g.r * g.r)
        ri = rho[a:b]
        if cons:
            rj = g.of(rho)
            s = (visc * rho0 / (ri[:, None] * rj) - (pr[a:b, None] + g.of(pr))) * g.F
            t1, t2 = ((q[a:b] / (ri * ri))[:, None] + g.of(q) / (rj * rj) for q in (Q1, Q2))
            ax = (s * dx - zeta * g.F * (t1 * dx + t2 * dy)).sum(1)
            ay = (s * dy - zeta * g.F * (t2 * dx - t1 * dy)).sum(1)
            ax, ay = ax * rho0 * L * L / n, ay * rho0 * L * L / n
        else:
            s = g.of(V) * g.F * (visc * (rho0 / ri)[:, None] - ri[:, None] * (pr[a:b, None] + g.of(pr)))
            wx, wy = (s * dx).sum(1), (s * dy).sum(1)
            ax = B11[a:b] * wx + B12[a:b] * wy + fx[a:b] / ri
            ay = B12[a:b] * wx + B22[a:b] * wy + fy[a:b] / ri
        su, sv = (dux * g.W).sum(1), (duy * g.W).sum(1)
        on = g.on.double()
        r0 = (g.r * on).sum(1) / on.sum(1)
        sc = dt * torch.sqrt(su * su + sv * sv) / sumW[a:b] * r0 * r0
        ir3 = on / g.r ** 3
        vx, vy = ux[a:b] + 0.5 * dt * ax, uy[a:b] + 0.5 * dt * ay
        out["AX"][a:b], out["AY"][a:b], out["UX"][a:b], out["UY"][a:b] = ax, ay, vx, vy
        out["X"][a:b] = _wrap(x[a:b] + 0.5 * dt * vx + sc * (dx * ir3).sum(1), L)
        out["Y"][a:b] = _wrap(y[a:b] + 0.5 * dt * vy + sc * (dy * ir3).sum(1), L)
    out["Q11"], out["Q12"], out["DRHO"] = Q1, Q2, dhat + 0.5 * dt * kr
    if rec is not None:
        rec.update(tend=torch.stack([out["AX"], out["AY"], m1s, m2s, l1s, l2s, dv, vo], 1))
    return out


def _start2(ic):
    S = {k: v.float().double() if k not in "XY" else v for k, v in ic.items()}   # as the context stores it
    for f in ("DRHO", "AX", "AY"):
        S[f] = torch.zeros_like(S["X"])
    return S


def _run2(case, side, ic, steps, prm=None):
    p = dict(_params2(case, side) if prm is None else prm)
    p["dt"] = 1e-4 if case.get("dt_check") else B_dt({"eta": p["eta"], "K": p["K"]}, side)
    S = _start2(ic)
    for _ in range(steps):
        S = _step2(p, S)
    return S


def _q3(q):
    z = -q[:, 0] - q[:, 3]
    return torch.stack([q[:, 0], q[:, 1], q[:, 2], q[:, 1], q[:, 3], q[:, 4], q[:, 2], q[:, 4], z], 1).reshape(-1, 3, 3)


def _step3(p, S):
    """One 3D step in FP64."""
    L, h, dt, n = 1.0, p["h"], p["dt"], S["x"][0].numel()
    rho0, Gam, lam, C, K, gam, c = 1.0, 0.34, 0.7, 1.0, 0.04, 7.0, 1.0 / 3.0
    ad = 3.0 / (359.0 * math.pi * h ** 3)
    W0 = 66.0 * ad
    u = [S["u"][k] + 0.5 * dt * S["a"][k] for k in range(3)]
    x = [_wrap(S["x"][k] + 0.5 * dt * u[k], L) for k in range(3)]
    q, dr = S["q"], S["dr"]
    nbr = _neighbours(x, L, 3.0 * h)
    parts = _chunks(n, nbr)
    new = lambda *s: torch.empty((n,) + s, dtype=torch.float64, device=DEV)   # noqa: E731
    sumW = new()
    for a, b in parts:
        sumW[a:b] = W0 + _Pairs(x, nbr, a, b, L, h, ad).W.sum(1)
    V = 1.0 / sumW
    Bm, kr, dh, qn = new(3, 3), new(), new(), new(5)
    for a, b in parts:
        g = _Pairs(x, nbr, a, b, L, h, ad)
        vf = g.of(V) * g.F
        e = [vf * g.d[k] for k in range(3)]
        al = torch.stack([-(e[i] * g.d[k]).sum(1) for i in range(3) for k in range(3)], 1).reshape(-1, 3, 3)
        Bi = torch.linalg.inv(al)
        du = [g.diff(u[k]) for k in range(3)]
        rhs = torch.stack([(du[i] * e[k]).sum(1) for i in range(3) for k in range(3)], 1).reshape(-1, 3, 3)
        D = rhs @ Bi
        kr[a:b] = -(1.0 + dr[a:b]) * (Bi * rhs).sum((1, 2))
        dh[a:b] = dr[a:b] + 0.5 * dt * kr[a:b]
        ir2 = 1.0 / (g.r * g.r)
        bd = sum(e[i] * Bi[:, i, k, None] * g.d[k] for i in range(3) for k in range(3)) * ir2
        lap = torch.stack([-2.0 * (bd * g.diff(q[:, k].contiguous())).sum(1) for k in range(5)], 1)
        Q, LQ = _q3(q[a:b]), _q3(lap)
        E, Om = 0.5 * (D + D.transpose(1, 2)), 0.5 * (D - D.transpose(1, 2))
        I = torch.eye(3, dtype=torch.float64, device=DEV)
        M = Q + c * I
        Q2 = Q @ Q
        tr2 = Q2.diagonal(dim1=1, dim2=2).sum(1)[:, None, None]
        H = -p["A"] * Q + p["B"] * (Q2 - tr2 / 3.0 * I) - C * Q * tr2 + K * LQ
        m = (lam * E + Om) @ M + M @ (lam * E - Om) - 2.0 * lam * M * (Q * D).sum((1, 2))[:, None, None] + Gam * H
        m = 0.5 * (m + m.transpose(1, 2)) - m.diagonal(dim1=1, dim2=2).sum(1)[:, None, None] / 3.0 * I
        m5 = torch.stack([m[:, 0, 0], m[:, 0, 1], m[:, 0, 2], m[:, 1, 1], m[:, 1, 2]], 1)
        Bm[a:b], qn[a:b] = Bi, q[a:b] + dt * m5
    c0 = max(10.0 * float(torch.sqrt(sum(v * v for v in u).max())), p["c0_min"])
    dhat = new()
    for a, b in parts:
        g = _Pairs(x, nbr, a, b, L, h, ad)
        dhat[a:b] = dh[a:b] + (g.diff(dh) * g.W).sum(1) / sumW[a:b]
    rho = rho0 * (1.0 + dhat)
    pr = rho0 * c0 * c0 / gam * torch.expm1(gam * torch.log1p(dhat)) / (rho * rho)
    nx, nu_, na = [new() for _ in range(3)], [new() for _ in range(3)], [new() for _ in range(3)]
    idx = ((0, 1, 2), (1, 3, 4), (2, 4, None))
    for a, b in parts:
        g = _Pairs(x, nbr, a, b, L, h, ad)
        Bi, ri = Bm[a:b], rho[a:b]
        vf = g.of(V) * g.F
        bd = [sum(Bi[:, i, k, None] * g.d[k] for k in range(3)) for i in range(3)]
        du = [-g.diff(u[k]) for k in range(3)]
        ud = sum(du[k] * g.d[k] for k in range(3))
        s = vf * (10.0 * p["eta"] * rho0 / ri[:, None] * ud / (g.r * g.r) - ri[:, None] * (pr[a:b, None] + g.of(pr)))
        dq = [g.diff(qn[:, k].contiguous()) for k in range(5)]
        dq.append(-dq[0] - dq[3])
        on = g.on.double()
        ir3 = on / g.r ** 3
        r0 = (g.r * on).sum(1) / on.sum(1)
        su = [(du[k] * g.W).sum(1) for k in range(3)]
        uv = torch.sqrt(sum(v * v for v in su)) / sumW[a:b]
        for i in range(3):
            dv = (vf * sum(dq[5 if idx[i][k] is None else idx[i][k]] * bd[k] for k in range(3))).sum(1)
            an = (s * bd[i]).sum(1) - p["zeta"] / ri * dv
            un = u[i][a:b] + 0.5 * dt * an
            na[i][a:b], nu_[i][a:b] = an, un
            nx[i][a:b] = _wrap(x[i][a:b] + 0.5 * dt * un + (g.d[i] * ir3).sum(1) * r0 * r0 * uv * dt, L)
    return {"x": nx, "u": nu_, "a": na, "q": qn, "dr": dhat + 0.5 * dt * kr}


def _mean_rows(x, y, h, radius):
    """Rows of the SPH mean: (neighbours within radius h, their weights / S, the own weight / S)."""
    ad = 7.0 / (478.0 * math.pi * h * h)
    nbr = _neighbours((x, y), 1.0, radius * h) if radius == 3.0 else None
    if nbr is None:   # closer than 2h, among the support's
        full = _neighbours((x, y), 1.0, 3.0 * h)
        g = _Pairs((x, y), full, 0, x.numel(), 1.0, h, ad)
        W, on = torch.where(g.r < radius * h, g.W, torch.zeros_like(g.W)), g.on & (g.r < radius * h)
        k = int(on.sum(1).max())
        at = torch.argsort((~on).to(torch.int8), dim=1, stable=True)[:, :k]
        j, W = torch.gather(g.j, 1, at), torch.gather(W * on, 1, at)
    else:
        g = _Pairs((x, y), nbr, 0, x.numel(), 1.0, h, ad)
        j, W = g.j, g.W
    S = 66.0 * ad + W.sum(1)
    return j, W / S[:, None], 66.0 * ad / S


def _agg(rows, f):
    """SPH mean of f (n, c): chunks of rows, each channel block summed over the neighbours."""
    j, w, w0 = rows
    out = [(w[a:a + 65536, :, None] * f[j[a:a + 65536]]).sum(1) for a in range(0, f.shape[0], 65536)]
    return w0[:, None] * f + torch.cat(out)


def _unflatten(flat):
    out, at = {}, 0
    for name, shape in SG_SHAPES:
        size = int(np.prod(shape))
        out[name] = flat[at:at + size].reshape(shape)
        at += size
    return out


def _network(w, g2, x):
    relu = torch.relu
    h1 = relu(torch.cat([x, _agg(g2, x)], 1) @ w["W1"].T + w["b1"])
    h2 = relu(torch.cat([h1, _agg(g2, h1 @ w["P1"].T)], 1) @ w["W2"].T + w["b2"])
    h3 = relu(torch.cat([h2, _agg(g2, h2 @ w["P2"].T)], 1) @ w["W3"].T + w["b3"])
    return h3 @ w["Wo"].T + w["bo"]


def _features(g3, S, tend, kdt, ysq, ysu):
    r = torch.stack([S["Q11"], S["Q12"], S["UX"] / SG_US, S["UY"] / SG_US], 1)
    gk = 0.34 * 0.02
    size = torch.tensor([kdt / ysu] * 2 + [kdt / ysq] * 2 + [gk * kdt / ysq] * 2 + [kdt] * 2,
                        dtype=torch.float64, device=DEV)
    return torch.cat([r, _agg(g3, r) - r, tend * size], 1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        parts = [_run2({}, s, _inputs2(s, seed, k + 1), case["steps"], p) for k, (s, p) in enumerate(_members(case))]
        return {f: torch.cat([q[f] for q in parts]) for f in STATE}
    if kind == "step3":
        side, p = case["side"], _params3(case["side"])
        if side ** 3 * case["steps"] > 1.1e7:
            return None
        ic = _inputs3(side, seed)
        zero = torch.zeros_like(ic["x"])
        S = {"x": [ic["x"], ic["y"], ic["z"]], "u": list(ic["u"].float().double().T.contiguous()), "a": [zero] * 3,
             "q": ic["q"].float().double(), "dr": zero}
        for _ in range(case["steps"]):
            S = _step3(p, S)
        return {"pos": torch.stack(S["x"], 1), "u": torch.stack(S["u"], 1), "q": S["q"]}
    side = case["side"]
    if kind == "step":
        if side * side * case["steps"] > 4e7:
            return None
        S = _run2(case, side, _inputs2(side, seed), case["steps"])
        return {f: S[f] for f in STATE}
    if kind == "roundtrip":
        return _run2(case, side, _inputs2(side, seed), 1)
    h, kdt = HOVER / side, SG_K * B_dt(case, side)
    if kind == "train":
        if side > 400:
            return None
        st, tend, target = _snapshot_pair(case, seed)
        S = {k: v.double() for k, v in st.items()}
        g3, g2 = _mean_rows(S["X"], S["Y"], h, 3.0), _mean_rows(S["X"], S["Y"], h, 2.0)
        flat = torch.from_numpy(_weights(seed)).to(DEV).double().requires_grad_(True)
        y = _network(_unflatten(flat), g2, _features(g3, S, tend.double(), kdt, SG_YSQ, SG_YSU))
        loss = ((y - target.double()) ** 2).mean()
        loss.backward()
        return {"loss": float(loss.detach()), "grads": flat.grad.detach()}
    if kind == "cycle":
        if side > 1100:
            return None
        p = dict(_params2(case, side), dt=B_dt(case, side))
        rec = {}
        S = _step2(p, _start2(_inputs2(side, seed)), rec)
        g3 = _mean_rows(S["X"], S["Y"], h, 3.0)
        tend = rec["tend"]
        x = _features(g3, S, tend, kdt, SG_YS_CYCLE, SG_YS_CYCLE)
        sm = _agg(g3, _agg(g3, tend[:, :2].contiguous()))
        del g3
        with torch.no_grad():
            w = _unflatten(torch.from_numpy(_weights(seed)).to(DEV).double())
            y = _network(w, _mean_rows(S["X"], S["Y"], h, 2.0), x)
        out = dict(S, Q11=S["Q11"] + kdt * tend[:, 2] + SG_YS_CYCLE * y[:, 0],
                   Q12=S["Q12"] + kdt * tend[:, 3] + SG_YS_CYCLE * y[:, 1],
                   UX=S["UX"] + kdt * sm[:, 0], UY=S["UY"] + kdt * sm[:, 1])
        out["X"] = torch.remainder(S["X"] + 0.5 * kdt * (S["UX"] + out["UX"]), 1.0)
        out["Y"] = torch.remainder(S["Y"] + 0.5 * kdt * (S["UY"] + out["UY"]), 1.0)
        return {f: out[f] for f in STATE}
    return _analysis(case, seed)


def _analysis(case, seed):
    side, M = case["side"], case["grid"]
    ic = {k: v.float().double() if k not in "XY" else v for k, v in _inputs2(side, seed).items()}
    h, R = HOVER / side, 3.0 * HOVER / side
    ad, nc = 7.0 / (478.0 * math.pi * h * h), int(math.floor(side / (3.0 * HOVER)))
    pos = [ic["X"], ic["Y"]]
    key = sum(torch.clamp((p * nc).long(), 0, nc - 1) * nc ** k for k, p in enumerate(pos))
    order = torch.argsort(key)
    cnt = torch.bincount(key, minlength=nc * nc)
    start, m = torch.cumsum(cnt, 0) - cnt, int(cnt.max())
    off = torch.cartesian_prod(*[torch.arange(-1, 2, device=DEV)] * 2)
    fields = [ic["UX"], ic["UY"], ic["Q11"], ic["Q12"]]
    grid = [torch.zeros(M * M, dtype=torch.float64, device=DEV) for _ in range(4)]
    rows = max(1, CHUNK_PAIRS // (9 * m))
    for a in range(0, M * M, rows):
        g = torch.arange(a, min(M * M, a + rows), device=DEV)
        node = [(g % M).double() / M, (g // M).double() / M]
        cell = [torch.clamp((v * nc).long(), 0, nc - 1) for v in node]
        c = sum(((cell[k][:, None] + off[None, :, k]) % nc) * nc ** k for k in range(2))
        slot = torch.arange(m, device=DEV)
        ok = (slot < cnt[c][:, :, None]).reshape(g.numel(), -1)
        j = (start[c][:, :, None] + slot).reshape(g.numel(), -1)
        j = order[torch.where(ok, j, torch.zeros_like(j))]
        r2 = 0.0
        for v, p in zip(node, pos):
            e = v[:, None] - p[j]
            e = e - torch.round(e)
            r2 = r2 + e * e
        b = torch.sqrt(r2) / h
        t3, t2, t1 = (torch.clamp(k - b, min=0.0) for k in (3.0, 2.0, 1.0))
        W = torch.where(ok & (r2 < R * R), ad * (t3 ** 5 - 6 * t2 ** 5 + 15 * t1 ** 5), torch.zeros_like(r2))
        s = W.sum(1)
        for f, o in zip(fields, grid):
            o[a:a + g.numel()] = (W * f[j]).sum(1) / s
    ux, uy = grid[0].reshape(M, M), grid[1].reshape(M, M)
    e = sum(0.5 * (torch.fft.fft2(v) / (M * M)).abs() ** 2 for v in (ux, uy))
    k = torch.round(torch.fft.fftfreq(M, d=1.0 / M, dtype=torch.float64, device=DEV))
    shell = torch.round(torch.sqrt(k[:, None] ** 2 + k[None, :] ** 2)).long()
    E = torch.bincount(shell.reshape(-1), weights=e.reshape(-1), minlength=int(round(M / math.sqrt(2.0))) + 1)
    j0 = M // 2
    om = ((torch.roll(uy[j0], -1) - torch.roll(uy[j0], 1)) - (ux[(j0 + 1) % M] - ux[j0 - 1])) / (2.0 / M)
    C = torch.stack([(torch.roll(om, -s) * om).sum() for s in range(M // 2 + 1)]) / (om * om).sum()
    return {"E": E, "C": C, "counts": None, "map": None}
