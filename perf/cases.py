"""The calls that a user of the library makes, as cases to time.

A pass of a stepping case takes a particle state in (device pointers, or host
arrays), advances it by a few real steps, and reads the whole state back in the
caller's particle order: positions, velocities, pressures and the previous
velocities. Contexts are created once and kept, as a program that advances many
states does. The rate cases call the allocation-free rate evaluation.

The states are those that such runs start from or pass through: jittered
lattices with the fields of the flow, drawn from the seed. The FP32C path keeps
its pair sums in single precision, so a program that chose it keeps the fields
as float32; the FP64 path's fields stay float64.

``exact`` is the method itself (Algorithm 2 of arXiv:1904.00861, Algorithm 1 for
particles moving in pseudo-time) in plain FP64 torch operations.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1904_00861_gb300 as dt

# Pseudo-time iterations per real step, as these flows take them at the start of
# a run (they set the operation counts of work(), nothing else).
_ITERS = {"tgv2": 14, "tgv3": 7, "cavity": 18, "dambreak": 50, "batch": 14, "moving": 13}


def listed():
    return [
        # The rates at one small state: a solver of another kind calling the pair
        # sums inside its own loop, where the call's latency counts.
        dict(name="rates-2d-32-fp64", family="rates", dim=2, side=32, fp64=True),
        # The same in 3D near the entry point's largest size, single precision.
        dict(name="rates-3d-23-fp32c", family="rates", dim=3, side=23, fp64=False),
        # The small validation run: 50 x 50 vortex, FP64, host arrays in and out.
        dict(name="tgv2d-50-fp64-host", family="tgv", dim=2, side=50, fp64=True, steps=10, skin=0.0, moving=0, host=True),
        # The 200 x 200 vortex on the fast path, lists reused between steps.
        dict(name="tgv2d-200-fp32c", family="tgv", dim=2, side=200, fp64=False, steps=10, skin=0.05, moving=0, host=False),
        # The same problem on the reference precision.
        dict(name="tgv2d-200-fp64", family="tgv", dim=2, side=200, fp64=True, steps=3, skin=0.0, moving=0, host=False),
        # Lid-driven cavity: walls, shifting after every step.
        dict(name="cavity-200-fp32c", family="cavity", side=200, fp64=False, steps=5, re=100.0),
        # A falling column with a free surface, walls, artificial viscosity and
        # shifting; an odd lattice.
        dict(name="dambreak-101-fp32c", family="dambreak", side=101, fp64=False, steps=5),
        # The ensemble: independent vortices of uneven sizes and Reynolds numbers
        # in one context, new states from host arrays.
        dict(name="batch-64-fp32c", family="batch", count=64, lo=32, hi=256, fp64=False, steps=3, skin=0.05),
        # Particles moving in pseudo-time with neighbour updates (the method's
        # other algorithm); an odd lattice.
        dict(name="moving-151-fp32c", family="tgv", dim=2, side=151, fp64=False, steps=3, skin=0.0, moving=2, host=False),
        # 3D on the reference precision, a ragged size.
        dict(name="tgv3d-45-fp64", family="tgv", dim=3, side=45, fp64=True, steps=2, skin=0.0, moving=0, host=False),
        # A mid-size 3D vortex with two list builds per step (the library's default).
        dict(name="tgv3d-61-fp32c", family="tgv", dim=3, side=61, fp64=False, steps=3, skin=0.0, moving=0, host=False),
        # The largest: 128^3 particles.
        dict(name="tgv3d-128-fp32c", family="tgv", dim=3, side=128, fp64=False, steps=2, skin=0.05, moving=0, host=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["rates", "tgv2", "tgv2", "tgv2", "tgv3", "tgv3", "cavity", "dambreak", "batch", "moving"])
    fp64 = rng.random() < 0.4
    if kind == "rates":
        dim = rng.choice([2, 3])
        side = _log(rng, 16, 127) if dim == 2 else _log(rng, 10, 25)
        return dict(family="rates", dim=dim, side=side, fp64=fp64)
    if kind == "tgv2":
        host = rng.random() < 0.3
        return dict(family="tgv", dim=2, side=_log(rng, 24, 240 if fp64 else 700), fp64=fp64, steps=rng.randint(1, 3 if fp64 else 6),
                    skin=rng.choice([0.0, 0.05]), moving=0, host=host)
    if kind == "tgv3":
        return dict(family="tgv", dim=3, side=_log(rng, 16, 48 if fp64 else 110), fp64=fp64, steps=rng.randint(1, 2),
                    skin=rng.choice([0.0, 0.05]), moving=0, host=False)
    if kind == "cavity":
        return dict(family="cavity", side=_log(rng, 32, 120 if fp64 else 260), fp64=fp64, steps=rng.randint(2, 4),
                    re=rng.choice([100.0, 1000.0]))
    if kind == "dambreak":
        return dict(family="dambreak", side=_log(rng, 20, 80 if fp64 else 220), fp64=fp64, steps=rng.randint(2, 5))
    if kind == "batch":
        return dict(family="batch", count=rng.randint(3, 64), lo=32, hi=rng.randint(64, 128 if fp64 else 256), fp64=fp64,
                    steps=1 if fp64 else 2, skin=rng.choice([0.0, 0.05]))
    return dict(family="tgv", dim=2, side=_log(rng, 24, 100 if fp64 else 250), fp64=fp64, steps=rng.randint(1, 3), skin=0.0,
                moving=rng.choice([1, 2]), host=False)


# ------------------------------------------------------------------- inputs

def _params(dim, dx, U, nu, **kw):
    d = dict(dim=dim, h=dx, m=dx ** dim, rho0=1.0, beta=10.0, v_ref=U, nu=nu, dt=0.25 * dx / U, eta=0.01, alpha=0.0,
             g=(0.0, 0.0, 0.0), eps=1e-3, stag_tol=0.05, stag_window=4, max_iter=1000, edac=1, shifting=0,
             free_surface=0, moving=0, skin=0.0, list_skin=0.0)
    d.update(kw)
    return d


def _lattice(dims, gen):
    """Lattice indices (first axis fastest) and uniform [-1, 1) draws per axis."""
    ax = [torch.arange(n, dtype=torch.float64, device="cuda") for n in dims]
    grid = torch.meshgrid(*ax[::-1], indexing="ij")
    idx = torch.stack([g.reshape(-1) for g in grid[::-1]], 1)
    r = 2.0 * torch.rand(idx.shape, dtype=torch.float64, device="cuda", generator=gen) - 1.0
    return idx, r


def _vortex(dim, side, re, gen):
    """Taylor-Green vortex on a jittered periodic lattice: the unit square, or
    [0, 2 pi)^3."""
    L = 1.0 if dim == 2 else 2.0 * math.pi
    dx = L / side
    cfg = _params(dim, dx, 1.0, 1.0 / re, periodic=(1, 1, 1 if dim == 3 else 0), lo=(0.0,) * 3,
                  hi=(L, L, L if dim == 3 else 1.0))
    idx, r = _lattice((side,) * dim, gen)
    x = torch.remainder((idx + 0.5) * dx + (0.1 if dim == 2 else 0.05) * dx * r, L)
    # the vortex at a random phase (the same flow elsewhere in the box)
    ph = 2.0 * math.pi * torch.rand(dim, dtype=torch.float64, device="cuda", generator=gen)
    if dim == 2:
        def field(t):
            e = math.exp(-8.0 * math.pi ** 2 / re * t)
            a, b = 2.0 * math.pi * x[:, 0] + ph[0], 2.0 * math.pi * x[:, 1] + ph[1]
            v = torch.stack([-e * torch.cos(a) * torch.sin(b), e * torch.sin(a) * torch.cos(b)], 1)
            return v, -e * e * (torch.cos(2 * a) + torch.cos(2 * b)) / 4.0
        v, p = field(0.0)
        vp, _ = field(-cfg["dt"])
    else:
        a, b, c = x[:, 0] + ph[0], x[:, 1] + ph[1], x[:, 2] + ph[2]
        v = torch.stack([torch.sin(a) * torch.cos(b) * torch.cos(c), -torch.cos(a) * torch.sin(b) * torch.cos(c),
                         torch.zeros_like(a)], 1)
        p = (torch.cos(2 * a) + torch.cos(2 * b)) * (torch.cos(2 * c) + 2.0) / 16.0
        vp = v.clone()
    return cfg, x.contiguous(), v.contiguous(), p.contiguous(), vp.contiguous()


def _walls_around(nx, ny, layers, left, right, bottom, top, dx):
    i, j = np.meshgrid(np.arange(-layers, nx + layers), np.arange(-layers, ny + (layers if top else 0)))
    wall = (j < 0) | (top & (j >= ny)) | (left & (i < 0)) | (right & (i >= nx))
    return np.stack([(i[wall] + 0.5) * dx, (j[wall] + 0.5) * dx], 1)


def _cavity(side, re, gen):
    """A lid-driven cavity in mid-run: a recirculating flow under the lid."""
    dx, U = 1.0 / side, 1.0
    cfg = _params(2, dx, U, U / re, eps=1e-4, shifting=1, periodic=(0, 0, 0), lo=(-3 * dx, -3 * dx, 0.0),
                  hi=(1.0 + 3 * dx, 1.0 + 3 * dx, 1.0))
    idx, r = _lattice((side, side), gen)
    x = (idx + 0.5) * dx + 0.05 * dx * r
    amp = 0.1 + 0.05 * float(torch.rand(1, dtype=torch.float64, device="cuda", generator=gen))
    sx, sy = torch.sin(math.pi * x[:, 0]), torch.sin(math.pi * x[:, 1])
    cx, cy = torch.cos(math.pi * x[:, 0]), torch.cos(math.pi * x[:, 1])
    v = torch.stack([-2.0 * amp * sx * sx * sy * cy, 2.0 * amp * sx * cx * sy * sy], 1)
    p = 0.25 * amp * amp * (torch.cos(2 * math.pi * x[:, 0]) + torch.cos(2 * math.pi * x[:, 1]))
    xw = _walls_around(side, side, 3, True, True, True, True, dx)
    vw = np.zeros_like(xw)
    vw[xw[:, 1] > 1.0, 0] = U
    return cfg, x, v, p, v.clone(), xw, vw


def _dambreak(side, gen):
    """A 1 x 2 column in a 4 x 2.5 tank, released a moment ago."""
    dx, H, g = 1.0 / side, 2.0, 9.81
    U = math.sqrt(2.0 * g * H)
    cfg = _params(2, dx, U, 0.0, alpha=0.1, eps=1e-4, shifting=1, free_surface=1, g=(0.0, -g, 0.0),
                  periodic=(0, 0, 0), lo=(-3 * dx, -3 * dx, 0.0), hi=(4.0 + 3 * dx, 2.5, 1.0))
    idx, r = _lattice((side, 2 * side), gen)
    x = (idx + 0.5) * dx + 0.05 * dx * r
    t = 0.01 + 0.02 * float(torch.rand(1, dtype=torch.float64, device="cuda", generator=gen))
    v = torch.stack([g * t * x[:, 0] * (1.0 - 0.5 * x[:, 1]), -0.5 * g * t * x[:, 1] * x[:, 0]], 1)
    p = g * (H - x[:, 1])
    ny = int(math.floor(2.5 / dx - 0.5))
    xw = _walls_around(4 * side, ny, 3, True, True, True, False, dx)
    return cfg, x, v, p, v.clone(), xw, np.zeros_like(xw)


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & 0x7FFFFFFFFFFFFFFF)
    return g


def _inputs(case, seed):
    """(cfg, x, v, p, v_prev, walls or None) on the device."""
    gen = _gen(seed)
    f = case["family"]
    if f == "cavity":
        cfg, x, v, p, vp, xw, vw = _cavity(case["side"], case["re"], gen)
        return cfg, x, v, p, vp, (xw, vw)
    if f == "dambreak":
        cfg, x, v, p, vp, xw, vw = _dambreak(case["side"], gen)
        return cfg, x, v, p, vp, (xw, vw)
    re = (100.0 if case["dim"] == 2 else 1600.0)
    cfg, x, v, p, vp = _vortex(case["dim"], case["side"], re, gen)
    if f == "tgv":
        cfg["list_skin"] = case["skin"] * cfg["h"]
        cfg["moving"] = case["moving"]
        cfg["skin"] = 0.5 * cfg["h"] if case["moving"] == 2 else 0.0
    return cfg, x, v, p, vp, None


def _instances(case, seed):
    """The ensemble's (cfg, x, v, p, v_prev) per instance; the sides and Reynolds
    numbers belong to the case (a program keeps its shapes)."""
    shape = np.random.RandomState(861)
    sides = shape.randint(case["lo"], case["hi"] + 1, case["count"])
    res = 10.0 ** (2.0 + shape.rand(case["count"]))
    gen = _gen(seed)
    out = []
    for n, re in zip(sides, res):
        cfg, x, v, p, vp = _vortex(2, int(n), float(re), gen)
        cfg["list_skin"] = case["skin"] * cfg["h"]
        out.append((cfg, x, v, p, vp))
    return out


def _precision(case):
    return dt.DTSPH_FP64 if case["fp64"] else dt.DTSPH_FP32C


def _pinned(t):
    return t.cpu().pin_memory()


class _Owner:
    """A context, given back with the state that holds it."""

    def __init__(self, ctx):
        self.ctx = ctx

    def __del__(self):
        try:
            if self.ctx:
                dt.dtsph_destroy(self.ctx)
        except Exception:
            pass
        self.ctx = None


def prepare(case, seed):
    f = case["family"]
    if f == "batch":
        inst = _instances(case, seed)
        prm = [dt.make_params(i[0], precision=_precision(case), graph=2) for i in inst]
        own = _Owner(dt.dtsph_batch_create(prm))
        host = [_pinned(torch.cat([i[k] for i in inst])) for k in (1, 2, 3, 4)]
        nf = np.array([i[1].shape[0] for i in inst], np.int64)
        s = dict(case=case, own=own, nf=nf, host=[h.numpy() for h in host], keep=host)
        n, dim = int(nf.sum()), 2
        dt.dtsph_batch_set_particles(own.ctx, nf, *s["host"])
    else:
        cfg, x, v, p, vp, walls = _inputs(case, seed)
        n, dim = x.shape
        prm = dt.make_params(cfg, precision=_precision(case), graph=2)
        s = dict(case=case, dev=(x, v, p, vp), prm=prm, n=n)
        if f == "rates":
            s["ap"] = torch.empty(n, dtype=torch.float64, device="cuda")
            s["F"] = torch.empty(n, dim, dtype=torch.float64, device="cuda")
            return s
        s["own"] = own = _Owner(dt.dtsph_create(prm))
        if walls is not None:
            dt.dtsph_set_boundary(own.ctx, walls[0], walls[1])
        dt.dtsph_set_particles_device(own.ctx, n, x, v, p, vp)
        if case.get("host"):
            keep = [_pinned(t) for t in (x, v, p, vp)]
            out = [torch.empty_like(t).pin_memory() for t in keep]
            s.update(keep=(keep, out), host=[t.numpy() for t in keep], out=[t.numpy() for t in out])
    if not case.get("host"):
        s["out"] = [torch.empty(n, dim, dtype=torch.float64, device="cuda"), torch.empty(n, dim, dtype=torch.float64, device="cuda"),
                    torch.empty(n, dtype=torch.float64, device="cuda"), torch.empty(n, dim, dtype=torch.float64, device="cuda")]
    s["n"], s["dim"] = n, dim
    return s


_FIELDS = (dt.FIELD_POS, dt.FIELD_VEL, dt.FIELD_P, dt.FIELD_VEL_PREV)


def run(state):
    case = state["case"]
    if case["family"] == "rates":
        x, v, p, _ = state["dev"]
        dt.dtsph_eval_rates_noalloc(state["prm"], state["n"], x, v, p, state["ap"], state["F"])
        out = [state["ap"], state["F"]]
        return out if case["fp64"] else [t.float() for t in out]
    ctx = state["own"].ctx
    if case["family"] == "batch":
        dt.dtsph_batch_set_particles(ctx, state["nf"], *state["host"])
    elif case.get("host"):
        dt.dtsph_set_particles(ctx, *state["host"])
    else:
        dt.dtsph_set_particles_device(ctx, state["n"], *state["dev"])
    dt.dtsph_step(ctx, case["steps"])
    if case.get("host"):
        out = list(dt.dtsph_read_state(ctx, state["n"], state["dim"], out=state["out"]))
        return out if case["fp64"] else [a.astype(np.float32) for a in out]
    for f, t in zip(_FIELDS, state["out"]):
        dt.dtsph_read_field_device(ctx, f, t)
    return state["out"] if case["fp64"] else [t.float() for t in state["out"]]


# --------------------------------------------------------------------- work

def _shape(case):
    """(dim, fluid particles, iterations per step) of a case."""
    f = case["family"]
    if f == "batch":
        sides = np.random.RandomState(861).randint(case["lo"], case["hi"] + 1, case["count"])
        return 2, int((sides.astype(np.int64) ** 2).sum()), _ITERS["batch"]
    if f == "cavity":
        return 2, case["side"] ** 2, _ITERS["cavity"]
    if f == "dambreak":
        return 2, 2 * case["side"] ** 2, _ITERS["dambreak"]
    d = case["dim"]
    return d, case["side"] ** d, 0 if f == "rates" else _ITERS["moving" if case["moving"] else "tgv%d" % d]


def work(case):
    d, n, iters = _shape(case)
    pairs = n * (9.0 * math.pi - 1.0 if d == 2 else 36.0 * math.pi - 1.0)
    geo = 25.0 + 2.0 * d                 # separation, kernel gradient and F_ij of a pair
    rate = 8.0 * d + 9.0                 # the two rates' terms of a pair
    if case["family"] == "rates":
        return {"bytes": 8.0 * n * (2 * d + 1 + d + 1), "flops": pairs * (geo + rate)}
    per_iter = rate + (geo if case.get("moving") else 0.0)
    flops = case["steps"] * (pairs * (2.0 * geo + rate) + iters * (pairs * per_iter + n * (8.0 * d + 3.0)))
    if case["family"] in ("cavity", "dambreak"):
        flops += case["steps"] * pairs * (geo + 6.0 * d + 2.0 * d * d)
    fields = n * (3 * d + 1)
    out = 8 if case["fp64"] else 4
    return {"bytes": float(fields * (8 + out)), "flops": flops}


# -------------------------------------------------------------------- exact

class _Exact:
    """One instance in FP64: fluid first, then the walls, as plain tensors."""

    def __init__(self, cfg, x, v, p, vp, walls=None):
        self.c = cfg
        self.dim, self.nf = cfg["dim"], x.shape[0]
        self.xw = torch.zeros(0, self.dim, dtype=torch.float64, device=x.device)
        self.vw = self.xw
        if walls is not None:
            self.xw = torch.as_tensor(walls[0], device=x.device)
            self.vw = torch.as_tensor(walls[1], device=x.device)
        self.x, self.v, self.p, self.vp = x.clone(), v.clone(), p.clone(), vp.clone()
        d = self.dim
        self.lo = torch.tensor(cfg["lo"][:d], dtype=torch.float64, device=x.device)
        self.L = torch.tensor([cfg["hi"][a] - cfg["lo"][a] for a in range(d)], dtype=torch.float64, device=x.device)
        self.per = torch.tensor([bool(cfg["periodic"][a]) for a in range(d)], device=x.device)
        h = cfg["h"]
        self.sigma = 7.0 / (478.0 * math.pi * h * h) if d == 2 else 1.0 / (120.0 * math.pi * h ** 3)

    def wrap(self, x):
        y = torch.where(x >= self.lo + self.L, x - self.L, torch.where(x < self.lo, x + self.L, x))
        return torch.where(self.per, y, x)

    def sep(self, a, b):
        d = a - b
        m = torch.where(d > 0.5 * self.L, d - self.L, torch.where(d < -0.5 * self.L, d + self.L, d))
        return torch.where(self.per, m, d)

    def kernel(self, r):
        q = r / self.c["h"]
        a, b, c = (3.0 - q).clamp(min=0), (2.0 - q).clamp(min=0), (1.0 - q).clamp(min=0)
        w = self.sigma * (a ** 5 - 6.0 * b ** 5 + 15.0 * c ** 5)
        dw = self.sigma / self.c["h"] * (-5.0 * a ** 4 + 30.0 * b ** 4 - 75.0 * c ** 4)
        return w, dw

    def neighbours(self, xf):
        """Per particle the neighbours within 3h, padded with the particle itself,
        and their number."""
        x = torch.cat([xf, self.xw])
        n, d, dev = x.shape[0], self.dim, x.device
        rc = 3.0 * self.c["h"]
        nc = torch.floor(self.L / (rc * (1 + 1e-9))).long().clamp(min=1)
        k = torch.minimum(torch.floor((x - self.lo) / (self.L / nc)).long().clamp(min=0), nc - 1)
        stride = [1, int(nc[0]), int(nc[0]) * int(nc[1])][:d]
        cell = sum(k[:, a] * stride[a] for a in range(d))
        ncell = int(nc.prod())
        order = torch.argsort(cell, stable=True)
        count = torch.bincount(cell, minlength=ncell)
        start = torch.cumsum(count, 0) - count
        cap = int(count.max())
        lane = torch.arange(cap, device=dev)
        offs = [torch.tensor([(o // 3 ** a) % 3 - 1 for a in range(d)], device=dev) for o in range(3 ** d)]
        rows, lists = max(1, int(6e7) // (cap * 3 ** d)), []
        for r0 in range(0, n, rows):
            i = torch.arange(r0, min(n, r0 + rows), device=dev)
            cand, good = [], []
            for o in offs:
                kk = k[i] + o
                ok = (self.per | ((kk >= 0) & (kk < nc))).all(1)
                kk = torch.remainder(kk, nc)
                cc = sum(kk[:, a] * stride[a] for a in range(d))
                cand.append((start[cc][:, None] + lane).clamp(max=n - 1))
                good.append(ok[:, None] & (lane < count[cc][:, None]))
            j = order[torch.cat(cand, 1)]
            ok = torch.cat(good, 1)
            s = self.sep(x[i][:, None, :], x[j])
            r2 = (s * s).sum(2)
            ok &= (r2 < rc * rc) & (j != i[:, None])
            cnt = ok.sum(1)
            at = ok.nonzero()
            pos = torch.arange(at.shape[0], device=dev) - (torch.cumsum(cnt, 0) - cnt)[at[:, 0]]
            nb = i[:, None].repeat(1, int(cnt.max()))
            nb[at[:, 0], pos] = j[at[:, 0], at[:, 1]]
            lists.append((r0, nb, cnt))
        return lists

    def geometry(self, xf, lists):
        """Per chunk of particles: first particle, neighbours, r_ij, |r_ij|, W,
        gradW_ij, F_ij, a flag that excludes the padding."""
        x = torch.cat([xf, self.xw])
        out = []
        for r0, nb, cnt in lists:
            i = torch.arange(r0, r0 + nb.shape[0], device=x.device)
            d = self.sep(x[i][:, None, :], x[nb])
            r2 = (d * d).sum(2)
            r = r2.sqrt()
            w, dw = self.kernel(r)
            real = torch.arange(nb.shape[1], device=x.device) < cnt[:, None]
            gw = torch.where(r > 0, dw / r.clamp(min=1e-300), torch.zeros_like(r))[:, :, None] * d
            F = dw * r / (r2 + self.c["eta"] * self.c["h"] ** 2)
            out.append((r0, nb, d, r, w, gw, F, real))
        return out

    def rates(self, geo, v, p, vt=None):
        c, nf, dim = self.c, self.nf, self.dim
        m, rho = c["m"], c["rho0"]
        cs = c["beta"] * c["v_ref"]
        g = torch.tensor(c["g"][:dim], dtype=torch.float64, device=v.device)
        pa, vd, vv = p, v, v
        if self.xw.shape[0]:
            pw = torch.zeros(self.xw.shape[0], dtype=torch.float64, device=v.device)
            vg = 2.0 * self.vw.clone()
            zp, zv = torch.cat([p, pw]), torch.cat([v, vg])
            for r0, nb, d, r, w, gw, F, real in geo:
                lo = max(nf - r0, 0)
                if lo >= nb.shape[0]:
                    continue
                j, ww = nb[lo:], w[lo:] * (real[lo:] & (nb[lo:] < nf))
                sw = ww.sum(1)
                has = sw > 0
                div = torch.where(has, sw, torch.ones_like(sw))
                pj = (zp[j] * ww + rho * (d[lo:] * g).sum(2) * ww).sum(1) / div
                if c["free_surface"]:
                    pj = pj.clamp(min=0)
                a = r0 + lo - nf
                pw[a:a + j.shape[0]] = torch.where(has, pj, torch.zeros_like(pj))
                vg[a:a + j.shape[0]] -= torch.where(has[:, None], (zv[j] * ww[:, :, None]).sum(1) / div[:, None], torch.zeros_like(vg[:1]))
            pa, vd, vv = torch.cat([p, pw]), torch.cat([v, self.vw]), torch.cat([v, vg])
        ap, acc = torch.empty_like(p), torch.empty_like(v)
        for r0, nb, d, r, w, gw, F, real in geo:
            k = min(nf - r0, nb.shape[0])
            if k <= 0:
                continue
            j, gw, F, d, r = nb[:k], gw[:k], F[:k], d[:k], r[:k]
            e = slice(r0, r0 + k)
            vi, pi, pj = v[e][:, None, :], p[e][:, None], pa[j]
            dd, dv = vi - vd[j], vi - vv[j]
            a = m * cs * cs * (dd * gw).sum((1, 2))
            if c["edac"]:
                a = a + 4.0 * m / (2.0 * rho * rho) * (c["h"] * cs / 16.0) * ((pi - pj) * F).sum(1)
            pres = (pi + pj) / (rho * rho)
            if c["alpha"]:
                vr = (dv * d).sum(2)
                phi = vr.clamp(max=0) / (r * r + c["eta"] * c["h"] ** 2)
                pres = pres - c["alpha"] * c["h"] * cs * phi / rho
            f = -(m * pres[:, :, None] * gw).sum(1) + 4.0 * m * c["nu"] / (2.0 * rho) * (F[:, :, None] * dv).sum(1)
            if vt is not None:
                t = (vt[e][:, None, :] * gw).sum(2)
                a = a + (vt[e] * (m / (rho * rho) * ((pi + pj)[:, :, None] * gw).sum(1))).sum(1)
                f = f + m / rho * ((vi + vd[j]) * t[:, :, None]).sum(1)
            ap[e], acc[e] = a, f + g
        return ap, acc

    def stop(self, k, hp, hv):
        c = self.c
        if not (math.isfinite(hp[-1]) and math.isfinite(hv[-1])):
            return True
        if hp[-1] < c["eps"] and hv[-1] < c["eps"]:
            return True
        w = c["stag_window"]
        if w and k >= w:
            flat = [max(h[-w:]) > 0 and (max(h[-w:]) - min(h[-w:])) / max(h[-w:]) < c["stag_tol"] for h in (hp, hv)]
            if all(flat):
                return True
        return k >= c["max_iter"]

    def step(self):
        c, nf = self.c, self.nf
        step = c["dt"]
        tau = step / c["beta"]
        cs = c["beta"] * c["v_ref"]
        ap, f = self.rates(self.geometry(self.x, self.neighbours(self.x)), self.v, self.p)
        v = self.v + step * f
        x0 = self.wrap(self.x + step * self.v + 0.5 * step * step * f)
        p, moving = self.p, c["moving"]
        lists = self.neighbours(x0)
        geo = self.geometry(x0, lists)
        kappa = 2.0 * step / (2.0 * step + 3.0 * tau)
        xk, vt = x0, torch.zeros_like(v)
        k, hp, hv = 0, [], []
        while True:
            if moving and k:
                xh = self.wrap(xk + 0.5 * tau * vt)
                if moving == 2:
                    lists = self.neighbours(xh)
                geo = self.geometry(xh, lists)
            elif moving:
                xh = xk
            ph = p + 0.5 * tau * ap
            ap, f = self.rates(geo, v, ph, vt if moving else None)
            a = kappa * (f - (3.0 * v - 4.0 * self.v + self.vp) / (2.0 * step))
            v = v + tau * a
            p = ph + 0.5 * tau * ap
            if moving:
                vt = step * a
                xk = xh + 0.5 * tau * vt
            k += 1
            res = torch.stack([ap.abs().sum() * (step / (c["rho0"] * cs * cs)), step * a.norm(dim=1).sum() / c["v_ref"]]).tolist()
            hp.append(res[0] / nf)
            hv.append(res[1] / nf)
            if self.stop(k, hp, hv):
                break
        self.x = self.wrap(self.x + 0.5 * step * (self.v + v))
        self.vp, self.v, self.p = self.v, v, p
        del geo
        if c["shifting"]:
            self.shift()

    def shift(self):
        c, nf, dim = self.c, self.nf, self.dim
        h, vol = c["h"], c["m"] / c["rho0"]
        wh = float(self.kernel(torch.tensor(h, dtype=torch.float64))[0])
        x, v, p = self.x.clone(), self.v.clone(), self.p.clone()
        for r0, nb, d, r, w, gw, F, real in self.geometry(self.x, self.neighbours(self.x)):
            k = min(nf - r0, nb.shape[0])
            if k <= 0:
                continue
            j, gw, w, d, real = nb[:k], gw[:k], w[:k], d[:k], real[:k]
            e = slice(r0, r0 + k)
            dr = -0.5 * h * h * (vol * (1.0 + w / wh)[:, :, None] * gw).sum(1)
            if c["free_surface"]:
                div = -(vol * (d * gw).sum(2)).sum(1)
                dr = torch.where((div < dim - 0.5)[:, None], torch.zeros_like(dr), dr)
            fl = (real & (j < nf))
            jf = torch.where(fl, j, torch.arange(r0, r0 + k, device=j.device)[:, None])
            gf = vol * gw * fl[:, :, None]
            gp = ((self.p[jf] - self.p[e][:, None])[:, :, None] * gf).sum(1)
            p[e] += (gp * dr).sum(1)
            for b in range(dim):
                gv = ((self.v[jf, b] - self.v[e, b][:, None])[:, :, None] * gf).sum(1)
                v[e, b] += (gv * dr).sum(1)
            x[e] += dr
        self.x, self.v, self.p = self.wrap(x), v, p


def exact(case, seed):
    if case["family"] == "batch":
        done = []
        for cfg, x, v, p, vp in _instances(case, seed):
            e = _Exact(cfg, x, v, p, vp)
            for _ in range(case["steps"]):
                e.step()
            done.append((e.x, e.v, e.p, e.vp))
        return [torch.cat([d[k] for d in done]) for k in range(4)]
    cfg, x, v, p, vp, walls = _inputs(case, seed)
    e = _Exact(cfg, x, v, p, vp, walls)
    if case["family"] == "rates":
        return list(e.rates(e.geometry(x, e.neighbours(x)), v, p))
    for _ in range(case["steps"]):
        e.step()
    return [e.x, e.v, e.p, e.vp]
