"""Walls in 3D: a closed box of fluid under gravity with a moving lid, against the FP64
oracle (the tolerances of the 2D cavity: FP64 1e-10, FP32C 1e-4), and the bits of
the loop drivers against each other. Every component of a wall particle's ghost
velocity and its pressure is formed by a lane of its own."""
import numpy as np
import pytest

import oracle
import paper_1904_00861_gb300 as dt
import synth

pytestmark = pytest.mark.gpu

F64, F32 = dt.DTSPH_FP64, dt.DTSPH_FP32C


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1904_00861_gb300 import build
    build.build()
    oracle.build()


def box(n=8, layers=3):
    dx = 1.0 / n
    cfg = synth.base_params(3, dx, 1.0, 0.01, eps=1e-4)
    lo, hi = -layers * dx, 1.0 + layers * dx
    cfg.update(periodic=(0, 0, 0), lo=(lo,) * 3, hi=(hi,) * 3, g=(0.1, -0.3, 0.2))
    i = np.indices((n + 2 * layers,) * 3).reshape(3, -1).T - layers
    wall = ((i < 0) | (i >= n)).any(1)
    xf, xw = (i[~wall] + 0.5) * dx, (i[wall] + 0.5) * dx
    rng = np.random.default_rng(6)
    xf = xf + 0.1 * dx * (2 * rng.random(xf.shape) - 1)
    v = 0.1 * rng.normal(size=xf.shape)
    vw = np.zeros_like(xw)
    vw[xw[:, 1] > 1.0] = (1.0, 0.0, 0.5)
    return dict(cfg=cfg, x=np.concatenate([xf, xw]), v=v, p=np.zeros(len(xf)), v_prev=v.copy(), vw=vw, nf=len(xf))


def run(d, prec, nsteps, **over):
    sim = dt.Simulation(d["cfg"], precision=prec, **over)
    nf = d["nf"]
    sim.set_state(d["x"][:nf], d["v"], d["p"], d["v_prev"], walls=(d["x"][nf:], d["vw"]))
    sim.step(nsteps)
    sim.sync()
    out = sim.x, sim.v, sim.p, [(s["iters"], s["reason"]) for s in sim.stats(0, nsteps)]
    sim.close()
    return out


def rel(a, b):
    return float(np.max(np.abs(a - b)) / np.max(np.abs(b)))


@pytest.mark.parametrize("lanes", [1, 4])
@pytest.mark.parametrize("prec", [F64, F32])
def test_box_with_walls(prec, lanes):
    d = box()
    orc = oracle.State(d["cfg"], d["x"], d["v"], d["p"], d["v_prev"], vw=d["vw"], nf=d["nf"])
    rec = orc.step(2)
    x, v, p, st = run(d, prec, 2, graph=2, lanes=lanes)
    nf = d["nf"]
    tol = 1e-10 if prec == F64 else 1e-4
    assert rel(v, orc.v[:nf]) < tol and rel(p, orc.p[:nf]) < tol
    if prec == F64:
        assert [s[0] for s in st] == [r["iters"] for r in rec]
    x1, v1, p1, st1 = run(d, prec, 2, graph=1, lanes=lanes)
    assert np.array_equal(x, x1) and np.array_equal(v, v1) and np.array_equal(p, p1) and st == st1
