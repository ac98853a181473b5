"""Kernel paths chosen by size, at the sizes where the choice changes: the list
builders, the resident loop of instances that fit one block per SM, the moving loop in
one launch, the batch loop's claims of two tiles and the allocation-free rates' overlapping
launches. Neighbour sets equal the oracle's;
every path computes its tiles and decisions as the launch-per-iteration graph (or the
solo run) does, so the comparisons are of bits.
"""
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


def run(d, prec, nsteps=2, **over):
    sim = dt.Simulation(d["cfg"], precision=prec, **over)
    nf = d["nf"]
    sim.set_state(d["x"][:nf], d["v"], d["p"], d["v_prev"], walls=None if d["vw"] is None else (d["x"][nf:], d["vw"]))
    sim.step(nsteps)
    sim.sync()
    out = (sim.x, sim.v, sim.p), [(s["iters"], s["reason"], s["rp"], s["rv"]) for s in sim.stats(0, nsteps)]
    sim.close()
    return out


def same(a, b):
    return all(np.array_equal(u, w) for u, w in zip(a[0], b[0])) and a[1] == b[1]


# 700 x 700: 54,289 cells (18,174 row segments of three; no multiple of the scan's
# pieces, more than one block scans); 3D boxes from the smallest number of cells up
@pytest.mark.parametrize("prec", [F64, F32])
@pytest.mark.parametrize("dim,n", [(2, 10), (2, 127), (2, 700), (3, 10), (3, 13), (3, 20)])
def test_list_builders(dim, n, prec):
    d = synth.tgv2d(n, seed=n) if dim == 2 else synth.tgv3d(n, jitter=0.2, seed=n)
    sim = dt.Simulation(d["cfg"], precision=prec)
    sim.set_state(d["x"], d["v"], d["p"], d["v_prev"])
    dt.dtsph_build_neighbors(sim.ctx)
    start, idx = oracle.neighbors(d["cfg"], d["x"])
    x = d["x"]
    some = np.concatenate([np.argsort(x[:, a])[s] for a in range(dim) for s in (slice(0, 12), slice(-12, None))])
    some = np.concatenate([some, np.random.default_rng(n).choice(len(x), min(len(x), 150), replace=False)])
    for i in some:
        assert np.array_equal(dt.dtsph_get_neighbors(sim.ctx, int(i)), idx[start[i]:start[i + 1]]), i
    sim.close()


# FP32C: 87,552 lanes of slots fit 152 SMs, FP64 48,640: the largest square that fits and
# the next one, at one lane and at eight; walls; 3D; a fraction of one block
@pytest.mark.parametrize("case,n,prec,lanes", [
    ("tgv2d", 295, F32, 1), ("tgv2d", 296, F32, 1), ("tgv2d", 104, F32, 8), ("tgv2d", 105, F32, 8),
    ("tgv2d", 220, F64, 1), ("tgv2d", 221, F64, 1), ("tgv2d", 77, F64, 8), ("tgv2d", 10, F32, 1), ("tgv2d", 10, F64, 4),
    ("cavity2d", 61, F32, 4), ("cavity2d", 61, F64, 1), ("cavity2d", 150, F32, 1),
    ("tgv3d", 43, F32, 1), ("tgv3d", 21, F32, 8), ("tgv3d", 17, F64, 4)])
def test_resident_loop(case, n, prec, lanes):
    d = getattr(synth, case)(n)
    for fixed in (7, 0):
        over = dict(lanes=lanes, fixed_iters=fixed, max_iter=40)
        assert same(run(d, prec, graph=2, **over), run(d, prec, graph=1, **over)), fixed


@pytest.mark.parametrize("lanes", [1, 2, 4, 8])
@pytest.mark.parametrize("prec", [F64, F32])
@pytest.mark.parametrize("case,n,moving", [("tgv2d", 37, 2), ("tgv3d", 11, 1), ("cavity2d", 23, 2)])
def test_moving_loop_in_one_launch(case, n, moving, prec, lanes):
    d = getattr(synth, case)(n)
    over = dict(moving=moving, lanes=lanes, max_iter=40)
    assert same(run(d, prec, graph=2, **over), run(d, prec, graph=1, **over))


# tiles of 32 slots (eight lanes): about 3,400 of them, more than six per block of three
# on each SM, in instances of odd and even tile counts
def test_batch_claims_of_two_tiles():
    insts = [synth.tgv2d(90 + i, re=100.0 + 40 * i, seed=i) for i in range(12)]
    b = dt.Batch([dict(d["cfg"], max_iter=30) for d in insts], precision=F32, graph=2, lanes=8, form=1)
    b.set_state(insts)
    b.step(2)
    b.sync()
    xs, vs, ps = b.field(dt.FIELD_POS), b.field(dt.FIELD_VEL), b.field(dt.FIELD_P)
    for i, d in enumerate(insts):
        (x, v, p), st = run(d, F32, graph=1, lanes=8, form=1, max_iter=30)
        assert np.array_equal(xs[i], x) and np.array_equal(vs[i], v) and np.array_equal(ps[i], p), i
        assert [(s["iters"], s["reason"], s["rp"], s["rv"]) for s in b.stats(i)] == st, i
    b.close()


# the overlapping launches of the allocation-free rates: calls back to back, where one
# call's kernels meet the scratch of the one before, against calls one at a time
@pytest.mark.parametrize("case,n,prec", [("tgv2d", 10, F64), ("tgv2d", 61, F32), ("cavity2d", 23, F64), ("tgv3d", 17, F32)])
def test_overlapping_rates(case, n, prec):
    import torch
    d = getattr(synth, case)(n)
    nf, dim = d["nf"], d["cfg"]["dim"]
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a, np.float64), device="cuda")
    x, p = dev(d["x"][:nf]), dev(d["p"])
    vs = [dev(d["v"] + 0.1 * k * np.random.default_rng(k).normal(size=d["v"].shape)) for k in range(6)]
    nw = len(d["x"]) - nf
    xw, vw = (dev(d["x"][nf:]), dev(d["vw"])) if nw else (None, None)
    prm = dt.make_params(d["cfg"], precision=prec)
    st = torch.cuda.Stream()
    F = [[torch.zeros(nf, dim, dtype=torch.float64, device="cuda") for _ in vs] for _ in range(2)]
    ap = [[torch.zeros(nf, dtype=torch.float64, device="cuda") for _ in vs] for _ in range(2)]
    torch.cuda.synchronize()
    for side in range(2):
        for k, v in enumerate(vs):
            dt.dtsph_eval_rates_noalloc(prm, nf, x, v, p, ap[side][k], F[side][k], nw=nw, xw=xw, vw=vw,
                                        stream=st.cuda_stream)
            if side:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
    for k in range(len(vs)):
        assert torch.equal(ap[0][k], ap[1][k]) and torch.equal(F[0][k], F[1][k]), k
    assert not torch.equal(F[0][0], F[0][1])
