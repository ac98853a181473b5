"""Kernels chosen by size, each case with the name of the kernel that ran: the resident
loop at the largest square that fits one block per SM and at the next one, for every
number of lanes, with walls and in 3D (bits against the launch-per-iteration graph);
the list builder of many segments with closed axes, walls, crowded cells and several
instances (sets against the oracle), and its rows cut at the capacity; the barrier of
every persistent loop giving up.
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


def run(d, prec, **over):
    sim = dt.Simulation(d["cfg"], precision=prec, **over)
    nf = d["nf"]
    sim.set_state(d["x"][:nf], d["v"], d["p"], d["v_prev"], walls=None if d["vw"] is None else (d["x"][nf:], d["vw"]))
    kernel = dt.dtsph_step_kernels(sim.ctx)[1]
    sim.step(2)
    sim.sync()
    out = sim.x, sim.v, sim.p, [(s["iters"], s["reason"], s["rp"], s["rv"]) for s in sim.stats(0, 2)]
    sim.close()
    return kernel, out


def same_bits(d, prec, want, lanes):
    over = dict(lanes=lanes, fixed_iters=7)
    a, b = run(d, prec, graph=2, **over), run(d, prec, graph=1, **over)
    assert (a[0], b[0]) == (want, "k_iterate")
    assert all(np.array_equal(u, w) for u, w in zip(a[1][:3], b[1][:3])) and a[1][3] == b[1][3]


def largest_resident(prec, lanes):
    """The side of the largest square whose slots fit: whole warps of slots dealt to the
    SMs, at most 576 (FP32C) or 320 (FP64) threads on them in a block, at most 384
    tiles of 256 / lanes slots."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    fits = lambda n: (lambda s: -(-(s // 32) // sms) * 32 * lanes <= (576 if prec == F32 else 320)
                      and s // (256 // lanes) <= 384)(-(-n * n // 256) * 256)
    return max(n for n in range(10, 400) if fits(n))


@pytest.mark.parametrize("lanes", [1, 2, 4, 8])
@pytest.mark.parametrize("prec", [F64, F32])
def test_resident_loop_and_the_next_size(prec, lanes):
    n = largest_resident(prec, lanes)
    same_bits(synth.tgv2d(n, seed=n), prec, "k_loop_res", lanes)
    same_bits(synth.tgv2d(n + 1, seed=n), prec, "k_loop", lanes)


@pytest.mark.parametrize("lanes", [1, 2, 4, 8])
@pytest.mark.parametrize("prec", [F64, F32])
def test_resident_loop_with_walls_and_in_3d(prec, lanes):
    same_bits(synth.cavity2d(50), prec, "k_loop_res", lanes)
    same_bits(synth.tgv3d(16, jitter=0.1), prec, "k_loop_res", lanes)


def sparse(nx, ny, periodic, n, seed, crowd=0):
    """n particles at random in nx x ny cells (h = 1), `crowd` more in three cells by
    three in the middle, and rows of wall particles along the first closed edge."""
    rng = np.random.default_rng(seed)
    L = np.array([3.0 * nx + 1.0, 3.0 * ny + 1.0])
    x = rng.random((n, 2)) * L
    edge = np.abs(rng.normal(size=(n // 4, 2))) * 4.0                # some in a corner
    mid = 0.5 * L + rng.random((crowd, 2)) * 9.0
    x = np.minimum(np.concatenate([x, edge, mid]), L * (1 - 1e-9))
    closed = [a for a in range(2) if not periodic[a]]
    xw = np.zeros((0, 2))
    if closed:
        xw = np.stack(np.meshgrid(np.linspace(0.2, min(60.0, L.min() - 1), 90), [0.1, 0.7]), -1).reshape(-1, 2)[:, ::1 if closed[-1] else -1]
    cfg = dict(dim=2, h=1.0, m=1.0, periodic=(*periodic, 0), lo=(0.0,) * 3, hi=(*L, 1.0), nu=0.0, dt=0.01,
               max_neighbors=512)
    return dict(cfg=cfg, x=np.concatenate([x, xw]), nf=len(x), v=np.zeros_like(x), p=np.zeros(len(x)), v_prev=None,
                vw=np.zeros_like(xw) if len(xw) else None)


def check_lists(ctx, insts, n_first):
    dt.dtsph_build_neighbors(ctx)
    NF = sum(d["nf"] for d in insts)
    fo, wo = 0, NF
    for d in insts:
        nf, nw = d["nf"], len(d["x"]) - d["nf"]
        glob = np.concatenate([fo + np.arange(nf), wo + np.arange(nw)])
        start, idx = oracle.neighbors(d["cfg"], d["x"])
        pick = np.unique(np.concatenate([np.arange(max(0, nf - n_first), nf + nw),
                                         np.random.default_rng(1).choice(nf, min(nf, 200), replace=False)]))
        for i in pick:
            want = np.sort(glob[idx[start[i]:start[i + 1]]])
            assert np.array_equal(dt.dtsph_get_neighbors(ctx, int(glob[i])), want), i
        fo += nf
        wo += nw


# 224 x 222 cells and more: at least 16,384 segments of three (the last of a row with two
# or one); 300 in nine cells: ten rounds of 32 a segment, staged in more than one piece
@pytest.mark.parametrize("prec", [F64, F32])
@pytest.mark.parametrize("nx,ny,periodic", [(224, 222, (0, 0)), (223, 224, (1, 0)), (222, 224, (0, 1)), (224, 224, (1, 1))])
def test_lists_of_many_segments(nx, ny, periodic, prec):
    d = sparse(nx, ny, periodic, 1500, seed=nx + ny, crowd=300)
    sim = dt.Simulation(d["cfg"], precision=prec, lanes=4, graph=1)
    sim.set_state(d["x"][:d["nf"]], d["v"], d["p"], walls=None if d["vw"] is None else (d["x"][d["nf"]:], d["vw"]))
    assert dt.dtsph_step_kernels(sim.ctx)[0] == "k_nlist_home"
    check_lists(sim.ctx, [d], 500)
    sim.close()


@pytest.mark.parametrize("prec", [F64, F32])
def test_lists_of_many_segments_in_several_instances(prec):
    insts = [sparse(nx, nx, (0, i % 2), 600, seed=i, crowd=60 * i) for i, nx in enumerate((130, 131, 132, 5))]
    b = dt.Batch([d["cfg"] for d in insts], precision=prec, lanes=4, graph=1)
    b.set_state(insts)
    assert dt.dtsph_step_kernels(b.ctx)[0] == "k_nlist_home"
    check_lists(b.ctx, insts, 250)
    b.close()


@pytest.mark.parametrize("prec", [F64, F32])
@pytest.mark.parametrize("nx,kernel", [(40, "k_nlist_cells2"), (224, "k_nlist_home")])
def test_a_cut_list_is_reported(nx, kernel, prec):
    """A capacity below the crowded cells' counts, at and off a multiple of eight (the rows'
    stride): the build says so; with room it is right."""
    for cap in (16, 19):
        d = sparse(nx, nx, (1, 1), 400, seed=5, crowd=200)
        sim = dt.Simulation(d["cfg"], precision=prec, lanes=4, graph=1, max_neighbors=cap)
        sim.set_state(d["x"], d["v"], d["p"])
        assert dt.dtsph_step_kernels(sim.ctx)[0] == kernel
        with pytest.raises(dt.DtsphError) as e:
            dt.dtsph_build_neighbors(sim.ctx)
        assert e.value.code == dt.DTSPH_E_CAPACITY
        sim.close()
    sim = dt.Simulation(d["cfg"], precision=prec, lanes=4, graph=1)
    sim.set_state(d["x"], d["v"], d["p"])
    check_lists(sim.ctx, [d], 300)
    sim.close()


@pytest.mark.parametrize("prec", [F64, F32])
@pytest.mark.parametrize("case,over,kernel", [
    ("tgv2d", dict(moving=1), "k_move_loop"), ("cavity2d", dict(moving=2), "k_move_loop"),
    ("tgv2d", dict(form=1), "k_loop_res"), ("cavity2d", dict(), "k_loop_res")])
def test_a_barrier_that_gives_up_ends_the_step_with_a_status(monkeypatch, case, over, kernel, prec):
    """A give-up time of zero: every persistent loop ends its step early and dtsph_sync says
    DTSPH_E_TIMEOUT; a context without the setting runs the same state to its end."""
    d = getattr(synth, case)(60)
    nf = d["nf"]
    walls = None if d["vw"] is None else (d["x"][nf:], d["vw"])
    monkeypatch.setenv("DTSPH_TEST_BARRIER_WAIT_NS", "0")
    for give_up in (True, False):
        sim = dt.Simulation(d["cfg"], precision=prec, graph=2, lanes=2, max_iter=60, **over)
        sim.set_state(d["x"][:nf], d["v"], d["p"], d["v_prev"], walls=walls)
        assert dt.dtsph_step_kernels(sim.ctx)[1] == kernel
        sim.step(1)
        if give_up:
            with pytest.raises(dt.DtsphError) as e:
                sim.sync()
            assert e.value.code == dt.DTSPH_E_TIMEOUT
        else:
            sim.sync()
            assert sim.stats()[0]["reason"] in (0, 1, 2)
        sim.close()
        monkeypatch.delenv("DTSPH_TEST_BARRIER_WAIT_NS", raising=False)
