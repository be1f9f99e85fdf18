"""Walks in cooperative rounds and exits recorded in batches.

A call with few walks gives every warp its share of them from the start, and
the lanes of the warp work for those walks together (two steps a lane and
round); a large call does so only once its queue is empty.  The walks must be
the same either way, record for record, at every number of walks a warp can
hold (1 .. 16 together, 17 and more one a lane), for every lookup program and
in both precisions, also when walks reach max_steps inside a round.
Reference: the same paths as part of a launch of fixed items, whose warps fill
their lanes.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1603_09311_gb300 import build as B
from paper_1603_09311_gb300 import inputs as I
from paper_1603_09311_gb300 import sdd

pytestmark = pytest.mark.gpu

BIG = 3000  # fixed items of 96 paths: 32 warps, each with full lanes


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()
    sdd.lib()


def _raster(model, K):
    m = dict(model)
    r = I.rasterize(model, 97, 65)
    # K materials: split the earth in bands (the material sets the counters used)
    z = np.arange(65)[:, None] * np.ones((1, 97), dtype=int)
    r = np.where(r > 0, 1 + (r + z // 9) % (K - 1), 0).astype(np.int8)
    m.update(raster=r, shapes=[], kappa=[[0.0] + [2.0 * (k + 1) for k in range(K - 1)]])
    return m


def _two_shapes():
    return {"domain": I.DOMAIN, "kappa": [[0.0, 2.0, 20.0, 7.0]], "bg": (0, 1), "g": ("columns", 1, 1),
            "shapes": [(0, 2, (-0.2, 0.3, -0.2, 0.3, 0.0, 0.0)), (1, 3, (-0.4, 0.2, 0.4, 0.3, 0.1, 0.8))]}


MODELS = {
    "layers": I.halfspace(), "contact": I.quarterspace(), "rect16": I.block_batched(), "triangle": I.triangle(),
    "shapes": _two_shapes(), "raster2": _raster(I.halfspace(), 2), "raster4": _raster(I.triangle(), 4),
    "raster8": _raster(I.triangle(), 8),
}


def _records(ctx, count, **cfg):
    return sdd.sdd_walk_records(ctx, 0.05, 0.35, 3, 11, count, 1e-3, 77, **cfg)


def _same(a, b, n):
    for k in b:
        assert np.array_equal(a[k][:n], b[k][:n]), k


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("name", sorted(MODELS))
def test_few_walks_equal_the_walks_of_a_large_launch(name, precision):
    ctx = sdd.sdd_create(MODELS[name])
    try:
        big = _records(ctx, BIG, precision=precision, chunk_paths=96)
        for n in (1, 2, 3, 5, 31, 700):
            _same(_records(ctx, n, precision=precision), big, n)
        # 1, 3, 5, 11, 16 and 17 walks a warp: one CTA of 32 threads on each SM
        for share in (1, 3, 5, 11, 16, 17):
            n = min(BIG, share * 152 - 7)
            _same(_records(ctx, n, precision=precision, block_threads=32, ctas_per_sm=1), big, n)
    finally:
        ctx.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("max_steps", [1, 8, 40, 264])
def test_truncation_inside_a_round(max_steps, precision):
    ctx = sdd.sdd_create(MODELS["contact"])
    try:
        big = _records(ctx, BIG, precision=precision, chunk_paths=96, max_steps=max_steps)
        for n in (1, 4, 300, 1900):
            _same(_records(ctx, n, precision=precision, max_steps=max_steps), big, n)
    finally:
        ctx.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("paths", [[1], [2, 1], [7, 64, 1, 33], [997] * 5])
def test_small_calls_match_the_oracle(paths, precision):
    w = I.workload("quarterspace")
    nodes = w["nodes"][5:5 + len(paths)]
    npth = np.array(paths)
    ctx = sdd.sdd_create(w["model"])
    try:
        mean, se, st = sdd.sdd_interface_values(ctx, nodes, npth, 1e-3, 9, precision=precision)
        again, _, _ = sdd.sdd_interface_values(ctx, nodes, npth, 1e-3, 9, precision=precision, chunk_paths=64)
    finally:
        ctx.close()
    ref = O.interface_values(w["model"], nodes, npth, 1e-3, 9, urule=32 if precision == "fp64" else 23)
    assert st["walks"] == npth.sum() and st["steps"] == ref["steps"]
    assert np.abs(mean - again).max() <= 1e-12
    # FP64: the oracle's walks (1e-10 of |g| <= 1).  FP32: its decisions, exit
    # points and phases rounded (1e-4), and at most one walk in a hundred, or
    # one, with a step counted in the neighbouring material (a phase of
    # (20 - 2) dt / 2)
    tol = 1e-10 if precision == "fp64" else 1e-4 + 9e-3 * (1.0 + 0.01 * npth) / npth
    assert np.all(np.abs(mean - ref["mean"])[:, 0] <= tol)
    one = npth == 1
    assert np.all(np.isnan(se[one])) and np.all(np.isfinite(se[~one]))


TM_MODELS = {
    "analytic": I.tm_analytic(),
    "three_strips": I.tm_strips((1.0, 4.0, 0.5), (-0.3, 0.25), [[2.0, 20.0, 7.0]]),
    "equal_pair": I.tm_strips((2.0, 2.0, 8.0, 1.0), (-0.4, 0.1, 0.6), [[2.0, 1.0, 3.0, 4.0]]),
    "eight": I.tm_strips([1.0, 2.0, 4.0, 2.0, 1.0, 0.5, 3.0, 1.0], np.linspace(-0.6, 0.6, 7), [np.arange(1.0, 9.0)]),
}


@pytest.mark.parametrize("name", sorted(TM_MODELS))
@pytest.mark.parametrize("x0,max_steps", [(0.07, 0), (-0.3, 0), (0.0, 0), (0.07, 40), (0.0, 8)])
def test_few_tm_walks_equal_the_walks_of_a_large_launch(name, x0, max_steps):
    # x0 = -0.3 and 0 lie on interfaces of some of the models (a hit at t = 0)
    ctx = sdd.sdd_create(TM_MODELS[name])

    def rec(count, **cfg):
        return sdd.sdd_walk_occupation(ctx, x0, 0.2, 3, 11, count, 1e-3, 77, max_steps=max_steps, **cfg)

    try:
        big = rec(BIG, chunk_paths=96)
        for n in (1, 2, 3, 5, 31, 700):
            _same(rec(n), big, n)
        for share in (1, 3, 5, 11, 16, 17):
            n = min(BIG, share * 152 - 7)
            _same(rec(n, block_threads=32, ctas_per_sm=1), big, n)
    finally:
        ctx.close()


@pytest.mark.parametrize("E", [1, 2, 3, 4, 5, 8, 9, 16, 17, 32])
def test_sums_of_several_evaluations_equal_each_alone(E):
    # the walks do not depend on the rates, so row e of E evaluations is the
    # evaluation alone; only the order of the FP64 sums differs (500 terms)
    kap = np.stack([np.zeros(E), np.geomspace(0.1, 200.0, E), np.geomspace(50.0, 0.3, E)], axis=1)
    model = dict(I.quarterspace(), kappa=kap)
    nodes, paths = I.nodes_line((0.0, 0.1), (0.0, 0.8), 3), np.array([500, 33, 470])
    ctx = sdd.sdd_create(model)
    mean, se, _ = sdd.sdd_interface_values(ctx, nodes, paths, 1e-3, 4)
    ctx.close()
    for e in {0, E // 2, E - 1}:
        one = sdd.sdd_create(dict(model, kappa=kap[e:e + 1]))
        m1, s1, _ = sdd.sdd_interface_values(one, nodes, paths, 1e-3, 4)
        one.close()
        assert np.abs(mean[:, e] - m1[:, 0]).max() <= 1e-13 and np.abs(se[:, e] - s1[:, 0]).max() <= 1e-13


@pytest.mark.parametrize("dt", [1e-3, 2e-2])
def test_phases_in_turns_equal_the_phases_in_doubles(dt):
    # a rate too large for the integer phases (kappa dt / 4 pi >= 2^20) puts the
    # whole model on the FP64 sum; the other rows must agree: the two phases
    # differ by about 1e-13, so at most a sample in 1e5 rounds to another float
    # (1.2e-7): 1e-9 of |g| <= 1 for 900 walks.  At dt = 0.02 the larger rates
    # turn more than once a step.
    rows = [[0.0, 0.7, 3.0], [0.0, 2000.0, 1.0e4], [0.0, 900.0, 0.01]]
    nodes = I.nodes_line((0.0, 0.1), (0.0, 0.8), 2)
    got = []
    for extra in ([], [[0.0, 5.0, 2.0e7 / dt]]):
        ctx = sdd.sdd_create(dict(I.quarterspace(), kappa=rows + extra, g=("affine", 1.0, 0.3, 0.2)))
        got.append(sdd.sdd_interface_values(ctx, nodes, 900, dt, 4)[0][:, :3])
        ctx.close()
    assert np.abs(got[0] - got[1]).max() <= 1e-9
    ref = O.interface_values(dict(I.quarterspace(), kappa=rows, g=("affine", 1.0, 0.3, 0.2)), nodes, 900, dt, 4, urule=23)
    # the first row's rates are small: a step counted in the neighbouring
    # material is a phase of 1.2 dt in one of 900 walks
    assert np.abs(got[0][:, 0] - ref["mean"][:, 0]).max() <= 1e-4
