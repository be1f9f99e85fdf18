"""Solves of several threads share the GPU, and solves of many launches.

How many CTAs a solve's grid has, and how many blocks of rows a CTA then takes,
depends on whether other solves are in flight; the sums do not, so the solution
is the same to the bit.  Sizes: a block of rows to two CTAs (60 x 60), one CTA a
block alone and several blocks a CTA beside other solves (220 x 220), several
blocks a CTA always (300 x 300).
"""
import threading
import time

import numpy as np
import pytest

from paper_1603_09311_gb300 import build as B
from paper_1603_09311_gb300 import inputs as I
from paper_1603_09311_gb300 import sdd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()
    sdd.lib()


def _problem(n, seed):
    rng = np.random.default_rng(seed)
    nodes, edge = I.rect_grid(0.0, 0.9, 0.0, 0.9, n, n)
    u = np.exp(-np.sqrt(20j) * nodes[:, 1]) * (1.0 + 0.1 * nodes[:, 0]) + 1e-3 * rng.standard_normal(len(nodes))
    return nodes, edge, np.where(edge == 1, u, 0.0), np.full(len(nodes), 20.0)


def _solve(case, **kw):
    return sdd.sdd_rbffd_solve(*case, n_stencil=9, eps=5.0, **{"tol": 1e-9, "max_iter": 20000, **kw})


def _together(cases):
    got, errors = [None] * len(cases), []

    def one(k):
        try:
            got[k] = _solve(cases[k])
        except Exception as e:
            errors.append(e)

    threads = [threading.Thread(target=one, args=(k,)) for k in range(len(cases))]
    t0 = time.perf_counter()
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    return got, time.perf_counter() - t0


@pytest.mark.parametrize("sizes", [(60,) * 8, (220,) * 3, (300,) * 3, (12, 60, 220, 300, 181, 30)])
def test_the_same_solution_beside_other_solves(sizes):
    cases = [_problem(n, k) for k, n in enumerate(sizes)]
    alone = [_solve(c) for c in cases]
    for _ in range(2):
        got, _ = _together(cases)
        for (u, st), (v, sv) in zip(alone, got):
            assert st["iterations"] == sv["iterations"] and np.array_equal(u, v)


def test_two_large_solves_overlap():
    # a solve waits on its barriers half of its time: two at once take about 1.5
    # times one, one after the other they take twice as long
    cases = [_problem(300, k) for k in range(2)]
    _together(cases)
    one = min(_together(cases[:1])[1] for _ in range(3))
    two = min(_together(cases)[1] for _ in range(3))
    assert two < 1.8 * one, (one, two)


def test_the_state_is_carried_from_launch_to_launch():
    # many launches, and turns, up to the tolerance; a cap one past 1024
    nodes, edge, values, kappa = case = _problem(400, 1)
    u, st = _solve(case)
    assert st["iterations"] > 1024 and st["status"] == sdd.SDD_OK
    stn, w = sdd.sdd_rbffd_weights(nodes, 9, 5.0)
    full = np.where(edge == 1, values, u)
    free = edge == 0
    row = (w * full[stn]).sum(1) - 1j * kappa * full
    b = (w * np.where(edge == 1, values, 0.0)[stn]).sum(1)
    assert np.linalg.norm(row[free]) <= 2e-9 * np.linalg.norm(b[free])
    _, st = _solve(case, max_iter=1025, allow_unconverged=True)
    assert st["iterations"] == 1025 and st["status"] == sdd.SDD_E_TIMEOUT
