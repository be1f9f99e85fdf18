"""The sub-domain solver's cuts of the rows.

The solver gives a block of 256 rows to two CTAs, to one, or several blocks to
one CTA, by the number of blocks against the chip's SMs; sizes here lie on both
sides of every change and at ragged ends of a block, and the largest takes more
iterations than one launch runs.  The solution is checked by its residual with
the matrix assembled from the library's weights: at most 2 tol (the recursive
residual the solver stops on drifts from the true one by rounding alone, about
1e-16 x iterations x the growth of the iterates, orders below tol = 1e-8).
"""
import numpy as np
import pytest

from paper_1603_09311_gb300 import build as B
from paper_1603_09311_gb300 import inputs as I
from paper_1603_09311_gb300 import sdd

pytestmark = pytest.mark.gpu
TOL = 1e-8


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()
    sdd.lib()


def _problem(nx, nz, seed):
    rng = np.random.default_rng(seed)
    nodes, edge = I.rect_grid(0.0, 0.9, 0.0, 0.9 * (nz - 1) / (nx - 1) if nx > 1 else 0.9, nx, nz)
    k = np.sqrt(20j)
    u = np.exp(-k * nodes[:, 1]) * (1.0 + 0.1 * nodes[:, 0]) + 1e-3 * rng.standard_normal(len(nodes))
    return nodes, edge, np.where(edge == 1, u, 0.0), rng.uniform(2.0, 20.0, len(nodes))


# unknowns: 1, 255, 256, 257; 19320 and 19600 (76 blocks and 77, half of 152
# SMs); 40000; 78120 and 96100 (306 blocks and 376: past two CTAs an SM)
@pytest.mark.parametrize("nx,nz", [(3, 3), (17, 19), (18, 18), (3, 259), (140, 142), (142, 142), (202, 202),
                                   (281, 282), (312, 312)])
def test_solution_satisfies_the_assembled_system(nx, nz):
    nodes, edge, values, kappa = _problem(nx, nz, nx + nz)
    eps = 5.0 if nx * nz < 60000 else 8.0
    u, st = sdd.sdd_rbffd_solve(nodes, edge, values, kappa, n_stencil=9, eps=eps, tol=TOL)
    stn, w = sdd.sdd_rbffd_weights(nodes, 9, eps)
    full = np.where(edge == 1, values, u)
    free = edge == 0
    assert st["unknowns"] == free.sum() and st["status"] == 0
    row = (w * full[stn]).sum(1) - 1j * kappa * full
    b = (w * np.where(edge == 1, values, 0.0)[stn]).sum(1)
    assert np.linalg.norm(row[free]) <= 2.0 * TOL * np.linalg.norm(b[free])
    assert np.array_equal(u[edge == 1], values[edge == 1])


@pytest.mark.parametrize("max_iter", [1, 7, 1024, 1025])
def test_iteration_cap(max_iter):
    # the cap is kept inside a launch and across two
    nodes, edge, values, kappa = _problem(300, 300, 1)
    _, st = sdd.sdd_rbffd_solve(nodes, edge, values, kappa, n_stencil=9, eps=8.0, tol=1e-300, max_iter=max_iter,
                                allow_unconverged=True)
    assert st["status"] == sdd.SDD_E_TIMEOUT and st["iterations"] <= max_iter
    if max_iter < 1024:
        assert st["iterations"] == max_iter


def test_solves_beside_walks_and_in_several_threads():
    # the solver's CTAs wait for one another: they must come through while
    # walks fill the GPU on another stream, and with solves in other threads
    import threading

    cases = [_problem(60, 60, k) for k in range(3)]
    alone = [sdd.sdd_rbffd_solve(*c, n_stencil=9, eps=5.0, tol=TOL)[0] for c in cases]
    w = I.workload("quarterspace")
    ctx = sdd.sdd_create(w["model"])
    req = sdd.sdd_interface_values_async(ctx, w["nodes"], w["n_paths"] * 5, w["dt"], 3)
    got = [None] * 3

    def solve(k):
        got[k] = sdd.sdd_rbffd_solve(*cases[k], n_stencil=9, eps=5.0, tol=TOL)[0]

    threads = [threading.Thread(target=solve, args=(k,)) for k in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert req.wait() == sdd.SDD_OK
    req.free()
    ctx.close()
    for a, b in zip(alone, got):
        assert np.array_equal(a, b)
