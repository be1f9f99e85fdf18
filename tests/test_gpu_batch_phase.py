"""The phase form of a batched model is its own.

Phases of rates below a limit (kappa dt / (4 pi) < 2^20) are summed as exact
turns, others in double precision.  Which of them a model gets must not depend
on the models it is batched with: its values are those it has alone, up to the
order of the FP64 sums (1e-12 of the largest, as for served requests).  The
rates here are near the limit, where a phase of some 1e8 radians is good to 1e-8
in double precision and the two forms give different samples.
"""
import numpy as np
import pytest

from paper_1603_09311_gb300 import build as B
from paper_1603_09311_gb300 import inputs as I
from paper_1603_09311_gb300 import sdd

pytestmark = pytest.mark.gpu


def _entry(kappa, n):
    m = I._model([[0.0, kappa]])
    m["raster"] = I.rasterize(m, 64, 48)
    nodes = I.nodes_line((-0.5, 0.2), (0.5, 0.3), n)
    return {"ctx": sdd.sdd_create(m), "nodes": nodes, "n_paths": np.full(n, 3000)}


@pytest.mark.parametrize("other", [3.0, 1.0e10, 2.0e10])
def test_values_do_not_depend_on_the_other_models(other):
    B.build()
    dt = 1e-3
    a, b = _entry(1.0e10, 8), _entry(other, 8)
    (alone,), _ = sdd.sdd_batch_values([a], dt, 5)
    (mixed, _), _ = sdd.sdd_batch_values([a, b], dt, 5)
    for x, y in zip(alone, mixed):
        assert np.abs(x - y).max() <= 1e-12 * np.abs(x).max()
