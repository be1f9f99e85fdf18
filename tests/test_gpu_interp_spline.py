"""The spline's banded weights and the cuts of its chains.

Reference: the dense spline of oracle/interp.py (a direct solve over all knots,
all weights in every sum) on spacings that decay fast and slowly, with knot
counts on both sides of the kept band (160 knots to each side), of a CTA's
columns and of the warm-up of the forward sweep.  Both sides eliminate a
diagonally dominant matrix without pivoting (errors of a few ulp a row) and sum
at most 700 terms of weights that add up to at most 3 in modulus: 700 x 1.1e-16
x 3 x 2 sides = 5e-13, with a factor of 20 for the weights' own errors: 1e-11
of the largest value (standard errors: relative).
"""
import numpy as np
import pytest

from oracle import interp as OI
from paper_1603_09311_gb300 import build as B
from paper_1603_09311_gb300 import sdd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()
    sdd.lib()


SPACINGS = {
    "even": lambda n, r: np.ones(n - 1),
    "random": lambda n, r: r.uniform(0.01, 1.0, n - 1),
    "alternating": lambda n, r: np.where(np.arange(n - 1) % 2, 1e-3, 1.0),
    "shrinking": lambda n, r: 0.97 ** np.arange(n - 1),
    "steps": lambda n, r: 10.0 ** (-3.0 * ((np.arange(n - 1) // 7) % 2)),
}


@pytest.mark.parametrize("spacing", sorted(SPACINGS))
@pytest.mark.parametrize("nk", [3, 4, 17, 20, 33, 161, 322, 323, 700])
def test_spline_equals_the_dense_one(spacing, nk):
    r = np.random.default_rng(nk)
    s = np.concatenate([[0.0], np.cumsum(SPACINGS[spacing](nk, r))])
    V = 3
    v, se = r.standard_normal((nk, V)), r.uniform(0.5, 1.5, (nk, V))
    t = np.sort(np.concatenate([s[::5], 0.5 * (s[1:] + s[:-1])[::3], r.uniform(s[0], s[-1], 40), s[[0, -1]]]))
    val, err = sdd.sdd_interpolate(s, v, se, t, 1)
    ref, ref_se = OI.interpolate(s, v, se, t, OI.SPLINE)
    assert np.abs(val - ref).max() <= 1e-11 * np.abs(ref).max()
    assert np.abs(err / ref_se - 1.0).max() <= 1e-11
    only, none = sdd.sdd_interpolate(s, v, None, t, 1)
    assert none is None and np.array_equal(only, val)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_a_value_that_is_not_finite_spoils_its_component(bad):
    # as when every knot's term is in every sum, also 400 knots away
    s = np.linspace(0.0, 1.0, 500)
    v, se = np.ones((500, 2)), np.ones((500, 2))
    v[499, 1] = bad
    se[499, 0] = bad
    val, err = sdd.sdd_interpolate(s, v, se, np.array([0.0333, 0.5, 0.77]), 1)
    assert np.all(np.isfinite(val[:, 0])) and not np.any(np.isfinite(val[:, 1]))
    assert not np.any(np.isfinite(err[:, 0])) and np.all(np.isfinite(err[:, 1]))
