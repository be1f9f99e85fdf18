"""The spline on knots whose spacing grows, and with values of any range.

A far knot's weight in a target's sum is a second derivative times the square
of the target's spacing.  On knots whose spacing grows fast enough it does not
fall off, so no column of weights may end early there; and a value far larger
than the others, or not finite, counts with any weight.

Reference: the dense weights of oracle/interp.py.  Tolerance: both sides
eliminate without pivoting, all terms of one sign, so an entry of the second
derivatives is good to 4 roundings a row; a weight is the sum of two such
entries, which can cancel, and a value the sum of n weights times values.  With
S = sum_j |v_j| (a [j = i] + b [j = i + 1] + (a^3 + a) h^2 / 6 |G_ij| +
(b^3 + b) h^2 / 6 |G_i+1,j|) the two sides differ by at most 16 n 2^-52 S.
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


def _bound(s, u, t):
    """16 n 2^-52 S per target and component."""
    G = np.abs(OI.spline_moments(s))
    n, out = len(s), []
    for x in t:
        i = OI.segment(s, x)
        h = s[i + 1] - s[i]
        a, b = (s[i + 1] - x) / h, (x - s[i]) / h
        c = (a ** 3 + a) * h * h / 6.0 * G[i] + (b ** 3 + b) * h * h / 6.0 * G[i + 1]
        c[i] += a
        c[i + 1] += b
        out.append(c @ np.abs(u))
    return 16 * n * 2.0 ** -52 * np.asarray(out)


@pytest.mark.parametrize("mirrored", [False, True])
@pytest.mark.parametrize("ratio,nk", [(1.5, 120), (2.0, 45), (2.0, 60), (2.2, 45), (2.5, 45), (2.5, 60), (3.0, 40),
                                      (3.0, 60), (10.0, 20)])
def test_growing_spacings_equal_the_dense_spline(ratio, nk, mirrored):
    r = np.random.default_rng(nk)
    s = np.concatenate([[0.0], np.cumsum(ratio ** np.arange(nk - 1.0))])
    if mirrored:
        s = -s[::-1]
    v, se = r.uniform(0.5, 1.5, (nk, 3)) * [1, -1, 1], r.uniform(0.5, 1.5, (nk, 3))
    t = np.concatenate([s, 0.3 * s[1:] + 0.7 * s[:-1]])
    val, err = sdd.sdd_interpolate(s, v, se, t, 1)
    ref, ref_se = OI.interpolate(s, v, se, t, OI.SPLINE)
    assert np.all(np.abs(val - ref) <= _bound(s, v, t))
    assert np.all(np.abs(err - ref_se) <= _bound(s, se, t))


@pytest.mark.parametrize("nk,far", [(200, 90), (700, 70), (700, 600)])
def test_an_outlier_counts_with_any_weight(nk, far):
    # 1e120 at a knot whose weights here are about 0.27^(rows away): the sum is its term
    r = np.random.default_rng(far)
    s = np.arange(float(nk))
    v, se = r.uniform(0.5, 1.5, (nk, 2)), r.uniform(0.5, 1.5, (nk, 2))
    v[far, 0] = se[far, 1] = 1e120
    t = np.sort(r.uniform(0.0, nk - 1.0, 60))
    val, err = sdd.sdd_interpolate(s, v, se, t, 1)
    ref, ref_se = OI.interpolate(s, v, se, t, OI.SPLINE)
    assert np.all(np.abs(val - ref) <= _bound(s, v, t))
    assert np.all(np.abs(err - ref_se) <= _bound(s, se, t))


def test_an_infinite_value_keeps_its_sign():
    # infinite with the sign of its weight, as in a sum over all knots
    nk = 300
    s = np.arange(float(nk))
    v, se = np.ones((nk, 3)), np.ones((nk, 3))
    v[20, 0], v[280, 1], se[280, 2] = np.inf, -np.inf, np.inf
    t = np.linspace(0.3, 298.6, 40)
    val, err = sdd.sdd_interpolate(s, v, se, t, 1)
    C = OI.weights(s, t, OI.SPLINE)
    assert np.all(C[:, [20, 280]] != 0.0)
    assert np.array_equal(val[:, 0], np.copysign(np.inf, C[:, 20]))
    assert np.array_equal(val[:, 1], np.copysign(np.inf, -C[:, 280]))
    assert np.all(np.isposinf(err[:, 2])) and np.all(np.isfinite(err[:, :2]))
    assert np.allclose(val[:, 2], 1.0, rtol=0, atol=16 * nk * 2.0 ** -52 * 3)
