"""The exit step's fraction of a phase is exact in single precision's fraction.

A walk's phase is the sum over its steps and the fraction theta of its last one
of kappa dt / (4 pi) turns, formed in integers modulo a turn.  For a rate near
the limit of that form (2^20 turns a step) every bit of a small theta counts:
cut off below 2^-40, a theta turns the sample by up to 2^-20 turns, 6e-6.

Reference: the phase in rationals from the walk's record and the double kappa dt
0.0796; the boundary value is 1, so the sample is exp(-i phase).  The library's
angle is rounded to single precision (pi 2^-24 = 1.9e-7), its sine and cosine to
2 units of 2^-24 (1.2e-7), their products to one more: below 5e-7.
"""
from fractions import Fraction

import numpy as np
import pytest

from paper_1603_09311_gb300 import build as B
from paper_1603_09311_gb300 import inputs as I
from paper_1603_09311_gb300 import sdd

pytestmark = pytest.mark.gpu


def test_a_small_last_fraction_counts_in_full():
    B.build()
    dt, seed, n = 1e-2, 11, 4_000_000
    kappa = 1.04e6 / (dt * 0.07957747154594767)
    ctx = sdd.sdd_create(I.uniform_model(kappa))
    rec = sdd.sdd_walk_records(ctx, 0.0, 0.2, 5, 0, n, dt, seed)
    theta = rec["exit"][:, 2]
    t = Fraction(float(kappa * dt * 0.07957747154594767))
    cut = np.floor(theta * 2.0 ** 40) * 2.0 ** -40
    lost = (theta - cut) * float(t) * 2.0 * np.pi
    at = np.argsort(lost)[-8:]
    assert lost[at[-1]] > 1.5e-6  # a walk that shows it
    sums, nv, _ = sdd.sdd_range_sums(ctx, np.tile([[0.0, 0.2]], (len(at), 1)), at, np.ones(len(at)), dt, seed,
                                     node_ids=np.full(len(at), 5))
    assert np.all(nv == 1)
    for k, p in enumerate(at):
        turns = t * (int(rec["counts"][p, 0]) + Fraction(float(theta[p])))
        ph = 2.0 * np.pi * float(turns - round(turns))
        assert abs(sums[k, 0, 0] - np.cos(ph)) <= 5e-7 and abs(sums[k, 0, 1] + np.sin(ph)) <= 5e-7
