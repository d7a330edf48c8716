"""Rounding of the FP64 path's building blocks, each against exact arithmetic (rational
numbers, or binary scalings that must commute with every operation), with bounds counted
from the operations' own roundings (2^-53 of each result)."""
from fractions import Fraction

import numpy as np
import pytest

import paper_2605_12915_gb300 as af

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53


class _Grid:
    def __init__(self, nx, ny, h=1.0):
        self.nx, self.ny, self.h = nx, ny, h


def test_centre_recovery_rounds_the_deviations_only():
    """The recovered density of the lightest centre (the reported minimum, all points
    being denser) against rational arithmetic.  The deviations are at most D: each is
    rounded once, their sums of four three times (2, 3, 4 D), weighted 1/16 and 1/4: 4.1 D;
    the weighted sum 1.25 D; the centre itself once."""
    rng = np.random.default_rng(11)
    nx = ny = 2
    solver = None
    for _ in range(200):
        st = np.zeros((16, ny, nx))
        for b in (4, 8, 12):
            st[b] = rng.uniform(1.0, 1.05, (ny, nx))
            st[b + 3] = 1.0
        st[0] = rng.uniform(0.98, 1.0, (ny, nx))
        st[3] = 2.5
        if solver is None:
            solver = af.Solver(_Grid(nx, ny), 1.4, st, precision="fp64")
        else:
            solver.set_state(st)
        got = solver.invariants()[8]
        F = np.vectorize(Fraction)
        u, V, X, Y = F(st[0]), F(st[4]), F(st[8]), F(st[12])
        roll = lambda a, dy, dx: np.roll(a, (-dy, -dx), (0, 1))
        exact = min((Fraction(9, 4) * u
                     - (V + roll(V, 0, 1) + roll(V, 1, 0) + roll(V, 1, 1)) / 16
                     - (X + roll(X, 0, 1) + Y + roll(Y, 1, 0)) / 4).ravel())
        D = 0.07
        assert abs(Fraction(got) - exact) <= EPS * (1.0 + 5.4 * D)
    solver.close()
