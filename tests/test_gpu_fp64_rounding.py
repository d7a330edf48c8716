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


def _scaling(a, b):
    """Factors of the sixteen planes for density times 2^a and pressure times 2^b, hence
    velocities times 2^((b - a) / 2)."""
    r, p, w = 2.0 ** a, 2.0 ** b, 2.0 ** ((b - a) // 2)
    return np.array([r, r * w, r * w, p] + 3 * [r, w, w, p])[:, None, None]


@pytest.mark.parametrize("variant", ["tai", "rb"])
@pytest.mark.parametrize("a,b,s", [(550, 480, 440), (200, 150, 0), (-100, 60, 0)])
def test_fp64_step_and_adjoint_scale_exactly(a, b, s, variant):
    """The same flow in other units, every factor a power of two (lambda's common one is
    2^s): all operations commute with it, so the step scales bitwise and the adjoint up to
    the order of its atomic sums.  In the first case the product of density and pressure
    leaves FP64's range; no value of the frozen coefficients does, nor, the variations
    being small, the products of the pressure increments with the density."""
    from workloads import inputs as I
    P = I.random_smooth(24, 19, seed=5, amp=1e-7)
    f = _scaling(a, b)
    dt = P.dt * (0.6 if variant == "rb" else 1.0)
    lam = np.random.default_rng(3).normal(size=P.state.shape)
    out = []
    for st, l, t in ((P.state, lam, dt),
                     (P.state * f, lam / f * 2.0 ** s, dt * 2.0 ** ((a - b) // 2))):
        h = af.Solver(P.grid, P.gamma, st, precision="fp64", variant=variant)
        l = h.adjoint(t, l)
        h.step(t, 3)
        out.append((h.state(), l))
        h.close()
    assert np.array_equal(out[1][0], out[0][0] * f)
    got = out[1][1] * f * 2.0 ** -s
    assert np.max(np.abs(got - out[0][1])) < 1e-13 * np.max(np.abs(out[0][1]))
