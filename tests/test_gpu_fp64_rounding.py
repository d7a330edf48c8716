"""Rounding of the FP64 path's building blocks, each against exact arithmetic (rational
numbers, or binary scalings that must commute with every operation), with bounds counted
from the operations' own roundings (2^-53 of each result)."""
import ctypes
import os
import subprocess
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


@pytest.fixture(scope="module")
def extended_step(tmp_path_factory):
    """The oracle's step with long double (64 or 113 bits of mantissa) for double."""
    import oracle
    tmp = tmp_path_factory.mktemp("extended")
    src, lib = str(tmp / "extended.c"), str(tmp / "extended.so")
    path = os.path.join(os.path.dirname(oracle.__file__), "af_oracle.c")
    with open(src, "w") as f:
        f.write("#include <complex.h>\n#include <math.h>\n#include <stdlib.h>\n"
                "#include <string.h>\n#include <tgmath.h>\n#undef M_PI\n"
                "#define M_PI 3.14159265358979323846264338327950288L\n"
                "#define double long double\n#include \"%s\"\n" % path)
    subprocess.check_call(["gcc", "-O2", "-std=gnu11", "-ffp-contract=off", "-fPIC", "-shared",
                           "-o", lib, src, "-lm"])
    fn = ctypes.CDLL(lib).orc_step
    i, d = ctypes.c_int, ctypes.c_longdouble
    fn.argtypes = [i, i, d, d, d, i, ctypes.c_void_p, ctypes.c_void_p]

    def step(state, h, gamma, dt, variant):
        a = np.ascontiguousarray(state, dtype=np.longdouble)
        out = np.empty_like(a)
        fn(a.shape[2], a.shape[1], h, gamma, dt, variant, a.ctypes.data, out.ctypes.data)
        return out

    return step


def test_additive_update_adds_the_increment_to_the_foot_value(extended_step):
    """u = u_f + du with u_f exact: on the row of one vertex u is 1.0625 there, 0.75 at the
    edge midpoint before it and 0.25 at the vertex before that; with dt / h = 1/2 both
    Picard stages have short dyadic coordinates and u_f = 0.85 without a rounding.  du is
    small (c dt / h = 2^-11), so its own roundings are far below those of u, except that the
    recovered centre pressures around the vertex are rounded as parts of an energy of 1/2:
    2^-54 each, times dt / h / rho and the stencil's weights, 0.2 x 2^-54 or so.  What is
    left is the rounding of the sum, half a unit in the last place of [0.5, 1) = 2^-54.
    (du recovered from 1.0625 + du would add that of [1, 2), twice as much.)"""
    rng = np.random.default_rng(5)
    nx, ny, gamma, dt = 6, 5, 1.4, 0.5
    worst = 0.0
    for _ in range(60):
        st = np.zeros((16, ny, nx))
        for b in (4, 8, 12):
            st[b], st[b + 1] = 1.0, 0.75
            st[b + 3] = 2.0 ** -20 / gamma * rng.uniform(1.0, 1.1, (ny, nx))
        st[5, 2, 3], st[5, 2, 2] = 1.0625, 0.25
        roll = lambda a, dy, dx: np.roll(a, (-dy, -dx), (0, 1))
        cons = [[w[0], w[0] * w[1], 0 * w[0], w[3] / (gamma - 1) + 0.5 * w[0] * w[1] ** 2]
                for w in (st[4:8], st[8:12], st[12:16])]
        for k, c in enumerate((1.0, 0.75, 0.0, 2.0 ** -20 / gamma / (gamma - 1) + 0.5 * 0.75 ** 2)):
            V, X, Y = (q[k] for q in cons)
            st[k] = 4 / 9 * (c + (V + roll(V, 0, 1) + roll(V, 1, 0) + roll(V, 1, 1)) / 16 +
                             (X + roll(X, 0, 1) + Y + roll(Y, 1, 0)) / 4)
        s = af.Solver(_Grid(nx, ny), gamma, st, precision="fp64", variant="rb")
        s.step(dt, 1)
        got = s.state()[5, 2, 3]
        s.close()
        want = extended_step(st, 1.0, gamma, dt, 1)[5, 2, 3]
        assert 0.8 < got < 0.9
        worst = max(worst, float(abs(got - want)))
    assert worst <= 1.4 * EPS / 2


def test_interpolation_at_the_foot_rounds_as_row_sums():
    """The new densities of a flow of uniform velocity and pressure are the Q2
    interpolation of the old ones at the foot.  Everything before it is exact here: gamma
    3/2, velocities -1/2 and -1/4, densities 1 + 9 k / 2^16 with averages that recover a
    density of 1 at every centre, and a time step of 23 bits, so that the foot and its
    Lagrange weights are exact.  The sum by rows rounds three partial sums per row and the
    three of the rows, each by a value spread evenly over a unit in its last place: the
    measured rms error is that prediction's, with a tenth for the spread not being quite
    even.  (With the nine weights' products formed first it is twice the prediction.)"""
    rng = np.random.default_rng(8)
    nx, ny, dth = 160, 125, 0.2890625 + 2.0 ** -22
    st = np.zeros((16, ny, nx))
    for b in (4, 8, 12):
        st[b] = 1 + 9 * rng.integers(0, 7282, (ny, nx)) / 2.0 ** 16
        st[b + 1], st[b + 2], st[b + 3] = -0.5, -0.25, 1.0
    V, X, Y = st[4], st[8], st[12]
    roll = lambda a, dy, dx: np.roll(a, (-dy, -dx), (0, 1))
    rest = ((V - 1) + (roll(V, 0, 1) - 1) + (roll(V, 1, 0) - 1) + (roll(V, 1, 1) - 1)) / 9 / 16 + \
           ((X - 1) + (roll(X, 0, 1) - 1) + (Y - 1) + (roll(Y, 1, 0) - 1)) / 9 / 4
    st[0] = 1 + 4 * rest
    st[1], st[2], st[3] = -0.5 * st[0], -0.25 * st[0], 2 + 5 / 32 * st[0]
    s = af.Solver(_Grid(nx, ny), 1.5, st, precision="fp64")
    s.step(dth, 1)
    got = s.state()
    s.close()
    for b in (4, 8, 12):  # exact, as said
        assert np.all(got[b + 1] == -0.5) and np.all(got[b + 3] == 1.0)

    def weights(t):
        return [t * (t - 1) / 2, 1 - t * t, t * (t + 1) / 2]
    lx, ly = weights(np.longdouble(dth - 1)), weights(np.longdouble(0.5 * dth - 1))
    one = np.ones_like(V)
    rows = [[V, Y, roll(V, 0, 1)], [X, one, roll(X, 0, 1)],
            [roll(V, 1, 0), roll(Y, 1, 0), roll(V, 1, 1)]]
    var = lambda a: np.spacing(np.abs(a).astype(np.float64)) ** 2 / 12
    total, spread = 0, 0
    for b in range(3):
        row, row_var = 0, 0
        for q in range(3):
            row = row + lx[q] * rows[b][q].astype(np.longdouble)
            row_var = row_var + var(row)
        total = total + ly[b] * row
        spread = spread + float(ly[b]) ** 2 * row_var + var(total)
    err = (got[4] - total).astype(np.float64)
    assert np.sqrt(np.mean(err ** 2)) <= 1.1 * np.sqrt(np.mean(spread))
