"""The invariants' reduction: table logarithm, filtered wave speed, integer minima.
Entropy, extrema and sums against numpy in FP64 on states whose density and
pressure span many binades (and sit around 1, where the logarithm is small), at
sizes around one block, one grid wave and a ragged remainder."""
import numpy as np
import pytest

import paper_2605_12915_gb300 as af

pytestmark = pytest.mark.gpu
G = 1.4


class _Grid:
    def __init__(self, nx, ny):
        self.nx, self.ny, self.h = nx, ny, 0.37


def _state(nx, ny, spread, seed):
    r = np.random.default_rng(seed)
    st = np.empty((16, ny, nx))
    for base in (4, 8, 12):
        st[base] = np.exp(spread * r.normal(size=(ny, nx)))
        st[base + 1:base + 3] = r.normal(size=(2, ny, nx))
        st[base + 3] = np.exp(spread * r.normal(size=(ny, nx)))
    return st


@pytest.mark.parametrize("spread", [1e-9, 0.3])
@pytest.mark.parametrize("shape", [(2, 2), (127, 1 + 1), (16, 8), (331, 470)])
def test_fp64_sums_and_extrema(shape, spread):
    nx, ny = shape
    st = _state(nx, ny, spread, nx + ny)
    # centres by the Simpson inversion of the averages
    def cons(w):
        return np.stack([w[0], w[0] * w[1], w[0] * w[2],
                         w[3] / (G - 1) + 0.5 * w[0] * (w[1] ** 2 + w[2] ** 2)])
    roll = lambda a, dy, dx: np.roll(a, (-dy, -dx), (1, 2))
    V, X, Y = cons(st[4:8]), cons(st[8:12]), cons(st[12:16])
    corners = V + roll(V, 0, 1) + roll(V, 1, 0) + roll(V, 1, 1)
    # averages whose recovered centres are the vertices' states: physical
    st[0:4] = (V + corners / 16 + (X + roll(X, 0, 1) + Y + roll(Y, 1, 0)) / 4) * 4 / 9
    uc = 9 / 4 * st[0:4] - corners / 16 - (X + roll(X, 0, 1) + Y + roll(Y, 1, 0)) / 4
    c = np.stack([uc[0], uc[1] / uc[0], uc[2] / uc[0], np.zeros_like(uc[0])])
    c[3] = (G - 1) * (uc[3] - 0.5 * (uc[1] * c[1] + uc[2] * c[2]))
    nodes = [st[4:8], st[8:12], st[12:16], c]
    ent = [-w[0] * (np.log(w[3]) - G * np.log(w[0])) for w in nodes]
    wts = [1 / 9, 2 / 9, 2 / 9, 4 / 9]
    h2 = 0.37 ** 2
    s = af.Solver(_Grid(nx, ny), G, st, precision="fp64")
    got = s.invariants()
    s.close()
    size = sum(w * np.sum(np.abs(e)) for w, e in zip(wts, ent)) * h2
    # each logarithm to 2 ulp of itself; the recovered centre to 1e-15 of the values
    # it is a difference of, which is an absolute error of that size in p and rho
    floor = h2 * nx * ny * 4e-15 * np.max(np.abs(st[:4])) / min(c[0].min(), c[3].min(), 1.0)
    assert abs(got[4] - h2 * sum(w * e.sum() for w, e in zip(wts, ent))) < 1e-14 * size + floor
    a = st[0:4]
    ke = 0.5 * (a[1] ** 2 + a[2] ** 2) / a[0]
    pa = (G - 1) * (a[3] - ke)
    ea = -a[0] * (np.log(pa) - G * np.log(a[0]))
    floor = h2 * nx * ny * 4e-15 * np.max(np.abs(a)) / min(pa.min(), 1.0)
    assert abs(got[5] - h2 * ea.sum()) < 1e-14 * h2 * np.abs(ea).sum() + floor
    for k in range(4):
        assert abs(got[k] - h2 * a[k].sum()) < 1e-13 * h2 * np.abs(a[k]).sum()
    assert abs(got[6] - h2 * ke.sum()) < 1e-13 * h2 * ke.sum()
    speed = max(float(np.max(np.hypot(w[1], w[2]) + np.sqrt(G * w[3] / w[0]))) for w in nodes)
    assert abs(got[7] - speed) < 1e-12 * speed
    assert abs(got[8] - min(w[0].min() for w in nodes)) < 1e-13 * np.max(np.abs(st[0]))
    assert abs(got[9] - min(w[3].min() for w in nodes)) < 1e-13 * np.max(np.abs(st[3]))


@pytest.mark.parametrize("precision", ["fp32", "fp32_comp", "fp64"])
@pytest.mark.parametrize("u", [0.0, 0.4])
def test_uniform_state_has_its_wave_speed(precision, u):
    """Every stored value of a uniform state at rest is 0 in the FP32 modes (offsets
    from the reference state): the maximum is still the sound speed."""
    from workloads import inputs as I
    P = I.uniform(37, 21, rho=1.3, u=u, v=0.0, p=0.9)
    s = af.Solver(P.grid, P.gamma, P.state, precision=precision)
    got = s.invariants()
    s.close()
    want = u + np.sqrt(P.gamma * 0.9 / 1.3)
    # the recovered centre carries the rounding of the averages in the working precision
    assert abs(got[7] - want) < (1e-6 if precision != "fp64" else 1e-13) * want
