"""Grids of very many rows: rows must not run into the limit of 65535 blocks in a
launch's y dimension.  Each grid is a small one repeated along y, whose results it has to
repeat."""
import numpy as np
import pytest

import paper_2605_12915_gb300 as af
from workloads import inputs as I

pytestmark = pytest.mark.gpu


class _Grid:
    def __init__(self, nx, ny, h):
        self.nx, self.ny, self.h = nx, ny, h


def _repeated(P, times):
    return _Grid(P.grid.nx, P.grid.ny * times, P.grid.h), np.tile(P.state, (1, times, 1))


@pytest.mark.parametrize("precision,rows", [("fp64", 131071), ("fp32_comp", 262141),
                                            ("fp64", 524280)])
def test_adjoint_step(precision, rows):
    """One row more than 65535 blocks of 2 (FP64) and 4 rows, and the most rows that
    blocks of 8 would take."""
    P = I.random_smooth(2, 7, seed=1, amp=0.04)
    times = -(-rows // 7)
    grid, st = _repeated(P, times)
    lam = np.random.default_rng(3).normal(size=P.state.shape)
    s = af.Solver(P.grid, P.gamma, P.state, precision=precision)
    want = s.adjoint(P.dt, lam)
    s.close()
    s = af.Solver(grid, P.gamma, st, precision=precision)
    got = s.adjoint(P.dt, np.tile(lam, (1, times, 1)))
    s.close()
    # (the atomic sums are taken in another order)
    tol = 1e-13 if precision == "fp64" else 2e-6
    err = np.abs(got.reshape(16, times, 7, 2) - want[:, None])
    assert np.max(err) < tol * np.max(np.abs(want))


def test_fp32_step():
    """One row more than 65535 tiles of 16 rows, the height that narrow grids choose."""
    P = I.random_smooth(2, 1771, seed=1, amp=0.04)
    times = -(-1048561 // 1771)
    s = af.Solver(P.grid, P.gamma, P.state, precision="fp32_comp")
    s.step(P.dt, 2)
    want = s.state()
    s.close()
    grid, st = _repeated(P, times)
    s = af.Solver(grid, P.gamma, st, precision="fp32_comp")
    s.step(P.dt, 2)
    got = s.state(out=st)
    s.close()
    assert np.array_equal(got.reshape(16, times, 1771, 2),
                          np.broadcast_to(want[:, None], (16, times, 1771, 2)))
