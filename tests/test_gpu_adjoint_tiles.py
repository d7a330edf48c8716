"""Tile geometries of the adjoint's fused sweep, chosen by the grid's size, and the
kernels per stage: each agrees with the FP64 adjoint, at sizes around the edges of
every geometry's tiles; the FP64 adjoint itself agrees with the transpose of the
step along random directions."""
import numpy as np
import pytest

import paper_2605_12915_gb300 as af
from workloads import inputs as I

pytestmark = pytest.mark.gpu


def _adjoint(P, lam, precision, variant="tai"):
    s = af.Solver(P.grid, P.gamma, P.state, precision=precision, variant=variant)
    out = s.adjoint(P.dt * (0.6 if variant == "rb" else 1.0), lam)
    again = s.adjoint(P.dt * (0.6 if variant == "rb" else 1.0), lam)  # cleared records
    s.close()
    # the second call differs by the order of the atomic sums only
    eps = 1e-6 if precision != "fp64" else 1e-13
    assert np.max(np.abs(out - again)) <= eps * np.max(np.abs(out))
    return out


@pytest.mark.parametrize("variant", ["tai", "rb"])
@pytest.mark.parametrize("shape", [
    (2, 3), (7, 9), (40, 33),   # 8 x 8 tiles
    (129, 96), (131, 120),      # 16 x 8
    (190, 185),                 # 16 x 16
    (256, 250), (255, 253),     # 32 x 8, two per SM
    (333, 251),                 # 32 x 24
    (400, 395),                 # 32 x 8, several waves
])
def test_fp32_sweep_geometries_match_fp64(shape, variant):
    P = I.random_smooth(*shape, seed=shape[0] + shape[1], amp=0.04)
    lam = np.random.default_rng(2).normal(size=P.state.shape)
    ref = _adjoint(P, lam, "fp64", variant)
    got = _adjoint(P, lam, "fp32_comp", variant)
    # 2e-5 of the largest entry, the tolerance of the FP32 adjoint elsewhere
    assert np.max(np.abs(got - ref)) < 2e-5 * np.max(np.abs(ref))


@pytest.mark.parametrize("shape", [(2, 2), (63, 65), (64, 33)])
def test_fp64_adjoint_is_the_transpose(shape):
    """<lambda, J d> against <J^T lambda, d> with J d by central differences of the
    FP64 step (eps 1e-6: truncation and rounding both below 1e-8 relative)."""
    P = I.random_smooth(*shape, seed=4, amp=0.04)
    rng = np.random.default_rng(7)
    lam = rng.normal(size=P.state.shape)
    d = rng.normal(size=P.state.shape)
    eps = 1e-6

    def step(x):
        s = af.Solver(P.grid, P.gamma, x, precision="fp64")
        s.step(P.dt, 1)
        out = s.state()
        s.close()
        return out

    jd = (step(P.state + eps * d) - step(P.state - eps * d)) / (2 * eps)
    jtl = _adjoint(P, lam, "fp64")
    lhs, rhs = np.sum(lam * jd), np.sum(jtl * d)
    scale = np.linalg.norm(lam) * np.linalg.norm(jd)
    assert abs(lhs - rhs) < 1e-7 * scale
