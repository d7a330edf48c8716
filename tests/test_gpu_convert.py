"""State conversion FP64 <-> working precision: bit for bit what numpy's casts give,
over rounding ties, the ends of the float range, subnormals, zeros of both signs,
infinities and NaN, at sizes around one block of the conversion kernels."""
import numpy as np
import pytest

import paper_2605_12915_gb300 as af
from workloads import inputs as I

pytestmark = pytest.mark.gpu


def _values(rng, shape):
    """Random bit patterns of doubles around the float range, and the special ones."""
    bits = rng.integers(0, 2 ** 63, size=shape, dtype=np.uint64) * 2 + \
        rng.integers(0, 2, size=shape, dtype=np.uint64)
    near = rng.normal(size=shape) * 10.0 ** rng.integers(-46, 40, size=shape)
    x = np.where(rng.random(shape) < 0.2, bits.view(np.float64), near)
    f = rng.normal(size=shape).astype(np.float32)
    ulp = np.spacing(f).astype(np.float64)
    ties = f.astype(np.float64) + ulp * rng.choice([0.5, -0.5, 0.25, 0.5000000001], size=shape)
    x = np.where(rng.random(shape) < 0.3, ties, x)
    special = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 2.0 ** -126, 2.0 ** -127, 2.0 ** -149,
                        2.0 ** -150, -2.0 ** -150, 1.5 * 2.0 ** -150, 3.4028235677973366e38,
                        3.4028235677973362e38, -3.4028235677973366e38, 1e300, 2.0 ** -1074])
    flat = x.reshape(-1)
    flat[rng.permutation(flat.size)[:special.size]] = special
    return x


@pytest.mark.parametrize("precision", ["fp32", "fp32_comp", "fp64"])
@pytest.mark.parametrize("shape", [(2, 2), (127, 1 + 1), (16, 8), (43, 9)])
def test_round_trip_is_the_cast(precision, shape):
    nx, ny = shape
    P = I.uniform(nx, ny)
    st = P.state.copy()
    st[4, 0, 0] = st[7, 0, 0] = -1.0  # no storage offsets
    s = af.Solver(P.grid, P.gamma, st, precision=precision)
    x = _values(np.random.default_rng(nx), st.shape)
    s.set_state(x)
    got = s.state()
    s.close()
    with np.errstate(all="ignore"):
        hi = x.astype(np.float32)
        want = hi.astype(np.float64)
        if precision == "fp32_comp":
            lo = (x[:4] - want[:4]).astype(np.float32).astype(np.float64)
            want[:4] = want[:4] + lo
        if precision == "fp64":
            want = x
    nan = np.isnan(want)
    assert np.array_equal(np.isnan(got), nan)
    assert np.array_equal(got[~nan], want[~nan])
