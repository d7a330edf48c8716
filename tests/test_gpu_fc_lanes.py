"""The foot-centred update's lane groups: grids smaller than one thread block, sizes
around its multiples, and feet on every side of the grid lines (each sign pair
assembles the four regions of a vertex differently)."""
import numpy as np
import pytest

import paper_2605_12915_gb300 as af
from workloads import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(2, 2), (3, 5), (16, 1 + 16), (31, 33)])
@pytest.mark.parametrize("flow", [(0.3, 0.2), (-0.3, 0.2), (-0.3, -0.2), (0.3, 0.0), (0.0, -0.2)])
def test_fc_lane_groups_match_oracle(orc, shape, flow):
    P = I.random_smooth(*shape, seed=sum(shape), amp=0.04, flow=flow)
    s = af.Solver(P.grid, P.gamma, P.state, precision="fp64", variant="fc")
    s.step(P.dt, 1)
    got = s.state()
    s.close()
    want, flags = orc.run(P.state, P.grid.h, P.gamma, P.dt, 1, orc.FC)
    assert flags == 0
    # 1e-12 of the state, the tolerance of the variant's other parity tests; a plane
    # of vanishing velocity is judged by the sound speed (1)
    scale = np.maximum(np.max(np.abs(want), axis=(1, 2)), 1.0)
    assert np.max(np.max(np.abs(got - want), axis=(1, 2)) / scale) < 1e-12
