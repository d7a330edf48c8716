"""Tile geometries of the fused FP32 step, chosen by the grid's size: each computes
bitwise what one CTA per 32 x 32 tile computes (AF_PIPE=0), at sizes around the
edges of every geometry's tiles and of its range, and under stream capture."""
import numpy as np
import pytest

import paper_2605_12915_gb300 as af
from workloads import inputs as I

pytestmark = pytest.mark.gpu


def _run(P, precision, variant, n):
    s = af.Solver(P.grid, P.gamma, P.state, precision=precision, variant=variant)
    s.step(P.dt * (0.6 if variant == "rb" else 1.0), n)
    out = s.state()
    s.close()
    return out


@pytest.mark.parametrize("precision,variant", [("fp32", "tai"), ("fp32_comp", "tai"),
                                               ("fp32_comp", "rb")])
@pytest.mark.parametrize("shape", [
    (2, 2), (3, 5), (8, 4), (9, 33),    # 8 x 4 tiles: smaller than one, one, remainders
    (97, 63), (96, 96),                 # 8 x 8
    (129, 120), (128, 152),             # 16 x 8
    (190, 185), (192, 208),             # 16 x 16
    (256, 256), (255, 290),             # 32 x 16
    (333, 250), (321, 334),             # 32 x 24
    (383, 400),                         # 32 x 32, one CTA per tile
    (512, 512), (500, 519),             # persistent, 28 rows
    (640, 608),                         # persistent, 32 rows
])
def test_step_geometry_is_bitwise_the_32x32_tiles(monkeypatch, shape, precision, variant):
    P = I.random_smooth(*shape, seed=shape[0] + 7 * shape[1], amp=0.05)
    got = _run(P, precision, variant, 5)
    monkeypatch.setenv("AF_PIPE", "0")
    want = _run(P, precision, variant, 5)
    assert np.array_equal(got, want)


@pytest.mark.parametrize("shape", [(40, 36), (512, 512)])
def test_captured_steps_equal_launched_steps(shape):
    """The steps' programmatic launches recorded in a CUDA graph and replayed."""
    import torch
    P = I.random_smooth(*shape, seed=3, amp=0.05)
    want = _run(P, "fp32_comp", "tai", 8)
    stream = torch.cuda.Stream()
    s = af.Solver(P.grid, P.gamma, P.state, precision="fp32_comp", stream=stream)
    s.step(P.dt, 4)
    s.sync()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        s.step(P.dt, 4)
    graph.replay()
    torch.cuda.synchronize()
    assert np.array_equal(s.state(), want)
    s.close()


def test_batch_on_24x16_tiles_is_bitwise_the_lone_steps(monkeypatch):
    """Four grids of 160 x 157 cells: 200 tiles of 32 x 16 (two waves) against 280 of
    24 x 16 (one wave of two per SM), so geometry 1 is the latter."""
    probs = [I.random_smooth(160, 157, seed=k, amp=0.05) for k in range(4)]
    monkeypatch.setenv("AF_BATCH_GEOM", "1")
    b = af.Batch(probs, precision="fp32_comp")
    b.step([p.dt for p in probs], 4)
    for k, p in enumerate(probs):
        assert np.array_equal(b.state(k), _run(p, "fp32_comp", "tai", 4)), k
    b.close()
