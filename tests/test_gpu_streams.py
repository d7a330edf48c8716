"""Work of other streams ahead of a call: a slow producer on a side stream writes the
planes that a call reads, the handle's stream waits for its event (or copies or fills
them itself) directly before the call, with the call's own kernels already running just
before; the result is that of planes that were ready long ago."""
import numpy as np
import pytest

import paper_2605_12915_gb300 as af
from workloads import inputs as I

pytestmark = pytest.mark.gpu

SLOW = 4_000_000  # clock cycles of the producer's delay, about 2 ms


def _slowly(torch, main, dst, src):
    """dst <- src on a side stream after the delay; `main` waits for it."""
    side = torch.cuda.Stream()
    side.wait_stream(main)
    with torch.cuda.stream(side):
        torch.cuda._sleep(SLOW)
        dst.copy_(src, non_blocking=True)
    main.wait_stream(side)
    dst.record_stream(side)


@pytest.mark.parametrize("precision", ["fp64", "fp32_comp"])
@pytest.mark.parametrize("shape", [(40, 36), (256, 256)])
def test_set_state_and_adjoint_after_a_wait(precision, shape):
    import torch
    P = I.random_smooth(*shape, seed=2, amp=0.04)
    st = torch.from_numpy(P.state).cuda()
    lam = torch.from_numpy(np.random.default_rng(1).normal(size=P.state.shape)).cuda()
    want_s = af.Solver(P.grid, P.gamma, P.state, precision=precision)
    want = want_s.adjoint(P.dt, lam.cpu().numpy())
    want_s.step(P.dt, 3)
    want_state = want_s.state()
    want_s.close()
    main = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(main):
        s = af.Solver(P.grid, P.gamma, torch.full_like(st, 1.0) * st, precision=precision,
                      stream=main)
        s.step(0.5 * P.dt, 2)  # another state, and kernels just before the wait
        planes = torch.ones_like(st)
        _slowly(torch, main, planes, st)
        s.set_state(planes)
        lin, out = torch.zeros_like(lam), torch.empty_like(lam)
        _slowly(torch, main, lin, lam)
        s.adjoint(P.dt, lin, out)
        s.step(P.dt, 3)
        got = torch.empty_like(st)
        s.state(got)
        torch.cuda.synchronize()
        s.close()
    tol = 1e-13 if precision == "fp64" else 2e-6  # (the order of the atomic sums)
    assert np.max(np.abs(out.cpu().numpy() - want)) < tol * np.max(np.abs(want))
    assert np.array_equal(got.cpu().numpy(), want_state)


@pytest.mark.parametrize("host", [False, True])
def test_sync_waits_for_the_exchanged_planes(host):
    """af_sync after an exchange, with the outgoing copy still in flight and steps just
    before it: `out` is complete when it returns."""
    import torch
    P = I.random_smooth(512, 512, seed=2, amp=0.04)
    st = torch.from_numpy(P.state)
    st = st.clone() if host else st.pin_memory()
    for _ in range(5):
        s = af.Solver(P.grid, P.gamma, P.state, precision="fp32_comp")
        out = torch.full_like(st, -1.0)
        out = out if host else out.pin_memory()
        before = s.state()
        s.exchange_async(out, st)
        s.step(P.dt, 1)
        s.sync()
        assert np.array_equal(out.numpy(), before)
        s.close()


@pytest.mark.parametrize("captured", [False, True])
def test_step_after_other_work_on_its_stream(captured):
    """Steps directly after a wait, a copy and a fill of the caller's on the handle's
    stream, launched and captured."""
    import torch
    P = I.random_smooth(96, 64, seed=2, amp=0.04)
    ref = af.Solver(P.grid, P.gamma, P.state, precision="fp32_comp")
    ref.step(P.dt, 6)
    want = ref.state()
    ref.close()
    main = torch.cuda.Stream()
    a, b = torch.zeros(1 << 20, device="cuda"), torch.ones(1 << 20, device="cuda")
    torch.cuda.synchronize()

    def work(s):
        with torch.cuda.stream(main):
            s.step(P.dt, 2)
            _slowly(torch, main, a, b)
            s.step(P.dt, 2)
            b.copy_(a, non_blocking=True)
            s.step(P.dt, 1)
            a.zero_()
            s.step(P.dt, 1)

    s = af.Solver(P.grid, P.gamma, P.state, precision="fp32_comp", stream=main)
    if captured:
        warm = af.Solver(P.grid, P.gamma, P.state, precision="fp32_comp", stream=main)
        warm.step(P.dt, 1)  # (set-up of the kernel outside the capture)
        warm.sync()
        warm.close()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=main):
            work(s)
        graph.replay()
    else:
        work(s)
    torch.cuda.synchronize()
    assert np.array_equal(s.state(), want)
    s.close()
