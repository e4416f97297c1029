"""Batches and pipelines created while the default stream has work queued: what the
library clears at creation is clear before any other stream uses it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2501_00011_gb300 import synth  # noqa: E402


@pytest.fixture(scope="module")
def cg():
    from paper_2501_00011_gb300 import build, chemgpu
    build.build()
    torch.cuda.init()
    return chemgpu


def _busy_default_stream():
    """Tens of milliseconds of matrix products on the default stream."""
    a = torch.randn(8192, 8192, device="cuda")
    for _ in range(60):
        a = (a @ a).clamp_(-1.0, 1.0)
    return a


@pytest.mark.parametrize("how", ["pipeline", "pipeline_host_work", "side_stream"])
def test_solve_right_after_creation_behind_a_busy_default_stream(cg, how):
    n = 700
    wl = synth.workload_tropo(n)
    mech = cg.Mechanism(wl.mech)
    ref = cg.Cells(mech, n, rtol=wl.rtol, atol=wl.atol, driver="persistent")
    ref.set_state(wl.cells.T, wl.cells.P, wl.cells.y)
    for _ in range(2):
        ref.solve_step(wl.dt)
    yr, sr = ref.get_state(), ref.get_stats()
    T, P = wl.cells.T.copy(), wl.cells.P.copy()
    y = cg.pinned_empty(wl.cells.y.shape)
    y[:] = wl.cells.y
    _busy_default_stream()                   # warm-up: the library handle and the memory
    torch.cuda.synchronize()
    keep = _busy_default_stream()
    if how == "side_stream":
        s = torch.cuda.Stream()
        c = cg.Cells(mech, n, rtol=wl.rtol, atol=wl.atol, driver="persistent")
        c.set_state(T, P, y, stream=s)
        for _ in range(2):
            c.solve_step(wl.dt, stream=s)
        got, st = c.get_state(stream=s), c.get_stats(stream=s)
    else:
        p = cg.Pipeline(mech, n, 4, rtol=wl.rtol, atol=wl.atol)
        st = p.run(T, P, y, wl.dt, 2, fn=(lambda c0, c1, step: None) if how == "pipeline_host_work" else None, stats=True)
        got = np.array(y)
    torch.cuda.synchronize()
    del keep
    assert np.array_equal(got, yr) and np.array_equal(st, sr)
