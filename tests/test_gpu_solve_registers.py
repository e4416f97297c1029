"""The solve kernels with fewer registers, which large batches of up to 32 species run:
the same results, cell by cell, as the kernels of smaller batches."""
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


def _solve(cg, mech, wl, n, driver, steps=1, prec=32, **kw):
    c = cg.Cells(mech, n, rtol=wl.rtol, atol=wl.atol, driver=driver, lu_precision=prec, **kw)
    c.set_state(wl.cells.T[:n], wl.cells.P[:n], np.ascontiguousarray(wl.cells.y[:, :n]))
    if steps == 1:
        c.solve_step(wl.dt)
    else:
        c.solve_steps(wl.dt, steps)
    out = c.get_state(), c.get_stats()
    c.close()
    return out


# the last batch of 80 cells per SM, the first above it, and one with a ragged last block
@pytest.mark.parametrize("driver", ["plain", "persistent"])
@pytest.mark.parametrize("extra", [0, 1, 1003])
def test_large_batch_equals_its_cells_in_small_batches(cg, driver, extra):
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    n = 80 * n_sm + extra
    wl = synth.workload_small(n_cells=n)
    mech = cg.Mechanism(wl.mech)
    steps = 2 if driver == "persistent" else 1
    y, st = _solve(cg, mech, wl, n, driver, steps)
    part = 80 * n_sm // 2
    for c0 in (0, n - part):
        sub = synth.workload_small(n_cells=n)
        sub.cells.T, sub.cells.P, sub.cells.y = (np.ascontiguousarray(a[..., c0:c0 + part])
                                                 for a in (wl.cells.T, wl.cells.P, wl.cells.y))
        ys, ss = _solve(cg, mech, sub, part, driver, steps)
        assert np.array_equal(y[:, c0:c0 + part].view(np.int64), ys.view(np.int64))
        assert np.array_equal(st[c0:c0 + part], ss)


# the plain driver's last batch of 12 cells per SM and the first above it
@pytest.mark.parametrize("kw", [{}, {"prec": 32}, {"record_adjoint": True, "tape_steps": 1500}],
                         ids=["fp64", "fp32", "recording"])
def test_plain_batch_equals_its_cells_in_small_batches(cg, kw):
    n = 12 * torch.cuda.get_device_properties(0).multi_processor_count + 1
    wl = synth.workload_small(n_cells=n)
    mech = cg.Mechanism(wl.mech)
    kw = {"prec": 64, **kw}
    y, st = _solve(cg, mech, wl, n, "plain", **kw)
    ys, ss = _solve(cg, mech, wl, n - 1, "plain", **kw)
    assert np.array_equal(y[:, :n - 1].view(np.int64), ys.view(np.int64)) and np.array_equal(st[:n - 1], ss)
