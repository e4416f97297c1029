"""Consecutive steps of a cell in one launch (solve_steps) against single solve_step
calls: recording batches, cells that fail or run into the step cap, the FP32
factorisation, the plain driver."""
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


@pytest.fixture(scope="module")
def tropo(cg):
    return cg.Mechanism(synth.mechanism_tropo())


def _steps(cg, mech, wl, n_steps, fused, J=None, **kw):
    c = cg.Cells(mech, wl.cells.n_cells, rtol=wl.rtol, atol=wl.atol, **kw)
    c.set_state(wl.cells.T, wl.cells.P, wl.cells.y)
    if J is not None:
        c.set_photolysis(J)
    if fused:
        c.solve_steps(wl.dt, n_steps)
    else:
        for _ in range(n_steps):
            c.solve_step(wl.dt)
    return c


def _same(a, b):
    assert np.array_equal(a.get_stats(), b.get_stats())
    assert np.array_equal(a.get_state().view(np.int64), b.get_state().view(np.int64))


@pytest.mark.parametrize("driver", ["plain", "persistent"])
@pytest.mark.parametrize("prec", [64, 32])
def test_cells_that_fail_or_stop(cg, tropo, driver, prec):
    # bad T, P and y, an overflowing photolysis rate (no finite rate constants), and a
    # step cap that the first, stiffest step exceeds in some cells and later steps do not
    wl = synth.workload_batching(61)
    wl.cells.T[1] = np.nan
    wl.cells.P[2] = -1.0
    wl.cells.y[5, 3] = np.inf
    J = wl.cells.J.copy()
    J[0, 4] = np.inf
    seen = set()
    for cap in (5000, 90, 60):
        one = _steps(cg, tropo, wl, 3, False, J, driver=driver, lu_precision=prec, max_steps=cap)
        all_ = _steps(cg, tropo, wl, 3, True, J, driver=driver, lu_precision=prec, max_steps=cap)
        _same(one, all_)
        seen |= set(one.get_stats()["status"].tolist())
        if cap == 5000:
            assert (one.get_stats()["status"][1:5] == 6).all()
        one.close()
        all_.close()
    assert {0, 1, 6} <= seen


@pytest.mark.parametrize("driver", ["plain", "persistent"])
def test_recording(cg, tropo, driver):
    # the tape of fused steps is the tape of single steps, event by event, also where a
    # cell's tape overflows in the second step or later
    wl = synth.workload_adjoint(24)
    n, S = 24, wl.mech.n_species
    w = synth.loss_weights(S, n)
    rows = []
    full = _steps(cg, tropo, wl, 3, False, driver=driver, record_adjoint=True)
    rows = [full.get_tape(k)[3].shape[0] for k in range(n)]
    full.close()
    for tape in (0, int(np.median(rows))):
        one = _steps(cg, tropo, wl, 3, False, driver=driver, record_adjoint=True, tape_steps=tape)
        all_ = _steps(cg, tropo, wl, 3, True, driver=driver, record_adjoint=True, tape_steps=tape)
        _same(one, all_)
        fits = [k for k in range(n) if tape == 0 or rows[k] <= tape]
        assert len(fits) == n if tape == 0 else 0 < len(fits) < n
        for k in fits:
            for a, b in zip(one.get_tape(k), all_.get_tape(k)):
                assert np.array_equal(a, b)
        (g1, l1, bad1), (g2, l2, bad2) = one.sensitivity(w), all_.sensitivity(w)
        assert bad1 == bad2 == n - len(fits)
        assert np.array_equal(g1, g2) and np.array_equal(l1, l2)
        one.close()
        all_.close()


def test_recording_with_a_cell_that_fails(cg, tropo):
    wl = synth.workload_adjoint(9)
    wl.cells.T[4] = -3.0
    one = _steps(cg, tropo, wl, 2, False, driver="persistent", record_adjoint=True)
    all_ = _steps(cg, tropo, wl, 2, True, driver="persistent", record_adjoint=True)
    _same(one, all_)
    w = synth.loss_weights(wl.mech.n_species, 9)
    (g1, l1, bad1), (g2, l2, bad2) = one.sensitivity(w), all_.sensitivity(w)
    assert bad1 == bad2 == 1
    assert np.array_equal(g1, g2) and np.array_equal(l1, l2)
    one.close()
    all_.close()
