"""The derivative kernel's tiles (one lane per cell) against the f program (one warp per
cell, eval_deriv) it replaces: the same operations in the same order, so the same bits."""
import numpy as np
import pytest
import torch

from paper_2501_00011_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cg():
    from paper_2501_00011_gb300 import build, chemgpu
    build.build()
    torch.cuda.init()
    return chemgpu


def _mechanism(name):
    if name == "yields":        # fractional yields and a net coefficient of zero
        m = synth.random_mechanism(50, 130, 40, 13, name="synthetic_50sp_130rx")
        m.yld[::3] *= 0.7
        return m
    return {"small": synth.mechanism_small, "tropo": synth.mechanism_tropo,
            "s128": lambda: synth.random_mechanism(128, 330, 100, 34, name="synthetic_128sp_330rx")}[name]()


# in rounds of 32 cells on every SM: no round, the first tile, one round and its edges
# (the rest by the gather or as more tiles), two rounds with a rest that is not a multiple of 32
@pytest.mark.parametrize("name", ["small", "tropo", "yields", "s128"])
@pytest.mark.parametrize("rounds,rest", [(0, 1), (0, 33), (0, 2975), (1, -1), (1, 0), (1, 1), (1, 3333), (2, 271)])
def test_tiles_equal_the_f_program(cg, name, rounds, rest):
    n = rounds * 32 * torch.cuda.get_device_properties(0).multi_processor_count + rest
    m = _mechanism(name)
    mech = cg.Mechanism(m)
    cells = synth.random_cells(m.n_species, n, T_range=(210, 310), P_range=(2e4, 1e5), seed=n)
    y = cells.y.copy()
    y[::7, ::3] = 0.0            # zero rates of either sign
    y[3::11, 1::5] *= -1.0
    c = cg.Cells(mech, n)
    c.set_state(cells.T, cells.P, y)
    ref = c.eval_deriv(y)
    for dev in (False, True):
        got = c.eval_deriv_design(cg.DERIV_GATHER, torch.from_numpy(y).cuda() if dev else y)
        got = got.cpu().numpy() if dev else got
        assert np.array_equal(got.view(np.int64), ref.view(np.int64)), (name, n, dev)
    c.close()
