"""Units of the warp programs that the interpreter runs as a whole, on the CPU."""
import numpy as np
import pytest

import program_emulator as pe
from paper_2501_00011_gb300 import synth

MECHS = {"small": synth.mechanism_small, "tropo": synth.mechanism_tropo,
         "s128": lambda: synth.random_mechanism(128, 330, 100, 34, name="synthetic_128sp_330rx")}


@pytest.mark.parametrize("name", list(MECHS))
def test_reciprocal_units_are_three_independent_passes(name, tmp_path):
    """A reciprocal unit runs its three passes with every load before the stores: no op
    of the three may touch what another writes, and a reciprocal's lane has no op in the
    second and third."""
    cp = pe.Compiled(pe.build_dumper(str(tmp_path)), MECHS[name](), str(tmp_path))
    ops, unit = cp.progs["lu"], cp.units["lu"]
    starts = np.nonzero(unit == 3)[0]
    assert starts.size > 0
    for p in starts:
        assert p + 2 < len(unit) and unit[p + 1] == 0 and unit[p + 2] == 0
        rcp = (ops[p, :, 0] != pe.EMPTY) & ((ops[p, :, 0] & pe.RECIP) != 0)
        assert rcp.any()
        assert np.all(ops[p + 1:p + 3, rcp, 0] == pe.EMPTY)
        writes, touched = set(), []
        for t, a, b, c in ops[p:p + 3].reshape(-1, 4).tolist():
            if t == pe.EMPTY:
                continue
            reads = {a} if t & pe.RECIP else {a, b, c}
            w = t & ~pe.RECIP
            assert w not in writes
            writes.add(w)
            touched.append((w, reads))
        for w, reads in touched:
            assert not (reads - {w}) & writes
    # no reciprocal outside such a unit
    inside = set(starts.tolist())
    for p in range(ops.shape[0]):
        if p not in inside:
            assert not np.any((ops[p, :, 0] != pe.EMPTY) & ((ops[p, :, 0] & pe.RECIP) != 0))
