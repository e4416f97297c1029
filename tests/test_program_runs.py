"""Runs of the warp programs, on the CPU.  In a run the kernels load a pass's operands
before they store the results of the pass before it, and a reciprocal unit's three
passes load before any of them stores: the compiler must keep such passes independent,
and the groups and the run table it hands to the device must cover every pass in order."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import program_emulator as pe
from paper_2501_00011_gb300 import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2501_00011_gb300", "csrc")
PIPE, PIPE1, RECIP, SEQ = 0, 1, 2, 3            # run kinds of the table
TABLED = ("f", "m", "lu", "nudot", "jt")        # the triangular solves run their passes in order, without a table


def _third_order(m):
    """Some reactions of m with a third reactant: another species, or one of the two again."""
    for i, j in enumerate(np.nonzero(m.n_reac == 2)[0][::5]):
        m.reac[j, 2] = (m.reac[j, 0] + 1 + i) % m.n_species if i % 2 else m.reac[j, 0]
        m.n_reac[j] = 3
    return m


MECHS = {"small": synth.mechanism_small, "tropo": synth.mechanism_tropo, "pressure": synth.mechanism_tropo_pressure,
         "s50": lambda: synth.random_mechanism(50, 130, 40, 13, name="synthetic_50sp_130rx"),
         "s100": lambda: synth.random_mechanism(100, 260, 80, 26, name="synthetic_100sp_260rx"),
         "s128": lambda: synth.random_mechanism(128, 330, 100, 34, name="synthetic_128sp_330rx"),
         "third": lambda: _third_order(synth.random_mechanism(50, 130, 40, 13, name="synthetic_50sp_3rd"))}


@pytest.fixture(scope="module")
def programs(tmp_path_factory):
    from paper_2501_00011_gb300 import chemgpu
    wd = str(tmp_path_factory.mktemp("rundump"))
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    exe = os.path.join(wd, "rundump")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(cuda, "include"), os.path.join(ROOT, "tests", "native", "rundump.cpp"),
                    os.path.join(CSRC, "mechanism.cpp"), "-L", os.path.join(cuda, "lib64"), "-lcudart", "-o", exe], check=True)
    out = {}
    for name, make in MECHS.items():
        m = make()
        rx = chemgpu.reactions_from_synth(m)
        src, txt = os.path.join(wd, name + ".bin"), os.path.join(wd, name + ".txt")
        with open(src, "wb") as fh:
            fh.write(np.array([m.n_species, m.n_reactions], np.int32).tobytes())
            fh.write(bytes(memoryview(rx))[:ctypes.sizeof(chemgpu.Reaction) * m.n_reactions])
        subprocess.run([exe, src, txt], check=True)
        progs, cur = {}, None
        for line in open(txt):
            key, *val = line.split()
            if key == "program":
                cur = progs[val[0]] = {}
            else:
                cur[key] = np.array(val, np.int64)
        for p in progs.values():
            p["ops"] = p["ops"].reshape(-1, 32, 4)
            p["groups"] = p["groups"].reshape(-1, 2)
            p["table"] = p["table"].reshape(-1, 2)
        out[name] = progs
    return out


def _writes_reads(ops):
    w, r = set(), set()
    for t, a, b, c in ops.tolist():
        if t == pe.EMPTY:
            continue
        w.add(t & ~pe.RECIP)
        r.update((a,) if t & pe.RECIP else (a, b, c))
    return w, r


def _device_order(p, name):
    """The passes as the device takes them: (pass, loads before the previous pass's stores?)."""
    g, order, at = p["groups"], [], 0
    if name not in TABLED:
        assert g.size == 0 or np.array_equal(g[:, 0], 2 * np.arange(len(g)))
        return [(int(x), False) for pair in g for x in pair if x >= 0]
    assert p["table"][-1].tolist() == [0, 0]        # the interpreter reads an entry ahead
    for kind, n in p["table"][:-1].tolist():
        assert n > 0
        if kind == RECIP:
            for u in range(n):
                (a, b), (c, none) = g[at + 2 * u], g[at + 2 * u + 1]
                assert none == -1 and (b, c) == (a + 1, a + 2)
                order += [(int(a), False), (int(b), True), (int(c), True)]
            at += 2 * n
            continue
        for i in range(n):
            a, b = g[at + i]
            last = i == n - 1
            assert b == a + 1 or (b == -1 and kind == PIPE1 and last)
            # the second slot of a PIPE1 run's last group is not used
            order += [(int(a), kind != SEQ and i > 0)]
            if b >= 0:
                assert not (kind == PIPE1 and last)
                order += [(int(b), kind != SEQ)]
        at += n
    assert at == len(g)
    return order


@pytest.mark.parametrize("name", list(MECHS))
def test_every_pass_once_in_order(programs, name):
    for prog, p in programs[name].items():
        assert [x for x, _ in _device_order(p, prog)] == list(range(len(p["ops"]))), prog


@pytest.mark.parametrize("name", list(MECHS))
def test_passes_that_load_early_do_not_touch_what_is_stored_late(programs, name):
    early = dependent = 0
    for prog, p in programs[name].items():
        wr = [_writes_reads(o) for o in p["ops"].reshape(-1, 32, 4)]
        order = _device_order(p, prog)
        unit = p["unit"]
        for i, (x, before) in enumerate(order):
            if not before:
                dependent += i > 0 and bool((wr[x][0] | wr[x][1]) & wr[order[i - 1][0]][0])
                continue
            early += 1
            # the pass before; in a reciprocal unit both passes before the third
            back = [i - 1] + ([i - 2] if i >= 2 and unit[order[i - 2][0]] == 3 else [])
            for k in back:
                w, _ = wr[order[k][0]]
                assert not (wr[x][0] | wr[x][1]) & w, (prog, x)
    assert early > 0 and dependent > 0          # the check sees passes of both sorts


@pytest.mark.parametrize("name", list(MECHS))
def test_early_loads_give_the_passes_in_order(programs, name):
    """Replay on random slots, every early load before the stores it may overtake, against
    the passes one after the other: the same bits."""
    rng = np.random.default_rng(5)
    for prog, p in programs[name].items():
        ops = p["ops"].reshape(-1, 32, 4)
        if not len(ops):
            continue
        live = ops[ops[:, :, 0] != pe.EMPTY]
        n = int(max((live[:, 0] & ~pe.RECIP).max(), live[:, 1].max(), live[:, 2:].max())) + 1
        W0 = rng.uniform(0.5, 2.0, n)
        ref, W, pending = W0.copy(), W0.copy(), []

        def load(x):
            new = {}
            for t, a, b, c in ops[x].tolist():
                if t != pe.EMPTY:
                    new[t & ~pe.RECIP] = -1.0 / W[a] if t & pe.RECIP else W[a] * W[b] + W[c]
            return new

        unit = p["unit"]
        with np.errstate(all="ignore"):
            pe.run(ops, ref)
            for x, before in _device_order(p, prog):
                keep = 2 if unit[x - 2] == 3 and x >= 2 and before else 1 if before else 0
                while len(pending) > keep:
                    for t, v in pending.pop(0).items():
                        W[t] = v
                pending.append(load(x))
            for new in pending:
                for t, v in new.items():
                    W[t] = v
        assert np.array_equal(W.view(np.int64), ref.view(np.int64)), prog
