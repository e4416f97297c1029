"""Reactions with three reactants on the GPU: every path that forms rates, partials or
the iteration matrix has code of its own for them (and the named workloads have none).
Against the oracle, and the derivative's tiles against the f program bit for bit."""
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


def _third_order(m):
    """Every third bimolecular reaction of m gets a third reactant: another species, the
    first once more (A + B + A), or three of a kind in turn, at a rate that matters
    beside the others for mixing ratios of 1e-12 to 1e-6."""
    for i, j in enumerate(np.nonzero(m.n_reac == 2)[0][::3]):
        a = m.reac[j, 0]
        m.reac[j, 2] = ((a + 1 + i) % m.n_species, a, a)[i % 3]
        if i % 3 == 2:
            m.reac[j, 1] = a
        m.n_reac[j] = 3
        m.A[j] *= 1e-11
    return m


MECHS = {"small": synth.mechanism_small,
         "s50": lambda: synth.random_mechanism(50, 130, 40, 13, name="synthetic_50sp_130rx"),
         "tropo": synth.mechanism_tropo,
         # 128 species and as many reactions as two groups' tiles of 32 cells leave room for
         "s128": lambda: synth.random_mechanism(128, 320, 100, 34, name="synthetic_128sp_320rx")}


def _workload(name, n, seed=41):
    m = _third_order(MECHS[name]())
    cells = synth.random_cells(m.n_species, n, T_range=(220.0, 310.0), P_range=(2e4, 1e5), seed=seed)
    return synth.Workload(m.name + "_3rd", m, cells, 600.0, 1, 1e-4, 1e-10)


# too few cells for a tile, with 1, 3 and 7 per block (3 and 7 do not divide its threads);
# one round of 32 cells on every SM and its edges; a ragged rest
@pytest.mark.parametrize("name", list(MECHS))
@pytest.mark.parametrize("rounds,rest", [(0, 1), (0, 33), (0, 437), (0, 1063), (1, -1), (1, 1), (1, 437), (1, 3333),
                                         (2, 271)])
def test_tiles_equal_the_f_program(oracle_lib, cg, name, rounds, rest):
    prop = torch.cuda.get_device_properties(0)
    n = rounds * 32 * prop.multi_processor_count + rest
    wl = _workload(name, n)
    m = wl.mech
    optin = getattr(prop, "shared_memory_per_block_optin", 232448)
    assert 2 * 32 * 8 * (m.n_species + m.n_reactions) <= optin - 1024      # the tiles fit: a round and more uses them
    y = wl.cells.y.copy()
    y[::7, ::3] = 0.0            # zero rates of either sign
    y[3::11, 1::5] *= -1.0
    c = cg.Cells(cg.Mechanism(m), n)
    c.set_state(wl.cells.T, wl.cells.P, y)
    ref = c.eval_deriv(y)
    got = c.eval_deriv_design(cg.DERIV_GATHER, y)
    assert np.array_equal(got.view(np.int64), ref.view(np.int64))
    for k in (0, n // 2, n - 1):
        kt = oracle_lib.rate_constants(m, wl.cells.T[k], wl.cells.P[k])
        J = oracle_lib.jacobian(m, kt, y[:, k])
        fo = oracle_lib.deriv(m, kt, y[:, k])
        # rate constants (a few ulp of |Ea/T| and their products) and the order of the sums
        assert np.all(np.abs(got[:, k] - fo) <= 1e-13 * (np.abs(J) @ np.abs(y[:, k]) + 1e-300))
    c.close()


@pytest.mark.parametrize("name", list(MECHS))
@pytest.mark.parametrize("prec", [64, 32])
def test_newton_solve_matches_dense(oracle_lib, cg, name, prec):
    wl = _workload(name, 9)
    m, cells = wl.mech, wl.cells
    c = cg.Cells(cg.Mechanism(m), 9, lu_precision=prec)
    c.set_state(cells.T, cells.P, cells.y)
    b = np.random.default_rng(3).standard_normal(cells.y.shape)
    tol = 1e-9 if prec == 64 else 2e-4
    for cc in (1e-3, 1.0, 30.0):
        x = c.eval_newton_solve(cc, cells.y, b)
        for k in range(9):
            kt = oracle_lib.rate_constants(m, cells.T[k], cells.P[k])
            Mk = np.eye(m.n_species) - cc * oracle_lib.jacobian(m, kt, cells.y[:, k])
            xr = np.linalg.solve(Mk, b[:, k])
            res = np.linalg.norm(Mk @ x[:, k] - b[:, k], np.inf)
            assert res <= tol * (np.linalg.norm(Mk, np.inf) * np.linalg.norm(xr, np.inf) + np.linalg.norm(b[:, k], np.inf))
    c.close()


@pytest.mark.parametrize("name", list(MECHS))
def test_solve_matches_oracle(oracle_lib, cg, name):
    from parity_util import compare
    wl = _workload(name, 61)
    yo, so = oracle_lib.solve_cells(wl.mech, wl.cells, wl.dt, wl.rtol, wl.atol)
    mech = cg.Mechanism(wl.mech)
    first = None
    for driver in ("plain", "persistent"):
        y, st = cg.solve(mech, wl.cells, wl.dt, wl.rtol, wl.atol, driver=driver)
        compare(y, st, yo, so, oracle_lib, wl, wl.cells, max_odd_frac=0.1, tight_flips=True, label=f"third order {name} {driver}")
        if first is None:
            first = y
        assert np.array_equal(y, first)


@pytest.mark.parametrize("name,n_steps", [("small", 2), ("tropo", 2), ("s128", 1)])
def test_adjoint_and_tangent_match_oracle(oracle_lib, cg, name, n_steps):
    wl = _workload(name, 5)
    m, cells = wl.mech, wl.cells
    c = cg.Cells(cg.Mechanism(m), 5, rtol=wl.rtol, atol=wl.atol, record_adjoint=True)
    c.set_state(cells.T, cells.P, cells.y)
    for _ in range(n_steps):
        c.solve_step(wl.dt)
    rng = np.random.default_rng(21)
    dy0, dth = rng.standard_normal(cells.y.shape) * cells.y, rng.standard_normal(m.n_reactions)
    w = synth.loss_weights(m.n_species, 5)
    dy, n_bad = c.tangent(dy0, dth)
    assert n_bad == 0
    gth, gy0, n_bad = c.sensitivity(w)
    assert n_bad == 0
    g_sum = np.zeros(m.n_reactions)
    for k in range(5):
        kind, q, val, rows = c.get_tape(k)
        y = np.zeros((kind.size, rows.shape[1]))
        y[(kind == 0) | (kind == 4) | (kind == 5)] = rows
        tape = oracle_lib.Tape(kind.astype(np.int32), q.astype(np.int32), val.astype(np.float64), y)
        kt = oracle_lib.rate_constants(m, cells.T[k], cells.P[k])
        ref = oracle_lib.tangent(m, kt, cells.y[:, k], tape, dy0[:, k], dth)
        assert np.all(np.abs(dy[:, k] - ref) <= 1e-8 * np.abs(ref) + 1e-12 * np.abs(ref).max()), k
        ly0, g = oracle_lib.adjoint(m, kt, cells.y[:, k], tape, w[:, k])
        g_sum += g
        assert np.all(np.abs(gy0[:, k] - ly0) <= 1e-8 * np.abs(ly0) + 1e-12 * np.abs(ly0).max()), k
    assert np.all(np.abs(gth - g_sum) <= 1e-8 * np.abs(g_sum) + 1e-12 * np.abs(g_sum).max())
    c.close()
