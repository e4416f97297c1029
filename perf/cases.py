"""The calls this library is used for, as cases that can be timed and compared.

A case is a dict of plain values; prepare() makes its inputs from a seed, run() is one
pass through the public binding (paper_2501_00011_gb300.chemgpu) as a model's program
makes it, with the state on the device unless the path works on host memory.

Kinds:
  solve     a new state into the batch, one solve_step, the state out
  steps     the same with n consecutive steps as one CUDA graph (solve_steps)
  grad      forward with tape through solve_with_grad and the gradient of a weighted
            sum of the final concentrations (discrete adjoint)
  tangent   the directional derivative along a recorded run (one direction of many)
  deriv     f(y) of the whole batch (the derivative kernel, rate constants kept)
  pipeline  host-resident state in chunks (Pipeline.run), copies and solves overlapped
"""
import math

import numpy as np
import torch

from paper_2501_00011_gb300 import chemgpu, synth

DT = 600.0                       # s, the chemistry step of every workload here

# mechanisms: this repository's workloads and the other sizes its tests use
_MAKE = {
    "small": synth.mechanism_small,                 # 20 species / 40 reactions
    "s50": lambda: synth.random_mechanism(50, 130, 40, 13, name="synthetic_50sp_130rx"),
    "tropo": synth.mechanism_tropo,                 # 72 / 186
    "pressure": synth.mechanism_tropo_pressure,     # 72 / 186, fall-off rate laws
    "s128": lambda: synth.random_mechanism(128, 330, 100, 34, name="synthetic_128sp_330rx"),
}
_compiled = {}                   # a program compiles its mechanism once and keeps it
_tables = {}


def _table(name):
    if name not in _tables:
        _tables[name] = _MAKE[name]()
    return _tables[name]


def _mechanism(name):
    if name not in _compiled:
        _compiled[name] = chemgpu.Mechanism(_table(name))
    return _compiled[name]


def listed():
    return [
        # a box model: ten cells of a small mechanism at tight tolerances, default driver
        {"name": "box_10", "kind": "solve", "mech": "small", "cells": 10, "driver": "plain", "rtol": 1e-8, "atol": 1e-14},
        # a few columns: a small, odd batch that leaves most of the chip without a cell of its own
        {"name": "columns_301", "kind": "solve", "mech": "tropo", "cells": 301, "driver": "persistent"},
        # the headline: one step of a fresh 10,000-cell batch
        {"name": "batch_10k", "kind": "solve", "mech": "tropo", "cells": 10000, "driver": "persistent"},
        # the same through the plain driver, the binding's default
        {"name": "plain_10k", "kind": "solve", "mech": "tropo", "cells": 10000, "driver": "plain"},
        # the same with the iteration matrix factored and solved in FP32
        {"name": "fp32lu_10k", "kind": "solve", "mech": "tropo", "cells": 10000, "driver": "persistent", "lu": 32},
        # a step of a running model: the state is past its initial transient, steps are few and cheap
        {"name": "running_10k", "kind": "solve", "mech": "tropo", "cells": 10000, "driver": "persistent", "spinup": 1},
        # pressure-dependent rate laws, an odd batch
        {"name": "pressure_3001", "kind": "solve", "mech": "pressure", "cells": 3001, "driver": "persistent"},
        # an hour of 50,000 cells with day and night photolysis as one graph
        {"name": "hour_50k", "kind": "steps", "mech": "tropo", "cells": 50000, "n_steps": 6, "photolysis": True},
        # a training step: four recorded steps forward, discrete adjoint back
        {"name": "grad_2k", "kind": "grad", "mech": "tropo", "cells": 2048, "n_steps": 4},
        # one forward-mode direction along a recorded run of four steps
        {"name": "tangent_2k", "kind": "tangent", "mech": "tropo", "cells": 2048, "n_steps": 4},
        # the derivative alone, as an operator-split or diagnostic call uses it
        {"name": "deriv_10k", "kind": "deriv", "mech": "tropo", "cells": 10000},
        # a host model that owns the state: pinned memory in and out, four chunks, day and night
        {"name": "pipeline_10k", "kind": "pipeline", "mech": "tropo", "cells": 10000, "chunks": 4, "photolysis": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Another case of the same ranges: batch sizes over their logarithm, any of the
    mechanisms, drivers and precisions, day or night photolysis, running or fresh states."""
    kind = rng.choice(["solve", "solve", "solve", "solve", "steps", "grad", "tangent", "deriv", "pipeline"])
    mech = rng.choice(["small", "s50", "tropo", "tropo", "pressure", "s128"])
    case = {"kind": kind, "mech": mech}
    if kind == "solve":
        case["cells"] = _log_int(rng, 5, 2000 if mech == "s128" else 20000)
        case["driver"] = rng.choice(["plain", "persistent", "persistent"])
        case["photolysis"] = rng.random() < 0.5
        case["spinup"] = int(rng.random() < 0.4)
        if rng.random() < 0.3:
            case["lu"] = 32
        elif mech == "small" and rng.random() < 0.5:
            case["rtol"], case["atol"] = 1e-8, 1e-14
    elif kind == "steps":
        case["cells"] = _log_int(rng, 50, 1000 if mech == "s128" else 20000)
        case["n_steps"] = rng.randint(2, 6)
        case["photolysis"] = rng.random() < 0.5
    elif kind in ("grad", "tangent"):
        case["cells"] = _log_int(rng, 10, 300 if mech == "s128" else 2500)
        case["n_steps"] = rng.randint(1, 4)
        case["photolysis"] = rng.random() < 0.5
    elif kind == "deriv":
        case["cells"] = _log_int(rng, 200, 200000)
    else:
        case["cells"] = _log_int(rng, 100, 1000 if mech == "s128" else 12000)
        case["chunks"] = rng.randint(1, 6)
        case["photolysis"] = rng.random() < 0.5
    return case


def _inputs(case, seed):
    """T, P, y (and photolysis J, or None) as the workloads draw them, on the host."""
    m, n = _table(case["mech"]), case["cells"]
    rng = np.random.Generator(np.random.PCG64([seed, n]))
    lo, hi = {"small": (250.0, 300.0), "pressure": (200.0, 310.0)}.get(case["mech"], (220.0, 310.0))
    if case.get("photolysis"):
        lo, hi = 200.0, 320.0
    T = rng.uniform(lo, hi, n)
    p_lo, p_hi = {"small": (1e5, 1e5), "pressure": (1e3, 1.05e5)}.get(case["mech"], (2e4, 1e5))
    P = np.exp(rng.uniform(math.log(p_lo), math.log(p_hi), n)) if p_lo < p_hi else np.full(n, p_lo)
    y = np.exp(rng.uniform(math.log(1e-12), math.log(1e-6), (m.n_species, n)))
    J = None
    if case.get("photolysis"):
        s = 1.0 - rng.uniform(0.0, 1.0, n)
        s[rng.random(n) < 0.3] = 0.0                 # night
        J = np.ascontiguousarray(m.J[m.photolysis_index][:, None] * s[None, :])
    return T, P, y, J


def _gpu(a):
    return None if a is None else torch.from_numpy(a).cuda()


def _cells(case, **kw):
    return chemgpu.Cells(_mechanism(case["mech"]), case["cells"], rtol=case.get("rtol", 1e-4),
                         atol=case.get("atol", 1e-10), driver=case.get("driver", "persistent"),
                         lu_precision=case.get("lu", 64), **kw)


def prepare(case, seed):
    m, kind = _table(case["mech"]), case["kind"]
    T, P, y, J = _inputs(case, seed)
    st = {"case": case}
    if kind == "pipeline":
        for k, a in (("T", T), ("P", P), ("y0", y), ("J", J)):
            st[k] = None
            if a is not None:
                st[k] = chemgpu.pinned_empty(a.shape)
                st[k][...] = a
        st["y"] = chemgpu.pinned_empty(y.shape)
        st["pipe"] = chemgpu.Pipeline(_mechanism(case["mech"]), case["cells"], case["chunks"])
        return st
    st["T"], st["P"], st["y"], st["J"] = _gpu(T), _gpu(P), _gpu(y), _gpu(J)
    st["out"] = torch.empty_like(st["y"])
    if kind in ("grad", "tangent"):
        # a 600 s step records some 150 rows; room for the initial transient and the steps after it
        st["cells"] = _cells(case, record_adjoint=True, tape_steps=2000)
    else:
        st["cells"] = _cells(case)
    if st["J"] is not None:
        st["cells"].set_photolysis(st["J"])
    rng = np.random.Generator(np.random.PCG64([seed, 7]))
    if kind == "solve" and case.get("spinup"):
        spin = _cells(case)
        if st["J"] is not None:
            spin.set_photolysis(st["J"])
        spin.set_state(st["T"], st["P"], st["y"])
        for _ in range(case["spinup"]):
            spin.solve_step(DT)
        spin.get_state(out=st["y"])
        torch.cuda.synchronize()
        spin.close()
    elif kind == "grad":
        st["theta"] = _gpu(rng.normal(0.0, 0.05, m.n_reactions)).requires_grad_(True)
        st["y"].requires_grad_(True)
        st["weights"] = _gpu(rng.uniform(0.0, 1.0, y.shape))
    elif kind == "tangent":
        st["cells"].set_state(st["T"], st["P"], st["y"])
        for _ in range(case["n_steps"]):
            st["cells"].solve_step(DT)
        st["dy0"] = _gpu(y * rng.normal(0.0, 1.0, y.shape))
        st["dtheta"] = _gpu(rng.normal(0.0, 1.0, m.n_reactions))
    elif kind == "deriv":
        st["cells"].set_state(st["T"], st["P"], st["y"])
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "pipeline":
        st["y"][...] = st["y0"]
        stats = st["pipe"].run(st["T"], st["P"], st["y"], DT, J=st["J"], stats=True)
        return {"y": st["y"], "status": stats["status"], "steps": stats["steps"]}
    c = st["cells"]
    if kind == "solve":
        c.set_state(st["T"], st["P"], st["y"])
        c.solve_step(DT)
        return c.get_state(out=st["out"])
    if kind == "steps":
        c.set_state(st["T"], st["P"], st["y"])
        c.solve_steps(DT, case["n_steps"])
        return c.get_state(out=st["out"])
    if kind == "grad":
        y = chemgpu.solve_with_grad(c, st["theta"], st["y"], st["T"], st["P"], DT, n_steps=case["n_steps"])
        gth, gy0 = torch.autograd.grad((st["weights"] * y).sum(), (st["theta"], st["y"]))
        return {"y": y.detach(), "dtheta": gth, "dy0": gy0}
    if kind == "tangent":
        dy, n_bad = c.tangent(st["dy0"], st["dtheta"], dy=st["out"])
        return {"dy": dy, "n_bad": n_bad}
    return c.eval_deriv_design(chemgpu.DERIV_GATHER, st["y"], out=st["out"])


def work(case):
    """Bytes: each input read and each output written once.  Flops: the arithmetic of the
    path at the step, Newton and factorisation counts typical of the workload (a fresh
    600 s step: about 85 steps, 118 iterations, 26 factorisations per cell; a running one
    11, 17 and 7), from the mechanism's own per-operation counts."""
    m, n = _table(case["mech"]), case["cells"]
    S, R = m.n_species, m.n_reactions
    reac = float(m.n_reac.sum())
    nu = float(m.n_reac.sum() + m.n_prod.sum())
    f = reac + 2.0 * nu
    lu, solve = 250.0 * S, 40.0 * S                  # sparse factorisation and its solves (72 species: 18.8k, 2.9k)
    jac = 2.0 * reac + 2.0 * nu * reac / max(R, 1)
    fresh = 120 * f + 26 * (lu + jac) + 118 * solve + 118 * 8 * S + 85 * 17 * S
    running = 18 * f + 7 * (lu + jac) + 17 * solve + 17 * 8 * S + 11 * 13 * S
    if case.get("rtol", 1e-4) < 1e-6:
        fresh, running = 3.5 * fresh, 3.5 * running  # tight tolerances: that many more steps
    state = 8.0 * n * (2 * S + 2 + (len(m.photolysis_index) if case.get("photolysis") else 0))
    kind = case["kind"]
    if kind == "deriv":
        return {"bytes": 8.0 * n * (2 * S + R), "flops": n * f}
    if kind in ("solve", "pipeline"):
        return {"bytes": state, "flops": n * (running if case.get("spinup") else fresh)}
    steps = fresh + (case["n_steps"] - 1) * running
    if kind == "steps":
        return {"bytes": state, "flops": n * steps}
    walk = 0.8 * steps                               # a walk along the tape: about the forward's solves and factorisations
    return {"bytes": 2.0 * state + 8.0 * R, "flops": n * (steps + walk if kind == "grad" else walk)}


# ---------------------------------------------------------------- 64-bit values
def _rates(m, T, P, J):
    """k [R, C] from the reaction tables (mixing-ratio units), plain numpy."""
    ext = synth.rate_ext(m)
    n_air = P / (1.380649e-23 * T) * 1e-6
    arr = lambda A, E, B: A * np.exp(-E / T) * (T / 300.0) ** B  # noqa: E731
    k = np.empty((m.n_reactions, T.size))
    photo = {int(j): i for i, j in enumerate(m.photolysis_index)}
    for j in range(m.n_reactions):
        if m.kind[j] == synth.PHOTOLYSIS:
            k[j] = m.J[j] if J is None else J[photo[j]]
            continue
        kj, e = arr(m.A[j], m.Ea[j], m.B[j]), ext[j]
        if m.kind[j] == synth.TROE:
            x = kj * n_air / arr(e[0], e[1], e[2])
            kj = kj * n_air / (1.0 + x) * e[6] ** (1.0 / (1.0 + (np.log10(x) / e[7]) ** 2))
        elif m.kind[j] == synth.PRESSURE_SUM:
            kj = kj + arr(e[0], e[1], e[2]) * n_air
        elif m.kind[j] == synth.FALLOFF_SUM:
            c = arr(e[3], e[4], e[5]) * n_air
            kj = kj + c / (1.0 + c / arr(e[0], e[1], e[2]))
        k[j] = kj * n_air ** (int(m.n_reac[j]) - 1)
    return k


def _deriv(m, k, y):
    f = np.zeros_like(y)
    for j in range(m.n_reactions):
        r = k[j].copy()
        for s in m.reac[j, :m.n_reac[j]]:
            r *= y[s]
        for s in m.reac[j, :m.n_reac[j]]:
            f[s] -= r
        for p, v in zip(m.prod[j, :m.n_prod[j]], m.yld[j, :m.n_prod[j]]):
            f[p] += v * r
    return f


def _jacobian(m, k, y):
    S, C = y.shape
    Jm = np.zeros((C, S, S))
    for j in range(m.n_reactions):
        reac = [int(s) for s in m.reac[j, :m.n_reac[j]]]
        for i, l in enumerate(reac):
            d = k[j].copy()
            for i2, s in enumerate(reac):
                if i2 != i:
                    d = d * y[s]
            for s in reac:
                Jm[:, s, l] -= d
            for p, v in zip(m.prod[j, :m.n_prod[j]], m.yld[j, :m.n_prod[j]]):
                Jm[:, int(p), l] += v * d
    return Jm


def _integrate(m, k, y0, dt, n_steps=900):
    """y(dt) by the three-stage Radau IIA method (order 5) on a geometric time grid."""
    S, C = y0.shape
    s6 = math.sqrt(6.0)
    A = np.array([[(88 - 7 * s6) / 360, (296 - 169 * s6) / 1800, (-2 + 3 * s6) / 225],
                  [(296 + 169 * s6) / 1800, (88 + 7 * s6) / 360, (-2 - 3 * s6) / 225],
                  [(16 - s6) / 36, (16 + s6) / 36, 1.0 / 9.0]])
    t = np.concatenate([[0.0], np.geomspace(1e-7, dt, n_steps)])
    y, eye = y0.copy(), np.eye(3 * S)
    for h in np.diff(t):
        M = eye - h * np.einsum("ij,cab->ciajb", A, _jacobian(m, k, y)).reshape(C, 3 * S, 3 * S)
        Mi = np.linalg.inv(M)
        z = np.zeros((3, S, C))
        for _ in range(4):
            F = np.stack([_deriv(m, k, y + z[i]) for i in range(3)])
            res = h * np.einsum("ij,jsc->isc", A, F) - z
            z = z + np.einsum("cab,bc->ac", Mi, res.reshape(3 * S, C)).reshape(3, S, C)
        y = y + z[2]
    return y


def exact(case, seed):
    m = _table(case["mech"])
    if case["kind"] == "deriv":
        T, P, y, J = _inputs(case, seed)
        return torch.from_numpy(_deriv(m, _rates(m, T, P, J), y))
    if case["kind"] == "solve" and case["mech"] == "small" and case["cells"] <= 12 and not case.get("spinup"):
        T, P, y, J = _inputs(case, seed)
        return torch.from_numpy(_integrate(m, _rates(m, T, P, J), y, DT))
    return None          # a tight stiff integration of these batches takes minutes on the host
