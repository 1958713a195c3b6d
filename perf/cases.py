"""What the solver library is timed on: one pass each through the calls a host model makes.

A chemistry model calls the library once (or a few times) per time step for
all of its grid cells: the batched solve of the Newton systems, its adjoint
for sensitivities, the FP32-inner refinement, the fused assembly + solve, the
whole Newton corrector, several mechanisms at once, or the solve of arrays
that live in host memory.  Mechanisms and cell states are drawn as the
benchmark's workloads are (mass-action mechanisms, concentrations log-uniform
in [1e-12, 1e-3], gamma log-uniform, right-hand sides N(0, 1)); the cells are
generated on the GPU from the seed, the mechanism belongs to the case.
"""
import functools
import math

import numpy as np
import torch

import synth
from paper_2405_17363_gb300 import camp

TOL, MAXIT = 1e-10, 500

# value ranges of the cells, by regime: rate constants (log10), gamma, concentrations
REGIMES = {
    "step": ((-6.0, 2.0), (1e-4, 1e-1), (1e-12, 1e-3)),    # a transport model's step (workloads 1, 3, 4)
    "long": ((-6.0, 2.0), (1e-4, 1.0), (1e-12, 1e-3)),     # longer steps, wider spread (workload 2)
    "hard": ((-4.0, 4.0), (1e-2, 10.0), (1e-3, 1.0)),      # stiff, strongly coupled cells (workload 5)
}
# about how many BiCGSTAB iterations a cell takes (for the operation counts)
ITERATIONS = {"step": 3.3, "long": 3.5, "hard": 51.0}


def listed():
    return [
        # one column of a small mechanism: the smallest call a model makes (latency)
        {"name": "solve_30sp_64", "kind": "solve", "n": 30, "R": 60, "cells": 64, "regime": "step", "mech": 1000},
        # one node's tile of a regional model on the intermediate mechanism: latency and launch count
        {"name": "solve_80sp_600", "kind": "solve", "n": 80, "R": 200, "cells": 600, "regime": "step", "mech": 1001},
        # the benchmark's batch: 10,000 cells of the intermediate mechanism
        {"name": "solve_80sp_10000", "kind": "solve", "n": 80, "R": 200, "cells": 10000, "regime": "step", "mech": 1001},
        # a reduced mechanism and a ragged batch, warm-started from the last step's solution
        {"name": "solve_guess_57sp_4001", "kind": "solve", "n": 57, "R": 140, "cells": 4001, "regime": "long",
         "mech": 1057, "guess": True},
        # stiff cells (sunrise, fresh emissions): tens to hundreds of iterations per cell
        {"name": "solve_hard_80sp_4000", "kind": "solve", "n": 80, "R": 200, "cells": 4000, "regime": "hard", "mech": 1005},
        # a large mechanism on a whole domain, all in FP64
        {"name": "solve_150sp_50000", "kind": "solve", "n": 150, "R": 400, "cells": 50000, "regime": "step", "mech": 1004},
        # the same by FP32-inner refinement to the same tolerance, the largest batch
        {"name": "mixed_150sp_100000", "kind": "mixed", "n": 150, "R": 400, "cells": 100000, "regime": "step", "mech": 1004},
        # sensitivities: forward solve, adjoint solve and the gradient of the matrix values
        {"name": "adjoint_80sp_10000", "kind": "adjoint", "n": 80, "R": 200, "cells": 10000, "regime": "step", "mech": 1003},
        # three mechanisms of different size in one call (uneven batching)
        {"name": "batch_40_80_150sp", "kind": "batch", "n": 40, "R": 90, "cells": 20000, "n2": 80, "R2": 200,
         "cells2": 5000, "n3": 150, "R3": 400, "cells3": 500, "regime": "long", "mech": 1002},
        # matrices assembled in the kernel from concentrations, then solved
        {"name": "assemble_80sp_10000", "kind": "assemble", "n": 80, "R": 200, "cells": 10000, "regime": "step", "mech": 1001},
        # the whole implicit step: rates, assembly and solve until Newton converges
        {"name": "newton_80sp_10000", "kind": "newton", "n": 80, "R": 200, "cells": 10000, "regime": "step", "mech": 1001},
        # a CPU host model's call: inputs and outputs in page-locked host memory
        {"name": "host_80sp_10000", "kind": "host", "n": 80, "R": 200, "cells": 10000, "regime": "step", "mech": 1001},
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more call: any kind, 21 to 160 species, a few cells to the largest batch of its kind."""
    kind = rng.choice(["solve", "solve", "solve", "mixed", "adjoint", "batch", "assemble", "newton", "host"])
    n = _spread(rng, 21, 160)
    case = {"kind": kind, "n": n, "R": int(n * rng.uniform(2.0, 2.7)), "regime": rng.choice(["step", "step", "long"]),
            "mech": rng.randrange(1 << 20)}
    if kind == "solve" and rng.random() < 0.3:
        case["regime"] = "hard"
        case["n"] = n = min(n, 110)
        case["R"] = int(n * rng.uniform(2.0, 2.7))
    if kind == "solve" and case["regime"] != "hard" and rng.random() < 0.3:
        case["guess"] = True
    # the most unknowns (cells x species) a call of the kind has here
    most = {"solve": 7.5e6, "mixed": 1.5e7, "adjoint": 1.6e6, "batch": 8e5, "assemble": 1.6e6, "newton": 8e5, "host": 1.6e6}[kind]
    if case["regime"] == "hard":
        most = 3.2e5
    top = max(64, int(most / n))
    case["cells"] = _spread(rng, 40, top)
    if kind == "batch":
        for q in ("2", "3"):
            case["n" + q] = m = _spread(rng, 21, 160)
            case["R" + q] = int(m * rng.uniform(2.0, 2.7))
            case["cells" + q] = _spread(rng, 20, max(64, int(4e5 / m)))
    return case


# ---- inputs ---------------------------------------------------------------

@functools.lru_cache(maxsize=64)
def _mechanism(n, R, seed, regime):
    """The mechanism, and its Jacobian as up to K terms per matrix entry (value, concentration factor)."""
    mech = synth.make_mechanism(n, R, seed, log10_k=REGIMES[regime][0])
    val = mech.contrib_sign * mech.k[mech.contrib_rxn]
    spec = np.where(mech.contrib_spec >= 0, mech.contrib_spec, n)   # column n of the factors is one
    order = np.argsort(mech.contrib_pos, kind="stable")
    pos = mech.contrib_pos[order]
    rank = np.arange(len(pos)) - np.searchsorted(pos, pos, side="left")
    K = int(rank.max()) + 1
    tv, ts = np.zeros((K, mech.nnz)), np.full((K, mech.nnz), n, dtype=np.int64)
    tv[rank, pos], ts[rank, pos] = val[order], spec[order]
    return mech, tv, ts


def _matrices(mech, tv, ts, conc, gamma):
    """A = I - gamma J for every cell, pattern order (a fixed order of sums)."""
    dev = conc.device
    tvd, tsd = torch.as_tensor(tv, device=dev), torch.as_tensor(ts, device=dev)
    diag = torch.as_tensor(mech.diag_pos(), device=dev)
    ext = torch.cat([conc, torch.ones(conc.shape[0], 1, dtype=conc.dtype, device=dev)], 1)
    A = torch.zeros(conc.shape[0], mech.nnz, dtype=torch.float64, device=dev)
    for c in range(0, conc.shape[0], 25000):
        part = A[c:c + 25000]
        for k in range(tv.shape[0]):
            used = torch.as_tensor(np.flatnonzero(tv[k]), device=dev)
            part[:, used] += ext[c:c + 25000][:, tsd[k][used]] * tvd[k][used]
        part *= -gamma[c:c + 25000, None]
        part[:, diag] += 1.0
    return A


def _cells(n, R, cells, regime, mech_seed, seed, dev="cuda"):
    """(mechanism, concentrations, gamma, b, generator): one batch of cells, from the seed."""
    mech, tv, ts = _mechanism(n, R, mech_seed, regime)
    _, gam, con = REGIMES[regime]
    g = torch.Generator(device=dev)
    g.manual_seed(seed)

    def log_uniform(shape, lo, hi):
        u = torch.rand(shape, dtype=torch.float64, device=dev, generator=g)
        return torch.exp(math.log(lo) + u * (math.log(hi) - math.log(lo)))

    conc = log_uniform((cells, n), *con)
    gamma = log_uniform((cells,), *gam)
    b = torch.randn((cells, n), dtype=torch.float64, device=dev, generator=g)
    return mech, tv, ts, conc, gamma, b, g


def _parts(case):
    """(n, R, cells, mechanism seed) of every mechanism of the case."""
    out = []
    for j, q in enumerate(("", "2", "3")):
        if "n" + q in case:
            out.append((case["n" + q], case["R" + q], case["cells" + q], case["mech"] + 10 * j))
    return out


def _inputs(case, seed):
    got = []
    for j, (n, R, cells, mech_seed) in enumerate(_parts(case)):
        mech, tv, ts, conc, gamma, b, g = _cells(n, R, cells, case["regime"], mech_seed, 7919 * seed + j)
        d = {"mech": mech, "conc": conc, "gamma": gamma, "b": b}
        if case["kind"] not in ("assemble", "newton"):
            d["A"] = _matrices(mech, tv, ts, conc, gamma)
        if case.get("guess"):
            d["x0"] = b + 0.1 * torch.randn(b.shape, dtype=torch.float64, device=b.device, generator=g)
        if case["kind"] == "adjoint":
            d["w"] = torch.randn(b.shape, dtype=torch.float64, device=b.device, generator=g)
        got.append(d)
    return got


def prepare(case, seed):
    parts = _inputs(case, seed)
    state = {"kind": case["kind"]}
    for d in parts:
        d["solver"] = camp.Solver(d["mech"].row_ptr, d["mech"].col_idx)
        if case["kind"] in ("assemble", "newton"):
            m = d["mech"]
            d["solver"].set_mechanism(m.reactants[:, 0], m.reactants[:, 1], m.products, m.k)
    if case["kind"] == "batch":
        state["batch"] = camp.Batch([d["solver"] for d in parts])
        state["A"] = [d["A"] for d in parts]
        state["b"] = [d["b"] for d in parts]
        state["parts"] = [d["solver"] for d in parts]
        return state
    d = parts[0]
    if case["kind"] == "host":
        cells, n = d["b"].shape
        state["solver"] = d["solver"]
        state["A"], state["b"] = (d[k].cpu().pin_memory() for k in ("A", "b"))
        state["out"] = [torch.empty(s, dtype=t).pin_memory() for s, t in (
            ((cells, n), torch.float64), ((cells,), torch.int32), ((cells,), torch.float64), ((cells,), torch.int32))]
        return state
    if case["kind"] == "adjoint":
        d["A"].requires_grad_(True)
        d["b"].requires_grad_(True)
    state.update({k: v for k, v in d.items() if k != "mech"})
    return state


def run(state):
    kind, s = state["kind"], state.get("solver")
    if kind == "solve":
        return s.solve(state["A"], state["b"], TOL, MAXIT, x0=state.get("x0"))
    if kind == "mixed":
        return s.solve_mixed(state["A"], state["b"], TOL)
    if kind == "adjoint":
        x, iters, resid, status = camp.solve(state["A"], state["b"], s, TOL, MAXIT)
        gA, gb = torch.autograd.grad(x, (state["A"], state["b"]), state["w"])
        return x.detach(), iters, resid, status, gA, gb
    if kind == "batch":
        return state["batch"].solve(state["A"], state["b"], TOL, MAXIT)
    if kind == "assemble":
        return s.assemble_solve(state["conc"], state["gamma"], state["b"], TOL, MAXIT)
    if kind == "newton":
        return s.newton_solve(state["conc"], state["gamma"], state["conc"])
    x, iters, resid, status = state["out"]
    camp.camp_solver_solve_host(s.h, x.shape[0], state["A"], state["b"], x, TOL, MAXIT, iters, resid, status)
    return x, iters, resid, status


# ---- what a pass cannot do without -----------------------------------------

def _nnz(n, R, mech_seed, regime):
    return _mechanism(n, R, mech_seed, regime)[0].nnz


def work(case):
    size = flops = 0
    for n, R, cells, mech_seed in _parts(case):
        nnz = _nnz(n, R, mech_seed, case["regime"])
        its = ITERATIONS[case["regime"]]
        kind = case["kind"]
        # one solve: staging, its iterations (two products, six dot products, six
        # updates, two scalings) and the true residual of the result
        solve = its * (4 * nnz + 26 * n) + 2 * nnz + 8 * n
        matrix = 8 * nnz
        if kind in ("assemble", "newton"):
            matrix = 8 * n + 8                       # concentrations and gamma
            solve += 2 * (R // 2 * 2 + (R - R // 2) * 6) + 2 * nnz
        per = matrix + 8 * n + 8 * n + 4 + 8 + 4      # b, x, iterations, residual, status
        if kind == "newton":
            solve = 2.5 * (solve + 8 * R)
            per = 8 * n + 8 + 2 * 8 * n + 4 + 4 + 8 + 8 + 4
        if kind == "adjoint":
            solve = 2 * solve + nnz
            per = 2 * 8 * nnz + 5 * 8 * n + 16
        if case.get("guess"):
            per += 8 * n
            solve += 2 * nnz
        size += cells * per
        flops += cells * solve
    return {"bytes": float(size), "flops": float(flops)}


# ---- the same in plain 64-bit arithmetic -------------------------------------

def _dense(mech, A, lo, hi):
    n = mech.n
    rows = torch.as_tensor(np.repeat(np.arange(n), np.diff(mech.row_ptr)), device=A.device)
    cols = torch.as_tensor(mech.col_idx.astype(np.int64), device=A.device)
    D = torch.zeros(hi - lo, n * n, dtype=torch.float64, device=A.device)
    D[:, rows * n + cols] = A[lo:hi]
    return D.view(hi - lo, n, n), rows, cols


def _solved(mech, A, b, transpose=False):
    x = torch.empty_like(b)
    for c in range(0, b.shape[0], 10000):
        hi = min(b.shape[0], c + 10000)
        D, _, _ = _dense(mech, A, c, hi)
        x[c:hi] = torch.linalg.solve(D.transpose(1, 2) if transpose else D, b[c:hi])
    return x


def _rates(mech, conc):
    f = torch.zeros_like(conc)
    for r in range(mech.R):
        a, b2 = (int(v) for v in mech.reactants[r])
        w = float(mech.k[r]) * conc[:, a] * (conc[:, b2] if b2 >= 0 else 1.0)
        f[:, a] -= w
        if b2 >= 0:
            f[:, b2] -= w
        f[:, int(mech.products[r])] += w
    return f


def exact(case, seed):
    got, kind = [], case["kind"]
    for j, d in enumerate(_inputs(case, seed)):
        mech, b = d["mech"], d["b"]
        tables = _mechanism(mech.n, mech.R, _parts(case)[j][3], case["regime"])[1:]
        if kind == "newton":
            y = d["conc"].clone()
            for _ in range(6):
                G = y - d["gamma"][:, None] * _rates(mech, y) - d["conc"]
                y -= _solved(mech, _matrices(mech, *tables, y, d["gamma"]), G)
            return {"y": y, "newton_iters": None, "lin_iters": None, "upd": None, "resid": None, "status": None}
        A = d["A"] if "A" in d else _matrices(mech, *tables, d["conc"], d["gamma"])
        x = _solved(mech, A, b)
        if kind == "mixed":
            return x, None, None, None, None
        if kind == "adjoint":
            lam = _solved(mech, A, d["w"], transpose=True)
            _, rows, cols = _dense(mech, A, 0, 1)
            return x, None, None, None, -lam[:, rows] * x[:, cols], lam
        got.append((x, None, None, None))
    return got if kind == "batch" else got[0]
