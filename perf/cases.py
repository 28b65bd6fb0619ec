"""The work that a circuit simulator has this library do, as measurable cases.

A case is one circuit (a generator of ``paper_2411_14082_gb300.inputs`` with
its sizes; ``topo`` seeds the topology) and one way of using the library on
it.  The seed of ``prepare`` draws the element values and the right-hand
sides, so another seed is another operating point of the same circuit, as
between the Newton iterations, time steps or corners of a simulation.

Kinds (the public entry points a pass goes through):
  newton   checked re-factorization and solve on device buffers, by two
           calls (``entry`` "calls") or one replayed graph ("step"), or the
           whole step from host buffers ("host");
  solve    the two triangular solves alone (a linear transient analysis
           factorizes once and solves every time step);
  batch    many value sets of one circuit (corners, Monte Carlo) at once;
  multi    circuits of different sizes in one launch;
  mixed    single-precision factors with double-precision refinement;
  first    the first factorization (structure, schedule, factors) and solve;
  serve    a burst of requests from concurrent simulations to the server.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2411_14082_gb300 import gblu, inputs

DEVICE = 0


# ------------------------------------------------------------------ circuits
@functools.lru_cache(maxsize=64)
def _circuit(gen, nx, ny, nz, extra, topo):
    """(circuit, n, Ap, Ai, Q) of one topology; Q is the library's own order."""
    if gen == "mna":            # 2D resistor grid, couplings, voltage sources (zero diagonals)
        ckt = inputs.mna_grid2d(nx, ny, seed=topo, n_vsrc=extra)
    elif gen == "mesh":         # post-layout RC mesh with transistor stamps
        ckt = inputs.rc_mesh3d(nx, ny, nz, seed=topo, n_fet=extra)
    else:                       # grid with dense-ish power and ground rails
        ckt = inputs.bordered_grid(nx, ny, n_rails=extra, seed=topo)
    n, Ap, Ai, _ = ckt.csc()
    Q, _ = gblu.order_auto(n, Ap, Ai)
    return ckt, n, Ap, Ai, Q


def _parts(case):
    """The circuits of a case: one, or for multi and serve a spread of sizes."""
    gen, extra, topo = case["gen"], case["extra"], case["topo"]
    count = case.get("count", 1)
    if case["kind"] not in ("multi", "serve"):
        return [(gen, case["nx"], case["ny"], case["nz"], extra, topo)]
    parts = []
    for i in range(count):   # side lengths spread over their logarithm, none alike
        f = i / max(1, count - 1)
        side = case["nx"] * (case["ny"] / case["nx"]) ** f
        a = max(8, int(side) + (i % 3))
        b = max(8, int(side * (1.0 + 0.13 * (i % 4))))
        parts.append((gen, a, b, case["nz"], max(4, int(extra * side / case["ny"])), topo + i))
    return parts


def _values(ckt, rng, sigma):
    """Element values of one operating point: every conductance and shunt
    times a log-normal factor, new transconductances."""
    out = ckt.copy()
    out.res_g = out.res_g * np.exp(rng.normal(0.0, sigma, len(out.res_g)))
    out.shunt = out.shunt * np.exp(rng.normal(0.0, sigma, len(out.shunt)))
    if len(out.vccs_gm):
        out = inputs.redraw_transistors(out, rng)
    return out.values()


def _step_values(ckt, rng):
    """The next Newton iteration's values: new transistor values on a mesh,
    a few changed conductances otherwise."""
    if len(ckt.vccs_gm):
        return inputs.redraw_transistors(ckt, rng).values()
    return inputs.perturb_elements(ckt, rng).values()


def _draw_inputs(case, seed):
    """Host values and right-hand sides of a case, made from the seed alone:
    per circuit (first values, values [nsets, nnz], b [nsets, n])."""
    rng = np.random.default_rng([int(seed), 14082])
    got = []
    for part in _parts(case):
        ckt, n, Ap, Ai, Q = _circuit(*part)
        if case["kind"] == "batch":
            sets = case["sets"]
            Ax = np.stack([_values(ckt, rng, math.log(1.2)) for _ in range(sets)])
            b = rng.uniform(-1.0, 1.0, (sets, n))
        elif case["kind"] == "serve":
            sets = case["sets"]
            Ax = np.stack([_step_values(ckt, rng) for _ in range(sets)])
            b = rng.uniform(-1.0, 1.0, (sets, n))
        else:
            Ax = _step_values(ckt, rng)[None]
            b = rng.uniform(-1.0, 1.0, (1, n))
        got.append((ckt.values(), Ax, b))
    return got


# --------------------------------------------------------------------- cases
def _case(name, kind, gen, nx, ny, nz=1, extra=0, topo=20241121, **more):
    return dict(name=name, kind=kind, gen=gen, nx=nx, ny=ny, nz=nz, extra=extra, topo=topo, **more)


def listed():
    return [
        # a small analog block in a Newton loop: the smallest ordinary call
        _case("newton_mna_2k", "newton", "mna", 40, 50, extra=20, entry="calls"),
        # a mid-size circuit, odd grid, whole step replayed as one graph
        _case("step_mna_10k", "newton", "mna", 101, 97, extra=53, topo=7, entry="step"),
        # a small post-layout net whose simulator keeps its vectors on the host
        _case("host_mesh_11k", "newton", "mesh", 53, 53, 4, extra=141, topo=11, entry="host"),
        # a block-level power mesh, one Newton iteration per pass
        _case("newton_mesh_48k", "newton", "mesh", 110, 109, 4, extra=600, topo=5, entry="calls"),
        # the post-layout power mesh: the largest single system
        _case("newton_mesh_160k", "newton", "mesh", 200, 200, 4, extra=2000, topo=20241122, entry="calls"),
        # linear transient analysis: one factorization, a solve per time step
        _case("solve_mesh_90k", "solve", "mesh", 150, 150, 4, extra=1100, topo=3),
        # Monte-Carlo corners of a net with power and ground rails
        _case("batch_rails_20k", "batch", "bordered", 141, 141, extra=50, topo=20241123, sets=256),
        # corners of a small net: many tiny systems
        _case("batch_grid_1k", "batch", "mesh", 37, 31, 1, extra=17, topo=9, sets=96),
        # subcircuits of different sizes solved together every iteration
        _case("multi_mna_1k_25k", "multi", "mna", 32, 150, extra=60, topo=31, count=20),
        # the mesh with single-precision factors and refinement
        _case("mixed_mesh_58k", "mixed", "mesh", 120, 120, 4, extra=720, topo=13),
        # the first factorization of a netlist that has to pivot
        _case("first_mna_5k", "first", "mna", 71, 69, extra=35, topo=17),
        # a burst of requests from concurrent simulations
        _case("serve_mesh", "serve", "mesh", 30, 100, 4, extra=400, topo=23, count=4, sets=6),
    ]


def draw(rng):
    def side(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["newton", "newton", "newton", "solve", "batch", "multi", "mixed", "first", "serve"])
    topo = rng.randrange(1, 1 << 20)
    if kind in ("newton", "solve", "mixed"):
        gen = "mesh" if kind == "mixed" else rng.choice(["mna", "mesh", "bordered"])
        entry = {"entry": rng.choice(["calls", "step", "host"])} if kind == "newton" else {}
        if gen == "mna":
            a = side(32, 160)
            b = max(8, int(a * rng.uniform(0.7, 1.2)))
            extra, nz = max(4, a * b // 150), 1
        elif gen == "mesh":
            a, nz = side(16, 180), rng.choice([1, 3, 4])
            b = max(8, int(a * rng.uniform(0.7, 1.1)))
            extra = max(4, a * b // 20)
        else:
            a, nz = side(32, 140), 1
            b = max(8, int(a * rng.uniform(0.7, 1.0)))
            extra = rng.randrange(8, 51)
        case = _case("", kind, gen, a, b, nz, extra, topo, **entry)
    elif kind == "batch":
        gen = rng.choice(["bordered", "mesh"])
        a = side(24, 120 if gen == "bordered" else 140)
        b = max(8, int(a * rng.uniform(0.7, 1.1)))
        extra = rng.randrange(8, 51) if gen == "bordered" else max(4, a * b // 60)
        case = _case("", kind, gen, a, b, 1, extra, topo, sets=side(4, 128))
    elif kind == "multi":
        case = _case("", kind, "mna", side(30, 50), side(60, 140), extra=rng.randrange(20, 61), topo=topo,
                     count=rng.randrange(3, 20))
    elif kind == "first":
        if rng.random() < 0.5:
            a = side(32, 75)
            case = _case("", kind, "mna", a, max(8, int(a * rng.uniform(0.7, 1.1))), extra=max(4, a // 2), topo=topo)
        else:
            a = side(24, 130)
            case = _case("", kind, "mesh", a, max(8, int(a * rng.uniform(0.7, 1.1))), 4, max(4, a * a // 20), topo)
    else:
        case = _case("", kind, "mesh", side(20, 40), side(50, 100), 4, rng.randrange(50, 400), topo,
                     count=rng.randrange(2, 5), sets=rng.randrange(2, 7))
    del case["name"]
    return case


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda(DEVICE)


def _solver(part, Ax0):
    _, n, Ap, Ai, Q = _circuit(*part)
    s = gblu.Solver(DEVICE)
    s.analyze(n, Ap, Ai, Q)
    if Ax0 is not None:
        s.factorize(_dev(Ax0))
    return s


def prepare(case, seed):
    kind, parts, host = case["kind"], _parts(case), _draw_inputs(case, seed)
    if kind == "serve":   # the server with its patterns; requests in pinned host memory
        srv = gblu.Server(DEVICE, hbm_budget=8 << 30, max_batch=8)
        jobs = []
        for part, (Ax0, Ax, b) in zip(parts, host):
            _, n, Ap, Ai, Q = _circuit(*part)
            pid, _ = srv.add_pattern(n, Ap, Ai, Q, Ax0)
            for i in range(case["sets"]):
                pin = [torch.from_numpy(v).pin_memory().numpy() for v in (Ax[i].copy(), b[i].copy(), np.zeros(n))]
                jobs.append((pid, *pin, i % 3 == 2))   # every third request in mixed precision
        return {"kind": kind, "server": srv, "jobs": jobs}
    state = {"kind": kind, "entry": case.get("entry")}
    solvers = [_solver(p, None if kind == "first" else Ax0) for p, (Ax0, _, _) in zip(parts, host)]
    state["solvers"] = solvers
    if kind == "newton" and case["entry"] == "host":
        state["host"] = [torch.from_numpy(v).pin_memory().numpy() for v in
                         (host[0][1][0].copy(), host[0][2][0].copy(), np.zeros(solvers[0].n))]
        return state
    if kind == "batch":
        s = solvers[0]
        st = s.stats()
        sets = case["sets"]
        state["Ax"], state["b"] = _dev(host[0][1]), _dev(host[0][2])
        state["x"] = torch.empty_like(state["b"])
        state["LUx"] = torch.empty((sets, st["nnz_l"] + st["nnz_u"]), dtype=torch.float64, device=f"cuda:{DEVICE}")
        return state
    state["Ax"] = [_dev(Ax[0]) for _, Ax, _ in host]
    state["b"] = [_dev(b[0]) for _, _, b in host]
    state["x"] = [torch.empty_like(b) for b in state["b"]]
    if kind == "solve":
        solvers[0].refactorize(state["Ax"][0])
    return state


def run(state):
    kind = state["kind"]
    if kind == "serve":
        srv = state["server"]
        ids = [srv.submit(pid, Ax, b, x, mixed) for pid, Ax, b, x, mixed in state["jobs"]]
        return [srv.wait(i)[0] for i in ids]
    s = state["solvers"][0]
    if kind == "newton" and state["entry"] == "host":
        Ax, b, x = state["host"]
        s.step_host(Ax, b, x)
        return x
    if kind == "batch":
        failed = s.step_batch(state["Ax"], state["LUx"], state["b"], state["x"])
        return {"x": state["x"], "failed": failed}
    if kind == "multi":
        gblu.refactorize_multi(state["solvers"], state["Ax"])
        return gblu.solve_multi(state["solvers"], state["b"], state["x"])
    Ax, b, x = state["Ax"][0], state["b"][0], state["x"][0]
    if kind == "newton":
        if state["entry"] == "step":
            return s.step(Ax, b, x)[0]
        s.refactorize(Ax)
        return s.solve(b, x)
    if kind == "solve":
        return s.solve(b, x)
    if kind == "mixed":
        s.refactorize_f32(Ax)
        return s.solve_refined(Ax, b, x)[0]
    s.factorize(Ax)               # kind == "first"
    return s.solve(b, x)


# ---------------------------------------------------------------------- work
def work(case):
    """Compulsory bytes and operations of one pass: A, b and the structure
    are read once, the factors written once and read once by the solves; the
    operations are those of the factorization and the solves, from the
    symmetric fill of the order (pivoting may add to it)."""
    nbytes = flops = 0.0
    for part in _parts(case):
        _, n, Ap, Ai, Q = _circuit(*part)
        fill, fl = gblu.symmetric_cost(n, Ap, Ai, Q)
        nnz, lu = float(Ap[-1]), 2.0 * fill + n
        sets = case.get("sets", 1)
        value = 4.0 if case["kind"] == "mixed" else 8.0
        solve_b = value * lu + 16.0 * n
        refac_b = 8.0 * nnz + value * lu
        index_b = 4.0 * (lu + nnz + n)
        if case["kind"] == "solve":
            nbytes += solve_b + index_b
            flops += 2.0 * lu
        else:
            nbytes += sets * (solve_b + refac_b) + index_b
            flops += sets * (fl + 2.0 * lu)
    return {"bytes": nbytes, "flops": flops}


# --------------------------------------------------------------------- exact
def _exact_x(n, Ap, Ai, Ax, b):
    """A x = b by dense LU in float64 with refinement on extended-precision
    residuals (numpy longdouble)."""
    col = np.repeat(np.arange(n), np.diff(Ap))
    rows = Ai.astype(np.int64)
    A = torch.zeros((n, n), dtype=torch.float64, device=f"cuda:{DEVICE}")
    A[torch.from_numpy(rows).cuda(DEVICE), torch.from_numpy(col).cuda(DEVICE)] = _dev(Ax)
    lu, piv = torch.linalg.lu_factor(A)
    del A
    order = np.argsort(rows, kind="stable")
    start = np.searchsorted(rows[order], np.arange(n))
    a, bl = Ax.astype(np.longdouble)[order], b.astype(np.longdouble)
    x = np.zeros(n, np.longdouble)
    for _ in range(4):
        r = bl - np.add.reduceat(a * x[col[order]], start)
        scale = float(np.abs(r).max()) or 1.0
        d = torch.linalg.lu_solve(lu, piv, _dev((r / scale).astype(np.float64))[:, None])[:, 0]
        x = x + d.cpu().numpy().astype(np.longdouble) * scale
    return x.astype(np.float64)


def exact(case, seed):
    """Solutions by dense float64 algebra; None above 12,000 unknowns (the
    dense factors would take too long) and for all but a batch's first sets."""
    if _parts(case)[0][1] * _parts(case)[0][2] * case["nz"] > 12000:
        return None
    kind, out = case["kind"], []
    for part, (_, Ax, b) in zip(_parts(case), _draw_inputs(case, seed)):
        _, n, Ap, Ai, _ = _circuit(*part)
        if kind == "batch":
            if n * len(Ax) > 400000:
                return None
            x = np.stack([_exact_x(n, Ap, Ai, Ax[i], b[i]) for i in range(len(Ax))])
            return {"x": x, "failed": None}
        if kind == "serve":
            out += [_exact_x(n, Ap, Ai, Ax[i], b[i]) if n <= 12000 and i < 3 else None for i in range(len(Ax))]
        elif n > 12000:
            out.append(None)
        else:
            out.append(_exact_x(n, Ap, Ai, Ax[0], b[0]))
    if kind in ("multi", "serve"):
        return out
    return out[0]
