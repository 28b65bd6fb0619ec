"""Panels, the trailing block and the column task list of batches, at the
sizes where they change: panel widths and remainders, one and several stages
of a run, the widest shared-memory unions, work vectors in a scratch, blocks
of 16 columns and their remainder, and blocks too small to be taken.

The same values through every route have to give the same bits (each value
gets the same multiply-adds in the same order), and the factors have to equal
the oracle's: its work-vector entries are sums of at most n products of
magnitude <= 1 (the matrices are scaled that way and diagonally dominant), so
two evaluation orders differ by at most n * 2^-52 * n relative to the
column's largest entry, below 1e-10 for every n here."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2411_14082_gb300 import gblu

pytestmark = pytest.mark.gpu

DEV = 0


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(f"cuda:{DEV}")


def band(n, half, tail, seed):
    """Symmetric pattern: |i - j| <= half, and `tail` dense last rows and
    columns; diagonally dominant values of magnitude <= 1."""
    rng = np.random.default_rng(seed)
    i, j = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
    mask = (np.abs(i - j) <= half) | (i >= n - tail) | (j >= n - tail)
    a = np.where(mask, rng.uniform(-1.0, 1.0, (n, n)), 0.0)
    off = np.abs(a).sum(1) - np.abs(np.diag(a))
    a /= max(1.0, 1.1 * off.max())
    np.fill_diagonal(a, 1.0)
    cols, rows = np.nonzero(mask.T)
    Ap = np.zeros(n + 1, np.int32)
    np.add.at(Ap, cols + 1, 1)
    return n, np.cumsum(Ap).astype(np.int32), rows.astype(np.int32), a[rows, cols]


def routes(n, Ap, Ai, Ax, sets):
    """Solutions of one system by the single-matrix and the batch routes."""
    s = gblu.Solver(DEV)
    s.analyze(n, Ap, Ai, np.arange(n, dtype=np.int32))
    s.factorize(dev(Ax))
    v = Ax * np.random.default_rng(n).uniform(0.9, 1.0, len(Ax))
    b = dev(np.random.default_rng(n + 1).uniform(-1.0, 1.0, n))
    _, rep = s.refactorize(dev(v))
    assert not rep
    f = s.export_factors()
    x = [s.solve(b)]
    for k in sets:
        LU, failed = s.refactorize_batch(dev(np.tile(v, (k, 1))))
        assert not failed.any()
        xb = s.solve_batch(LU, b.expand(k, n).contiguous())
        assert bool((xb == xb[0]).all())
        x.append(xb[0])
    return s, v, f, x


@pytest.mark.parametrize("n,half,tail", [(2, 1, 0), (5, 4, 0), (9, 8, 0), (17, 16, 0), (33, 32, 0), (127, 126, 0),
                                         (128, 127, 0), (129, 128, 0), (300, 299, 0), (301, 7, 3), (400, 15, 1),
                                         (400, 16, 33), (420, 40, 130), (523, 90, 0)])
def test_routes_agree_and_match_the_oracle(n, half, tail):
    n, Ap, Ai, Ax = band(n, half, tail, 7)
    s, v, f, x = routes(n, Ap, Ai, Ax, (1, 120))
    for y in x[1:]:
        assert torch.equal(x[0], y)
    lu = O.refactorize(O.factorize(n, Ap, Ai, Ax, np.arange(n, dtype=np.int32), 1e-3), Ap, Ai, v)
    assert np.array_equal(f["piv"], lu.piv)
    dense = np.zeros((n, n))
    for p, i, val in ((f["Lp"], f["Li"], f["Lx"]), (f["Up"], f["Ui"], f["Ux"])):
        dense[i, np.repeat(np.arange(n), np.diff(p))] = val
    want = np.zeros((n, n))
    for p, i, val in ((lu.Lp, lu.Li, lu.Lx), (lu.Up, lu.Ui, lu.Ux)):
        want[i, np.repeat(np.arange(n), np.diff(p))] = val
    scale = np.maximum(np.abs(want).max(0), np.abs(np.diag(want)))
    assert (np.abs(dense - want) <= 1e-10 * scale).all()


@pytest.mark.parametrize("n,half,tail", [(1150, 1149, 0), (1500, 255, 20), (2600, 1250, 0)])
def test_long_unions(n, half, tail):
    """Unions around the shared-memory limits and beyond (scratch panels),
    by route; the residual bounds the solution."""
    n, Ap, Ai, Ax = band(n, half, tail, 11)
    s, v, _, x = routes(n, Ap, Ai, Ax, (2,))
    assert torch.equal(x[0], x[1])
    b = np.random.default_rng(n + 1).uniform(-1.0, 1.0, n)
    assert O.residual(n, Ap, Ai, v, x[0].cpu().numpy(), b) <= 1e-12


@pytest.mark.parametrize("col", [3, 60, 255, 290])
def test_failed_check_inside_a_panel(col):
    """A pivot that fails its check in the middle of a panel or of the
    trailing block: the restart ends with the oracle's pivots."""
    n, Ap, Ai, Ax = band(300, 299, 0, 13)
    s = gblu.Solver(DEV)
    q = np.arange(n, dtype=np.int32)
    s.analyze(n, Ap, Ai, q)
    s.factorize(dev(Ax))
    v = Ax.copy()
    p = Ap[col] + int(np.searchsorted(Ai[Ap[col]:Ap[col + 1]], col))
    v[p] = 1e-9
    _, rep = s.refactorize(dev(v))
    lu = O.refactorize(O.factorize(n, Ap, Ai, Ax, q, 1e-3), Ap, Ai, v)
    assert rep == (not np.array_equal(lu.piv, q))
    assert np.array_equal(s.export_factors()["piv"], lu.piv)
    b = np.ones(n)
    assert O.residual(n, Ap, Ai, v, s.solve(dev(b)).cpu().numpy(), b) <= 1e-12


def test_server_budget_without_room_for_panel_scratches():
    """A budget that holds the factors but not the CTAs' scratches: the
    pattern is taken without panels and gives the same bits."""
    m, k, tail = 64, 45, 4   # dense blocks of m, a border of 4: one scratch panel
    n = m * k + tail
    rng = np.random.default_rng(5)
    cols = [np.r_[(j // m) * m:(j // m) * m + m, n - tail:n] if j < m * k else np.arange(n) for j in range(n)]
    Ap = np.r_[0, np.cumsum([len(c) for c in cols])].astype(np.int32)
    Ai = np.concatenate(cols).astype(np.int32)
    Ax = rng.uniform(-1.0, 1.0, len(Ai)) / n
    Ax[Ai == np.repeat(np.arange(n), np.diff(Ap))] = 1.0
    q = np.arange(n, dtype=np.int32)
    s = gblu.Solver(DEV)
    s.analyze(n, Ap, Ai, q)
    s.factorize(dev(Ax))
    full = s.stats()["device_bytes"]
    v, b = Ax * rng.uniform(0.9, 1.0, len(Ax)), rng.uniform(-1.0, 1.0, n)
    s.refactorize(dev(v))
    want = s.solve(dev(b)).cpu().numpy()
    budget = full - (10 << 20)
    srv = gblu.Server(DEV, hbm_budget=budget, max_batch=1)
    pid, slots = srv.add_pattern(n, Ap, Ai, q, Ax)
    assert slots == 1 and srv.pattern_info(pid)["footprint_bytes"] <= budget
    x = np.zeros(n)
    srv.wait(srv.submit(pid, v, b, x))
    srv.close()
    assert np.array_equal(x, want)
