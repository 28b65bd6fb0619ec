"""Panels that are given up: a check that fails in one column of a value set
stops the other panels of that set while their copies are in flight, and the
CTAs go on to other sets in the same shared memory.  The sets whose checks
pass have to come out the same bits as alone, on every repetition."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2411_14082_gb300 import gblu, inputs

pytestmark = pytest.mark.gpu

DEV = 0


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(f"cuda:{DEV}")


def band(n, half, tail, seed):
    """|i - j| <= half and `tail` dense last rows and columns, dominant diagonal."""
    rng = np.random.default_rng(seed)
    i, j = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
    mask = (np.abs(i - j) <= half) | (i >= n - tail) | (j >= n - tail)
    a = np.where(mask, rng.uniform(-1.0, 1.0, (n, n)) / (2 * half + tail), 0.0)
    np.fill_diagonal(a, 1.0)
    cols, rows = np.nonzero(mask.T)
    Ap = np.r_[0, np.cumsum(np.bincount(cols, minlength=n))].astype(np.int32)
    return n, Ap, rows.astype(np.int32), a[rows, cols], np.arange(n, dtype=np.int32)


def system(name):
    if name == "band":   # one long chain of panels, several stages each
        return band(700, 90, 8, 3)
    ckt = inputs.bordered_grid(30, 30, n_rails=6, density=0.3) if name == "rails" else \
        inputs.rc_mesh3d(20, 20, 4, seed=5, n_fet=40)
    n, Ap, Ai, Ax = ckt.csc()
    return n, Ap, Ai, Ax, inputs.grid_nd_order(ckt)


def with_failing_pivot(n, Ap, Ai, Ax, Q, lu0, k):
    """Values whose step k' >= k (the first with L rows below it) has a pivot
    of about 1e-9 of what it was, by the oracle's elimination."""
    ref = O.refactorize(lu0, Ap, Ai, Ax)
    assert ref.n_rejected == 0
    while True:
        c = Q[k]
        hit = np.nonzero(Ai[Ap[c]:Ap[c + 1]] == lu0.piv[k])[0]
        if len(hit) and ref.Lp[k + 1] > ref.Lp[k]:
            break
        k += 1
    out = Ax.copy()
    out[Ap[c] + hit[0]] -= ref.Ux[ref.Up[k + 1] - 1] * (1.0 - 1e-9)
    assert O.refactorize(lu0, Ap, Ai, out).n_rejected > 0
    return out


@pytest.mark.parametrize("name", ["band", "mesh", "rails"])
def test_failing_sets_leave_the_others_alone(name):
    n, Ap, Ai, Ax0, Q = system(name)
    lu0 = O.factorize(n, Ap, Ai, Ax0, Q, 1e-3)
    rng = np.random.default_rng(8)
    nsets = 36   # of these sizes, a batch this small takes the panels
    vals = np.stack([Ax0 * rng.uniform(0.98, 1.02, len(Ax0)) for _ in range(nsets)])
    bad = list(range(1, nsets, 3))
    for i, s in enumerate(bad):   # at places spread over the whole factorization
        vals[s] = with_failing_pivot(n, Ap, Ai, vals[s], Q, lu0, n // 20 + i * (17 * n // 20) // len(bad))
    good = [s for s in range(nsets) if s not in bad]
    s = gblu.Solver(DEV)
    s.analyze(n, Ap, Ai, Q)
    s.factorize(dev(Ax0))
    alone = []
    for i in good:
        LU, failed = s.refactorize_batch(dev(vals[i:i + 1]))
        assert not failed.any()
        alone.append(LU[0].clone())
    want = torch.stack(alone)
    Ax = dev(vals)
    for _ in range(25):
        LU, failed = s.refactorize_batch(Ax)
        assert np.nonzero(failed)[0].tolist() == bad
        assert torch.equal(LU[good], want)


@pytest.mark.parametrize("k", [40, 333, 560])
def test_single_precision_after_a_given_up_panel(k):
    """The float panels: a failed check sends the call to double precision,
    and the next call on passing values gives the earlier bits."""
    n, Ap, Ai, Ax0, Q = system("band")
    lu0 = O.factorize(n, Ap, Ai, Ax0, Q, 1e-3)
    v = Ax0 * np.random.default_rng(4).uniform(0.98, 1.02, len(Ax0))
    w = with_failing_pivot(n, Ap, Ai, v, Q, lu0, k)
    b = dev(np.random.default_rng(5).uniform(-1.0, 1.0, n))
    s = gblu.Solver(DEV)
    s.analyze(n, Ap, Ai, Q)
    s.factorize(dev(Ax0))
    assert not s.refactorize_f32(dev(v))
    want = s.solve_refined(dev(v), b, max_iter=0, tol=1.0)[0].clone()
    for _ in range(10):
        assert s.refactorize_f32(dev(w))
        assert not s.refactorize_f32(dev(v))
        assert torch.equal(s.solve_refined(dev(v), b, max_iter=0, tol=1.0)[0], want)


@pytest.mark.parametrize("name", ["band", "mesh", "rails"])
def test_failing_handles_of_one_launch_leave_the_others_alone(name):
    """The same in a launch over several handles: those whose check fails
    restart alone, the others give what they give alone."""
    n, Ap, Ai, Ax0, Q = system(name)
    lu0 = O.factorize(n, Ap, Ai, Ax0, Q, 1e-3)
    rng = np.random.default_rng(9)
    vals = [Ax0 * rng.uniform(0.98, 1.02, len(Ax0)) for _ in range(6)]
    bad = {1: n // 3, 4: 2 * n // 3}
    for i, k in bad.items():
        vals[i] = with_failing_pivot(n, Ap, Ai, vals[i], Q, lu0, k)
    b = dev(rng.uniform(-1.0, 1.0, n))
    Ax = [dev(v) for v in vals]
    solvers = []
    for _ in vals:
        s = gblu.Solver(DEV)
        s.analyze(n, Ap, Ai, Q)
        s.factorize(dev(Ax0))
        solvers.append(s)
    want = {}
    for i, s in enumerate(solvers):
        if i not in bad:
            assert not s.refactorize(Ax[i])[1]
            want[i] = s.solve(b).clone()
    for _ in range(10):
        for i in bad:
            solvers[i].factorize(dev(Ax0))
        rep = gblu.refactorize_multi(solvers, Ax)
        assert [i for i, r in enumerate(rep) if r] == sorted(bad)
        for i, s in enumerate(solvers):
            x = s.solve(b)
            if i in bad:
                assert O.residual(n, Ap, Ai, vals[i], x.cpu().numpy(), b.cpu().numpy()) <= 1e-12
            else:
                assert torch.equal(x, want[i])
