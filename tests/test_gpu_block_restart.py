"""A check that fails on a structure with a trailing block: one pass with the
block finds the first failing step, and the restart goes on from the columns
that passed, through gblu_refactorize and through a replayed gblu_step."""
import time

import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2411_14082_gb300 import gblu
from tests.factor_compare import compare_factors
from tests.test_gpu_panel_abort import band, dev, with_failing_pivot

pytestmark = pytest.mark.gpu

DEV = 0


def solver(sys_):
    n, Ap, Ai, Ax0, Q = sys_
    s = gblu.Solver(DEV)
    s.analyze(n, Ap, Ai, Q)
    s.factorize(dev(Ax0))
    return s


def launches(s, call):
    before = s.stats()["kernel_launches"]
    out = call()
    return s.stats()["kernel_launches"] - before, out


# 200 dense last rows and columns, the block, behind too few columns for any
# to be a wide one
@pytest.mark.parametrize("k", [100, 220, 390])
def test_a_failed_check_costs_one_pass_with_the_block(k):
    n, Ap, Ai, Ax0, Q = band(400, 30, 200, 3)
    for r, c in ((k, k + 1), (k + 1, k)):   # steps k and k + 1 exchange rows and no other step moves
        Ax0[Ap[c] + int(np.searchsorted(Ai[Ap[c]:Ap[c + 1]], r))] = 0.9
    sys_ = n, Ap, Ai, Ax0, Q
    rng = np.random.default_rng(2)
    lu0 = O.factorize(n, Ap, Ai, Ax0, Q, 1e-3)
    v = Ax0 * rng.uniform(0.98, 1.02, len(Ax0))
    w = with_failing_pivot(n, Ap, Ai, v, Q, lu0, k)
    lu = O.refactorize(lu0, Ap, Ai, w)
    assert np.nonzero(lu.piv != lu0.piv)[0].tolist() == [k, k + 1]
    b = rng.uniform(-1.0, 1.0, n)
    g, p = solver(sys_), solver(sys_)
    ok_pass, (_, rep) = launches(p, lambda: p.refactorize(dev(v)))
    assert not rep and ok_pass > 13   # a block of 200 columns takes 13 launches of its own
    solve, _ = launches(p, lambda: p.solve(dev(b)))
    replay, (_, rep) = launches(g, lambda: g.step(dev(v), dev(b)))
    assert not rep and replay == ok_pass + solve
    bad_pass, (_, rep) = launches(p, lambda: p.refactorize(dev(w)))
    assert rep and p.stats()["last_first_bad"] == k
    bad_step, (x, rep) = launches(g, lambda: g.step(dev(w), dev(b)))
    assert rep and g.stats()["last_first_bad"] == k
    # the failed replay stands for the first pass; what the restart adds is
    # the same through both calls
    assert bad_step - replay - solve == bad_pass - ok_pass
    for s in (g, p):
        compare_factors(s.export_factors(), lu, 1e-10)
        assert s.stats()["n_repivot"] == 1 and s.stats()["n_refactor"] == 2
    assert O.residual(n, Ap, Ai, w, x.cpu().numpy(), b) <= 1e-12


def test_the_block_keeps_to_max_sms():
    """With one SM's share of CTAs the block's launches take several tasks per
    CTA: the same bits, at a small part of the device's speed (the block is
    all of the arithmetic here, and 152 SMs share it otherwise)."""
    sys_ = band(1400, 1399, 0, 3)
    n, Ap, Ai, Ax0, _ = sys_
    s = solver(sys_)
    v = dev(Ax0 * np.random.default_rng(2).uniform(0.98, 1.02, len(Ax0)))

    def run():
        s.refactorize(v)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        s.refactorize(v)
        torch.cuda.synchronize()
        return time.perf_counter() - t0, s.export_factors()

    t_all, want = run()
    s.set_opts(max_sms=1)
    t_one, got = run()
    for k in want:
        assert np.array_equal(want[k], got[k]), k
    assert t_one > 8 * t_all


def bordered_blocks(tail, wide, blocks=300):
    """`blocks` dense 2 x 2 blocks and `tail` dense last columns: the last
    `wide` of them touch every block (a run of dependencies each), the others
    one block in turn."""
    n = 2 * blocks + tail
    rng = np.random.default_rng(9)
    a = np.zeros((n, n), bool)
    for j in range(blocks):
        a[2 * j:2 * j + 2, 2 * j:2 * j + 2] = True
        a[2 * j:2 * j + 2, n - wide:] = True
        a[2 * j:2 * j + 2, 2 * blocks + j % (tail - wide)] = True
    a |= a.T
    a[2 * blocks:, 2 * blocks:] = True
    cols, rows = np.nonzero(a.T)
    Ap = np.r_[0, np.cumsum(np.bincount(cols, minlength=n))].astype(np.int32)
    Ax = np.where(rows == cols, 1.0, rng.uniform(-1.0, 1.0, len(rows)) / n)
    return n, Ap, rows.astype(np.int32), Ax, np.arange(n, dtype=np.int32)


@pytest.mark.parametrize("wide,taken", [(3, 0), (40, 40)])
def test_columns_that_are_barely_wide_leave_the_block(wide, taken):
    """Three last columns of 301 runs, 0.7% of the flops, do not count as wide
    ones and the block of 700 columns (44 steps) is factored densely; forty
    hold more and count.  Both ways the factors are the oracle's, and the
    batch's route gives the same bits."""
    sys_ = bordered_blocks(700, wide)
    n, Ap, Ai, Ax0, Q = sys_
    s = solver(sys_)
    assert s.stats()["wide_cols"] == taken
    v = Ax0 * np.random.default_rng(2).uniform(0.98, 1.02, len(Ax0))
    passes, (_, rep) = launches(s, lambda: s.refactorize(dev(v)))
    assert not rep and (passes > 44) == (taken == 0)
    lu = O.refactorize(O.factorize(n, Ap, Ai, Ax0, Q, 1e-3), Ap, Ai, v)
    compare_factors(s.export_factors(), lu, 1e-10)
    b = dev(np.random.default_rng(4).uniform(-1.0, 1.0, n))
    LU, failed = s.refactorize_batch(dev(v[None]))
    assert not failed.any() and torch.equal(s.solve_batch(LU, b[None])[0], s.solve(b))


def test_wide_panels_whose_columns_lack_some_rows_of_their_neighbours():
    """Wide columns that touch different nine tenths of the blocks: panels of
    them hold zeros where a column has no entry."""
    n, Ap, Ai, Ax0, Q = bordered_blocks(200, 40, blocks=400)
    rng = np.random.default_rng(12)
    cols = np.repeat(np.arange(n), np.diff(Ap))
    keep = np.ones(len(Ai), bool)
    for c in range(n - 40, n):   # drop a block's two entries and the two across the diagonal
        for j in rng.choice(400, 40, replace=False):
            keep &= ~(((cols == c) & (Ai // 2 == j)) | ((Ai == c) & (cols // 2 == j)))
    Ap = np.r_[0, np.cumsum(np.bincount(cols[keep], minlength=n))].astype(np.int32)
    sys_ = n, Ap, Ai[keep], Ax0[keep], Q
    s = solver(sys_)
    assert s.stats()["wide_cols"] == 40
    v = sys_[3] * np.random.default_rng(2).uniform(0.98, 1.02, len(sys_[3]))
    _, rep = s.refactorize(dev(v))
    lu = O.refactorize(O.factorize(*sys_[:4], Q, 1e-3), Ap, sys_[2], v)
    assert not rep and lu.n_rejected == 0
    compare_factors(s.export_factors(), lu, 1e-10)
    b = dev(np.random.default_rng(4).uniform(-1.0, 1.0, n))
    LU, failed = s.refactorize_batch(dev(np.tile(v, (5, 1))))
    x = s.solve_batch(LU, b.expand(5, n).contiguous())
    assert not failed.any() and bool((x == s.solve(b)).all())


@pytest.mark.parametrize("n,half,tail", [(2, 1, 0), (9, 8, 0), (33, 32, 0), (129, 128, 0), (200, 20, 3)])
def test_batches_large_enough_for_the_column_list_equal_the_panels(n, half, tail):
    """A batch takes short columns one per warp from 1,800 / sqrt(n) sets."""
    sys_ = band(n, half, tail, 7)
    s = solver(sys_)
    v = dev(sys_[3] * np.random.default_rng(2).uniform(0.98, 1.02, len(sys_[3])))
    one, _ = s.refactorize_batch(v[None])
    many, failed = s.refactorize_batch(v.expand(int(1800 / n ** 0.5) + 2, len(v)).contiguous())
    assert not failed.any() and bool((many == one[0]).all())
