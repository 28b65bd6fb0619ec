"""Batches of structures with wide columns: up to 5/4 of the CTAs (152 SMs,
three each) the wide columns are taken alone, beyond that in panels of four.
Every value set gives the bits that it gives in a batch of its own, on both
sides of the line and with failing sets among the others."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2411_14082_gb300 import gblu, inputs
from tests.factor_compare import compare_factors
from tests.test_gpu_block_restart import bordered_blocks
from tests.test_gpu_panel_abort import dev, with_failing_pivot

pytestmark = pytest.mark.gpu

DEV = 0
LINE = 152 * 3 * 5 // 4


def system(name):
    if name == "blocks":
        return bordered_blocks(200, 40, blocks=400)
    if name == "short":   # wide columns of at most 640 entries
        return bordered_blocks(20, 8, blocks=300)
    nx, rails = (70, 6) if name == "grid6" else (60, 19)
    ckt = inputs.bordered_grid(nx, nx, n_rails=rails, seed=77)
    n, Ap, Ai, Ax = ckt.csc()
    return n, Ap, Ai, Ax, gblu.order_auto(n, Ap, Ai)[0]


@pytest.mark.parametrize("name", ["grid6", "grid19", "blocks", "short"])
@pytest.mark.parametrize("mode", ["auto", "level", "syncfree"])
def test_both_sides_of_the_line(name, mode):
    n, Ap, Ai, Ax0, Q = system(name)
    lu0 = O.factorize(n, Ap, Ai, Ax0, Q, 1e-3)
    s = gblu.Solver(DEV, sched_mode=mode)
    s.analyze(n, Ap, Ai, Q)
    s.factorize(dev(Ax0))
    wide = s.stats()["wide_cols"]
    assert wide > 0
    line = LINE // wide
    rng = np.random.default_rng(3)
    vals = np.stack([Ax0 * rng.uniform(0.98, 1.02, len(Ax0)) for _ in range(line + 2)])
    bad = {1: n // 3, line - 1: n - 2 * wide}   # below the line too, and in both sides' batches
    for i, k in bad.items():
        vals[i] = with_failing_pivot(n, Ap, Ai, vals[i], Q, lu0, k)
    want = []
    for i in range(line + 2):
        LU, failed = s.refactorize_batch(dev(vals[i:i + 1]))
        assert bool(failed[0]) == (i in bad)
        want.append(LU[0].clone())
    assert not s.refactorize(dev(vals[0]))[1]
    compare_factors(s.export_factors(), O.refactorize(lu0, Ap, Ai, vals[0]), 1e-10)
    f = s.export_factors()
    assert np.array_equal(np.sort(want[0].cpu().numpy()), np.sort(np.r_[f["Lx"], f["Ux"]]))
    for count in (line - 1, line, line + 1, line + 2):
        LU, failed = s.refactorize_batch(dev(vals[:count]))
        for i in range(count):
            assert bool(failed[i]) == (i in bad)
            assert i in bad or torch.equal(LU[i], want[i]), (count, i)
