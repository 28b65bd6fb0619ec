"""The pool of the pivoting kernel: how it grows, and what it does without
room for its first size."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2411_14082_gb300 import gblu

pytestmark = pytest.mark.gpu

DEV = 0


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(f"cuda:{DEV}")


def arrow(n):
    """Dense last row and column.  At every step the row displaced by the
    last one holds twice the diagonal entry, so partial pivoting takes it
    and U fills to n^2 / 2, against a symmetric estimate of 3 n."""
    d = 2.0 ** -np.arange(n - 1)
    cols = [np.array([j, n - 1]) for j in range(n - 1)] + [np.arange(n)]
    Ap = np.r_[0, np.cumsum([len(c) for c in cols])].astype(np.int32)
    Ax = np.concatenate([np.r_[v, 2.0] for v in d] + [np.r_[d, 1.0]])
    return n, Ap, np.concatenate(cols).astype(np.int32), Ax, np.arange(n, dtype=np.int32)


def test_a_full_pool_grows_from_the_capacity_that_was_tried():
    s = gblu.Solver(DEV, pivot_tol=1.0, speculate_first=0)
    for n in (300, 500):
        n, Ap, Ai, Ax, Q = arrow(n)
        s.analyze(n, Ap, Ai, Q)
        before = s.stats()["kernel_launches"]
        s.factorize(dev(Ax))
        runs = (s.stats()["kernel_launches"] - before) / 3
        lu = O.factorize(n, Ap, Ai, Ax, Q, 1.0)
        assert len(lu.Ux) > n * n // 2 and np.array_equal(s.export_factors()["piv"], lu.piv)
    # 300 unknowns left buffers of at least 45,000 entries and at most twice
    # that; 500 need 125,000: one run at what is there, and one or two more
    assert 2 <= runs <= 3
