"""The pool of the pivoting kernel: how it grows, and factorizations on a
device with little room."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2411_14082_gb300 import gblu, inputs

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


@pytest.mark.parametrize("taken", [0.6, 1.35])
def test_first_factorization_with_little_room(taken):
    """A device with room for the factors (1 time the estimate's entries) and
    a pool of 1.25 times them, but not for the larger pool of 2.5 times, while
    the structure is installed or from the beginning: the factorization runs,
    with the same bits.  taken: entries that are missing, in estimates."""
    ckt = inputs.rc_mesh3d(80, 80, 4, seed=5, n_fet=300)
    n, Ap, Ai, Ax = ckt.csc()
    Q = inputs.grid_nd_order(ckt)
    Axd, b = dev(Ax), dev(np.random.default_rng(1).uniform(-1.0, 1.0, n))
    x = torch.empty_like(b)
    entries = 2 * gblu.symmetric_fill(n, Ap, Ai, Q) + n
    assert 2.5 * entries < 32 << 20   # both sizes come from the estimate

    def factorize():
        s = gblu.Solver(DEV, speculate_first=0)
        s.analyze(n, Ap, Ai, Q)
        s.factorize(Axd)
        s.solve(b, x)
        torch.cuda.synchronize()
        return s

    s = factorize()
    want = x.clone()
    torch.cuda.empty_cache()
    hold = []
    try:
        # every byte but a few MB beside the handle, then some (12 bytes an
        # entry) in its place
        hold.append(torch.empty(torch.cuda.mem_get_info(DEV)[0] - (8 << 20), dtype=torch.uint8, device=f"cuda:{DEV}"))
        s.close()
        hold.append(torch.empty(int(taken * entries * 12), dtype=torch.uint8, device=f"cuda:{DEV}"))
        x.zero_()
        s = factorize()
        assert torch.equal(x, want)
        s.close()
    finally:
        hold.clear()
        torch.cuda.empty_cache()


def test_predicted_structure_with_little_room():
    """Less and less room beside a handle, until the factorization is refused:
    up to there it gives up the panels' workspaces, with the same bits."""
    ckt = inputs.rc_mesh3d(60, 60, 4, seed=5, n_fet=150)
    n, Ap, Ai, Ax = ckt.csc()
    Q = inputs.grid_nd_order(ckt)
    Axd, b = dev(Ax), dev(np.random.default_rng(1).uniform(-1.0, 1.0, n))
    x = torch.empty_like(b)

    def factorize():
        s = gblu.Solver(DEV)
        s.analyze(n, Ap, Ai, Q)
        s.factorize(Axd)
        s.solve(b, x)
        torch.cuda.synchronize()
        return s

    s = factorize()
    want, full = x.clone(), s.stats()["device_bytes"]
    torch.cuda.empty_cache()
    hold, held = [], []
    try:
        hold.append(torch.empty(torch.cuda.mem_get_info(DEV)[0] - (4 << 20), dtype=torch.uint8, device=f"cuda:{DEV}"))
        s.close()
        while True:
            x.zero_()
            try:
                s = factorize()
            except gblu.GbluError as e:
                assert e.code == gblu.ERR_NOMEM
                break
            assert torch.equal(x, want)
            held.append(s.stats()["device_bytes"])
            s.close()
            hold.append(torch.empty(4 << 20, dtype=torch.uint8, device=f"cuda:{DEV}"))
    finally:
        hold.clear()
        torch.cuda.empty_cache()
    assert held[0] == full and min(held) < full - (4 << 20)
