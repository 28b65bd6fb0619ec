"""Panels of single-precision factors: the same bits as the column kernels
give (a handle with a dense tail has no panels, and single precision leaves
the tail to the columns), at unions around the shared-memory limits of both
configurations and beyond them."""
import numpy as np
import pytest

from paper_2411_14082_gb300 import gblu, inputs
from tests.test_gpu_panel_abort import band, dev

pytestmark = pytest.mark.gpu

DEV = 0


def widened_solution(sys_, v, b, **opts):
    n, Ap, Ai, Ax0, Q = sys_
    s = gblu.Solver(DEV, **opts)
    s.analyze(n, Ap, Ai, Q)
    s.factorize(dev(Ax0))
    assert not s.refactorize_f32(dev(v))
    x, iters, _ = s.solve_refined(dev(v), b, max_iter=0, tol=1.0)
    assert iters == 0
    return x.cpu().numpy(), s.stats()["dense_rows"]


@pytest.mark.parametrize("case", [(9, 8, 0), (300, 40, 3), (640, 639, 0), (670, 669, 0), (1150, 1149, 0), (1500, 255, 20),
                                  (2300, 2290, 0), (2600, 1250, 0), "mesh", "rails"])
def test_panels_equal_the_column_kernels(case):
    if isinstance(case, tuple):
        sys_ = band(*case, 11)
    else:
        ckt = inputs.rc_mesh3d(40, 40, 4, seed=5, n_fet=100) if case == "mesh" else inputs.bordered_grid(60, 60, n_rails=6)
        n, Ap, Ai, Ax0 = ckt.csc()
        sys_ = n, Ap, Ai, Ax0, inputs.grid_nd_order(ckt)
    rng = np.random.default_rng(3)
    v = sys_[3] * rng.uniform(0.95, 1.05, len(sys_[3]))
    b = dev(rng.uniform(-1.0, 1.0, sys_[0]))
    want, rows = widened_solution(sys_, v, b, dense_min_rows=1)
    assert rows > 0
    got, rows = widened_solution(sys_, v, b)
    assert rows == 0 and np.array_equal(got, want)
