"""What a budget of the server holds: as many sets, and as many patterns, as
the handles need without what only makes them faster."""
import numpy as np
import pytest
import torch

from paper_2411_14082_gb300 import gblu

pytestmark = pytest.mark.gpu

DEV = 0
M, K, TAIL = 64, 45, 4   # dense blocks of 64, a border of 4: one panel in a scratch of every CTA


def system(seed):
    n = M * K + TAIL
    rng = np.random.default_rng(seed)
    cols = [np.r_[(j // M) * M:(j // M) * M + M, n - TAIL:n] if j < M * K else np.arange(n) for j in range(n)]
    Ap = np.r_[0, np.cumsum([len(c) for c in cols])].astype(np.int32)
    Ai = np.concatenate(cols).astype(np.int32)
    Ax = rng.uniform(-1.0, 1.0, len(Ai)) / n
    Ax[Ai == np.repeat(np.arange(n), np.diff(Ap))] = 1.0
    return n, Ap, Ai, np.arange(n, dtype=np.int32), Ax


def alone(sys_, v, b):
    s = gblu.Solver(DEV)
    s.analyze(*sys_[:4])
    for Ax in (sys_[4], v):
        (s.factorize if Ax is sys_[4] else s.refactorize)(torch.from_numpy(Ax).cuda(DEV))
    x = s.solve(torch.from_numpy(b).cuda(DEV)).cpu().numpy()
    full = s.stats()["device_bytes"]
    s.close()
    return x, full


def lean_footprint(sys_, full):
    """One set in a budget that has no room for the scratches."""
    srv = gblu.Server(DEV, hbm_budget=full - (10 << 20), max_batch=1)
    pid, slots = srv.add_pattern(*sys_)
    assert slots == 1
    fp = srv.pattern_info(pid)["footprint_bytes"]
    srv.close()
    return fp


def request(seed, sys_):
    rng = np.random.default_rng(seed)
    return sys_[4] * rng.uniform(0.9, 1.0, len(sys_[4])), rng.uniform(-1.0, 1.0, sys_[0])


def test_a_budget_holds_as_many_sets_as_without_panels():
    sys_ = system(5)
    n, Ap, Ai = sys_[:3]
    v, b = request(6, sys_)
    want, full = alone(sys_, v, b)
    lean = lean_footprint(sys_, full)
    lu = sum(len(c) for c in np.split(Ai, Ap[1:-1]))   # the blocks and the border are full: no fill
    per_set = 8 * (len(Ai) + lu + 2 * n + 4) + 44 * n + 1024
    srv = gblu.Server(DEV, hbm_budget=lean + 15 * per_set + (1 << 20), max_batch=16)
    pid, slots = srv.add_pattern(*sys_)
    assert slots == 16
    x = np.zeros(n)
    srv.wait(srv.submit(pid, v, b, x))
    srv.close()
    assert np.array_equal(x, want)


def test_a_later_pattern_takes_the_room_of_earlier_panels():
    one, two = system(5), system(7)
    (v1, b1), (v2, b2) = request(6, one), request(8, two)
    x1, full = alone(one, v1, b1)
    x2, _ = alone(two, v2, b2)
    lean = lean_footprint(one, full)
    probe = gblu.Server(DEV, hbm_budget=1 << 30, max_batch=1)
    with_panels = probe.pattern_info(probe.add_pattern(*one)[0])["footprint_bytes"]
    probe.close()
    budget = with_panels + lean // 2
    assert budget >= 2 * lean + (1 << 20)
    srv = gblu.Server(DEV, hbm_budget=budget, max_batch=1)
    p1, _ = srv.add_pattern(*one)
    assert srv.pattern_info(p1)["footprint_bytes"] == with_panels
    ids = [srv.submit(p1, v1, b1, np.zeros(one[0])) for _ in range(8)]   # in flight meanwhile
    p2, slots = srv.add_pattern(*two)
    assert slots == 1
    st = srv.stats()
    assert st["reserved_bytes"] <= budget and st["reserved_bytes"] == sum(
        srv.pattern_info(p)["footprint_bytes"] for p in (p1, p2))
    ids += [srv.submit(p1, v1, b1, np.zeros(one[0]))]
    for i in ids:
        assert np.array_equal(srv.wait(i)[0], x1)
    assert np.array_equal(srv.wait(srv.submit(p2, v2, b2, np.zeros(two[0])))[0], x2)
    with pytest.raises(gblu.GbluError) as e:   # and no more than the budget holds
        for _ in range(budget // lean - 1):
            srv.add_pattern(*one)
    assert e.value.code == gblu.ERR_NOMEM and srv.stats()["reserved_bytes"] <= budget
    srv.close()
