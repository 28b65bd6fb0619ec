"""Host work that runs on several threads: calls from several threads at once,
each with its own set of host threads, give what one call alone gives."""
import threading

import numpy as np

from paper_2411_14082_gb300 import gblu, inputs


def patterns():
    for a, b, nz in ((60, 54, 4), (45, 40, 4), (24, 20, 3)):   # two above the size from which threads share the work
        ckt = inputs.rc_mesh3d(a, b, nz, seed=5, n_fet=40)
        n, Ap, Ai, _ = ckt.csc()
        yield n, Ap, Ai, inputs.grid_nd_order(ckt)


def test_structures_from_several_threads():
    pats = list(patterns())
    want = [gblu.symmetric_structure(*p) for p in pats]
    wrong = []

    def work(i):
        for r in range(6):
            j = (i + r) % len(pats)
            got = gblu.symmetric_structure(*pats[j])
            if not all(np.array_equal(x, y) for x, y in zip(got, want[j])):
                wrong.append((i, j))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong
