"""Handles on streams of their own, their iterations queued at once from one
thread and from several: the one-launch forms take turns on the device (every
block of a launch waits for the others of it, never for another handle's), and
each handle's result is what it is alone."""
import threading

import numpy as np
import pytest

from paper_2003_09956_gb300 import nsli, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="session", autouse=True)
def built_library():
    from paper_2003_09956_gb300 import _build
    _build.build()
    nsli.load()


SYSTEMS = [("f32", 2000, 500), ("f64", 513, 256), ("bf16", 20, 300), ("f32", 9000, 1025), ("fp8", 76, 2048),
           ("f32", 8, 8192)]


@pytest.mark.parametrize("threads", [False, True])
def test_handles_side_by_side(threads):
    alone, made = [], []
    for k, (storage, m, n) in enumerate(SYSTEMS):
        p = workloads.dense_system(m, n, seed=k)
        src = p["A"].astype(np.float64) if storage == "f64" else p["A"]
        made.append((p, nsli.Solver(src, p["b0"], p["x0"], Av=p["Av"], storage=storage)))
    try:
        for p, s in made:
            s.iterate(300, rho=1e-4)
            r = s.solve(stop="step", eps=1e-12, max_iter=50)
            alone.append((s.get_x(), r["iters"], r["status"]))
        for rnd in range(3):
            got = [None] * len(made)
            for p, s in made:
                s.set_x(p["x0"])
                s.update_b(tick=0)

            def work(k):
                s = made[k][1]
                s.iterate(300, rho=1e-4)
                r = s.solve(stop="step", eps=1e-12, max_iter=50)
                got[k] = (s.get_x(), r["iters"], r["status"])
            if threads:
                ts = [threading.Thread(target=work, args=(k,)) for k in range(len(made))]
                for t in ts:
                    t.start()
                for t in ts:
                    t.join()
            else:
                for p, s in made:
                    s.iterate(300, rho=1e-4)
                for k, (p, s) in enumerate(made):
                    r = s.solve(stop="step", eps=1e-12, max_iter=50)
                    got[k] = (s.get_x(), r["iters"], r["status"])
            for a, b in zip(alone, got):
                np.testing.assert_array_equal(a[0], b[0])
                assert a[1:] == b[1:]
    finally:
        for _, s in made:
            s.close()
