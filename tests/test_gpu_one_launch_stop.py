"""The step rule inside one launch: ||dx|| is known to a block only after the
next Map, from words that every block writes and reads.  The threshold is put
between the step lengths of two iterations of a binary64 reference, so the
iteration at which the run has to stop is known; shapes with several rounds
of columns per block, and with many blocks that have no columns."""
import numpy as np
import pytest

from paper_2003_09956_gb300 import nsli, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="session", autouse=True)
def built_library():
    from paper_2003_09956_gb300 import _build
    _build.build()
    nsli.load()


def step_lengths(p, steps):
    A, x = p["A"].astype(np.float64), p["x0"].copy()
    n2 = (A * A).sum(1)
    out = []
    for _ in range(steps):
        r = np.maximum(A @ x - p["b0"], 0.0)
        dx = ((r / n2) @ A) / (r > 0).sum()
        x -= dx
        out.append(np.linalg.norm(dx))
    return np.array(out)


SHAPES = [("f32", 20, 8000), ("f32", 40, 8000), ("f64", 20, 4000), ("f32", 150, 8191), ("f32", 3000, 96), ("f64", 2432, 500),
          ("f32", 9001, 128), ("bf16", 500, 2048)]


@pytest.mark.parametrize("storage,m,n", SHAPES)
def test_step_rule_stops_after_the_same_step(storage, m, n):
    p = workloads.dense_system(m, n, seed=5, grid="bf16" if storage == "bf16" else None)
    d = step_lengths(p, 60)
    src = p["A"].astype(np.float64) if storage == "f64" else p["A"]
    with nsli.Solver(src, p["b0"], p["x0"], storage=storage) as s:
        for stop_at in (1, 2, 3, 8, 33, 34, 59):
            # consecutive lengths differ by 5e-4 at least, binary32 runs by 1e-5
            # from the reference at most
            eps = float(np.sqrt(d[stop_at - 1] * d[stop_at]))
            assert d[stop_at - 1] / d[stop_at] > 1.0005 and np.all(d[:stop_at] > eps)
            got = []
            for block in [0] * 4 + [32]:
                s.set_x(p["x0"])
                s.update_b(tick=0)
                r = s.solve(stop="step", eps=eps, max_iter=100, block_iters=block)
                got.append((r["status"], r["iters"], r["tick"], r["last_step_norm"], s.get_x()))
            for g in got:
                assert g[:3] == (nsli.OK, stop_at + 1, stop_at + 1)
                np.testing.assert_allclose(g[3], got[-1][3], rtol=1e-14)
                np.testing.assert_array_equal(g[4], got[-1][4])


@pytest.mark.parametrize("storage,m,n", [("f32", 20, 8000), ("f32", 40, 8000), ("f32", 3000, 96)])
def test_modap_step_is_lambda_long(storage, m, n):
    """A ModAP step is lambda long: just above it the rule holds at once,
    just below it the run goes to its last iteration."""
    p = workloads.dense_system(m, n, seed=5)
    with nsli.Solver(p["A"], p["b0"], p["x0"], storage=storage) as s:
        for eps, status, iters in ((1.001e-2, nsli.OK, 1), (0.999e-2, nsli.NOT_CONVERGED, 70)):
            got = []
            for block in (0, 0, 0, 32):
                s.set_x(p["x0"])
                r = s.solve(lam=1e-2, rule="modap", stop="step", eps=eps, max_iter=70, block_iters=block)
                got.append((r["status"], r["iters"], s.get_x()))
            for g in got:
                assert g[:2] == (status, iters)
                np.testing.assert_array_equal(g[2], got[-1][2])


@pytest.mark.parametrize("eps,iters", [(1e-100, 333), (1e-149, 495), (1e-151, 502), (1e-165, 538)])
def test_step_rule_at_thresholds_whose_square_underflows(eps, iters):
    """x <= 0 from x = 1 with half steps: step k is 2^-k long, its square 0
    from k = 538 on.  ||dx|| is the root of the sum of squares in a one-launch
    run too, and on one CTA."""
    one = np.ones(1)
    dense = nsli.Solver(np.ones((1, 1)), np.zeros(1), one, storage="f64")
    sparse = nsli.SparseSolver(1, 1, np.array([0, 1]), np.array([0], np.int32), one, np.zeros(1), one, storage="f64")
    with dense, sparse:
        for s, block in ((dense, 0), (dense, 32), (sparse, 0), (sparse, 7)):
            s.set_x(one)
            r = s.solve(lam=0.5, stop="step", eps=eps, max_iter=1000, block_iters=block)
            assert (r["status"], r["iters"], s.get_x()[0]) == (nsli.OK, iters, 2.0 ** -iters)
