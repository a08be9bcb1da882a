"""Whole iterations in one launch, and the row teams of the Map.

Without block_iters, nsli_iterate and nsli_solve run many iterations of a
register-resident dense system in one cooperative launch; with it, they
replay Map and Reduce launches.  Both take the same steps in the same
arithmetic order, so the results are equal bit for bit.  The shapes sit at
the edges of the launch shape: one team and several, rows at the limits of
what one, two, four, eight and sixteen warps hold, blocks that fit the
shared-memory ring and blocks that run through it many times, rows that do
not fill their vectors or groups."""
import numpy as np
import pytest

import oracle
import parity
from paper_2003_09956_gb300 import nsli, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="session", autouse=True)
def built_library():
    from paper_2003_09956_gb300 import _build
    _build.build()
    nsli.load()


SHAPES = [("f32", 1, 1), ("f64", 7, 513), ("bf16", 152, 8), ("f32", 2432, 500), ("f32", 2433, 500),
          ("bf16", 20000, 33), ("f32", 9001, 128), ("fp8", 12000, 130), ("f32", 9000, 1025), ("bf16", 5000, 2049),
          ("f64", 4000, 513), ("f64", 1300, 2049), ("fp8", 9000, 4097), ("f32", 3001, 4100), ("bf16", 2500, 8193),
          ("f32", 700, 8191), ("f64", 500, 8192), ("fp8", 1500, 16384), ("f32", 310, 16383)]


def stored(A32, storage):
    if storage == "bf16":
        return oracle.quantize_bf16(A32)
    return oracle.quantize_e4m3_rows(A32)[0] if storage == "fp8" else A32


def solver(p, storage):
    src = p["A"].astype(np.float64) if storage == "f64" else p["A"]
    return nsli.Solver(src, p["b0"], p["x0"], Av=p["Av"], storage=storage)


@pytest.mark.parametrize("storage,m,n", SHAPES)
def test_iterations_in_one_launch_equal_separate_launches(storage, m, n):
    p = workloads.dense_system(m, n, seed=17 * n + m)
    for rule, lam in (("relaxed", 1.0), ("modap", 5.0 / np.sqrt(n))):
        with solver(p, storage) as a, solver(p, storage) as b:
            y, h, st = a.map_reduce()
            sms = __import__("torch").cuda.get_device_properties(0).multi_processor_count
            parity.check_map_reduce(y, h, st, stored(p["A"], storage), p["b0"], p["x0"], storage,
                                    depth=parity.dense_y_depth(m, sms), levels=parity.dot_levels(n))
            c0 = a.launch_count()
            a.iterate(11, lam=lam, rule=rule, rho=1e-3)
            a.sync()
            assert a.launch_count() - c0 == 2          # the run's set-up and one launch
            b.iterate(11, lam=lam, rule=rule, rho=1e-3, block_iters=4)
            np.testing.assert_array_equal(a.get_x(), b.get_x())
            ra, rb = a.result(), b.result()
            assert ra["tick"] == rb["tick"] == 11 and ra["iters"] == rb["iters"] == 11
            np.testing.assert_allclose(ra["last_step_norm"], rb["last_step_norm"], rtol=1e-14)


@pytest.mark.parametrize("stop,eps,max_iter", [("step", 1e-8, 100000), ("epsmem", 1e-7, 100000),
                                               ("maxviol_rel", 1e-6, 100000), ("step", 1e-8, 37), ("none", 0.0, 70)])
def test_solves_in_one_launch_stop_where_separate_launches_do(stop, eps, max_iter):
    p = workloads.model_system(96, seed=3)
    res = []
    for block in (0, 32):
        with nsli.Solver(p["A"], p["b0"], p["x0"], storage="f64") as s:
            r = s.solve(stop=stop, eps=eps, max_iter=max_iter, block_iters=block)
            res.append((r["status"], r["iters"], r["tick"], r["h"], r["rejected"], s.get_x()))
    assert res[0][:5] == res[1][:5]
    np.testing.assert_array_equal(res[0][5], res[1][5])
