"""Bounded waits of a one-launch run, without a GPU fault: one block waits for
a copy that is never issued, the others for that block at the grid's counter.
All waits end, the call reports it, a launch that follows in the same run
leaves at once, and the next run is unaffected."""
import time

import numpy as np
import pytest

from paper_2003_09956_gb300 import nsli, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="session", autouse=True)
def built_library():
    from paper_2003_09956_gb300 import _build
    _build.build()
    nsli.load()


# several teams with a block that fits the ring, several that refill it, one
# row per team of warps, one team of all warps
@pytest.mark.parametrize("storage,m,n,slot", [("f32", 4000, 1000, 1), ("bf16", 20000, 2049, 3), ("f64", 1300, 2049, 0),
                                              ("f32", 3000, 16383, 1)])
def test_a_block_that_never_arrives_ends_the_run(storage, m, n, slot):
    p = workloads.dense_system(m, n, seed=71)
    src = p["A"].astype(np.float64) if storage == "f64" else p["A"]
    with nsli.Solver(src, p["b0"], p["x0"], Av=p["Av"], storage=storage) as s, \
            nsli.Solver(src, p["b0"], p["x0"], Av=p["Av"], storage=storage) as t:
        s.iterate(3, rho=1e-3)
        t.iterate(3, rho=1e-3)
        t0 = time.monotonic()
        assert s.inject_timeout(slot=slot) == nsli.ERR_TIMEOUT
        assert time.monotonic() - t0 < 30.0
        assert s.inject_timeout(slot=1 << 20) == nsli.OK     # no such slot: nothing waits
        np.testing.assert_array_equal(s.get_x(), t.get_x())
        assert s.result() == t.result()
        s.iterate(5, rho=1e-3)
        t.iterate(5, rho=1e-3)
        np.testing.assert_array_equal(s.get_x(), t.get_x())
        a, b = s.result(), t.result()
        assert a == b and a["tick"] == 8
