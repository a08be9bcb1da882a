"""A new tick alone: set by a copy, or by a kernel where the stream is being
captured (a graph that is replayed later has to hold the value itself)."""
import numpy as np
import pytest

from paper_2003_09956_gb300 import nsli, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="session", autouse=True)
def built_library():
    from paper_2003_09956_gb300 import _build
    _build.build()
    nsli.load()


def test_tick_set_by_a_call_and_in_a_captured_graph():
    import torch
    p = workloads.dense_system(400, 100, seed=4)
    stream = torch.cuda.Stream()
    with nsli.Solver(p["A"], p["b0"], p["x0"], Av=p["Av"], stream=stream.cuda_stream) as s, \
            nsli.Solver(p["A"], p["b0"], p["x0"], Av=p["Av"]) as t:
        for k in range(50):              # one call after another, none waited for
            s.update_b(tick=k)
        s.update_b(tick=7)
        s.iterate(1, rho=1e-2)
        s.sync()
        assert s.result()["tick"] == 8
        s.set_x(p["x0"])
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
            s.update_b(tick=1 << 40)
            s.iterate(2, rho=1e-9)
        s.update_b(tick=3)
        s.sync()                         # (the graph is replayed on another stream)
        graph.replay()
        graph.replay()
        torch.cuda.synchronize()
        assert s.result()["tick"] == (1 << 40) + 2
        for _ in range(2):
            t.update_b(tick=1 << 40)
            t.iterate(2, rho=1e-9)
        np.testing.assert_array_equal(s.get_x(), t.get_x())
