"""Dense systems of few rows: which form their iterations take by default (one
launch, or Map and Reduce launches where a block would have many columns to
reduce), and the same results either way."""
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


def stored(A32, storage):
    if storage == "bf16":
        return oracle.quantize_bf16(A32)
    return oracle.quantize_e4m3_rows(A32)[0] if storage == "fp8" else A32


@pytest.mark.parametrize("storage,m,n", [
    ("f32", 1, 224), ("f32", 1, 225), ("f32", 1, 16384), ("f32", 20, 8000), ("f32", 36, 8000), ("f32", 40, 8192),
    ("f32", 251, 2500), ("f32", 501, 5000), ("f32", 608, 2049), ("f32", 609, 2049), ("f32", 601, 16383),
    ("f64", 1, 96), ("f64", 1, 97), ("f64", 20, 4000), ("f64", 90, 8192), ("f64", 251, 2500),
    ("bf16", 300, 6000), ("bf16", 5, 4097), ("fp8", 600, 9000), ("fp8", 3, 16384)])
def test_few_rows(storage, m, n):
    import torch
    p = workloads.dense_system(m, n, seed=7 * n + m)
    src = p["A"].astype(np.float64) if storage == "f64" else p["A"]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    blocks = -(-n // 32)
    one_launch = blocks <= (3 if storage == "f64" else 7) * min(m, sms)
    for rule, lam in (("relaxed", 1.0), ("modap", 5.0 / np.sqrt(n))):
        with nsli.Solver(src, p["b0"], p["x0"], Av=p["Av"], storage=storage) as a, \
                nsli.Solver(src, p["b0"], p["x0"], Av=p["Av"], storage=storage) as b:
            y, h, st = a.map_reduce()
            parity.check_map_reduce(y, h, st, stored(p["A"], storage), p["b0"], p["x0"], storage,
                                    depth=parity.dense_y_depth(m, sms), levels=parity.dot_levels(n))
            c0 = a.launch_count()
            a.iterate(11, lam=lam, rule=rule, rho=1e-3)
            a.sync()
            assert a.launch_count() - c0 == (2 if one_launch else 1 + 2 * 11)
            b.iterate(11, lam=lam, rule=rule, rho=1e-3, block_iters=4)
            np.testing.assert_array_equal(a.get_x(), b.get_x())
            assert a.result()["tick"] == b.result()["tick"] == 11
