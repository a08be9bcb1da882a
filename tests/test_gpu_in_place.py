"""New x and right-hand sides read from device memory in place: a buffer that
ends with its allocation, a part of one, one that is not aligned for a
kernel's loads, and host memory give the same state."""
import numpy as np
import pytest

from paper_2003_09956_gb300 import nsli, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="session", autouse=True)
def built_library():
    from paper_2003_09956_gb300 import _build
    _build.build()
    nsli.load()


@pytest.mark.parametrize("n", [1, 513, 262144])
def test_buffers_at_any_place_of_an_allocation(n):
    import torch
    m = 3
    p = workloads.dense_system(m, n, seed=n)
    rng = np.random.default_rng(n)
    x, b = rng.normal(size=n), rng.normal(size=m)

    def at_the_end(v):       # the allocation's last bytes (2 MiB: a block of its own)
        buf = torch.empty(1 << 18, dtype=torch.float64, device="cuda")
        out = buf[buf.numel() - len(v):]
        return out.copy_(torch.from_numpy(v))

    def odd(v):              # 4 bytes past an 8-byte boundary
        raw = torch.empty(8 * len(v) + 8, dtype=torch.uint8, device="cuda")
        raw[4:4 + 8 * len(v)] = torch.from_numpy(v.view(np.uint8).copy()).cuda()
        return raw[4:4 + 8 * len(v)]

    with nsli.Solver(p["A"], p["b0"], p["x0"], Av=p["Av"]) as s:
        states = []
        for put in (lambda v: v, lambda v: torch.from_numpy(v).cuda(), at_the_end, odd):
            gx, gb = put(x), put(b)
            torch.cuda.synchronize()
            ptr = (lambda v: v.ctypes.data if isinstance(v, np.ndarray) else v.data_ptr())
            lib = nsli.load()
            assert lib.nsli_set_x(s._h, ptr(gx)) == nsli.OK
            assert lib.nsli_update_b(s._h, ptr(gb), 4) == nsli.OK
            s.iterate(1, rho=1e-3)
            states.append(s.get_x())
        for st in states[1:]:
            np.testing.assert_array_equal(st, states[0])
