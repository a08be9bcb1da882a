"""The squared norm behind a row's record (the quick sum of two entries at a
time) at odd lengths and at entries whose squares leave the binary32 range,
for rows created and rows replaced: one violated row, so that y is
r / ||a||^2 a (Eq. 7) and shows the norm."""
import numpy as np
import pytest

import oracle
from paper_2003_09956_gb300 import nsli

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="session", autouse=True)
def built_library():
    from paper_2003_09956_gb300 import _build
    _build.build()
    nsli.load()


def stored_values(A32, storage):
    if storage == "bf16":
        return oracle.quantize_bf16(A32)
    if storage == "fp8":
        q, _ = oracle.quantize_e4m3_rows(A32)
        return q
    return A32


@pytest.mark.parametrize("storage", ["f32", "bf16", "fp8"])
@pytest.mark.parametrize("n", [1, 2, 255, 257, 511, 513, 4099])
def test_norm_of_a_row_created_and_replaced(storage, n):
    rng = np.random.default_rng(n)
    # the second row's entries lie on both sides of 2^-60, where the squares
    # are taken in binary64
    plain = rng.uniform(0.25, 1.0, n).astype(np.float32)
    tiny = plain * np.where(np.arange(n) % 3 == 0, np.float32(2.0 ** -58), np.float32(2.0 ** -60)).astype(np.float32)
    x = rng.uniform(0.25, 1.0, n)
    x = x.astype(np.float32).astype(np.float64)

    def system(row):
        q = np.asarray(stored_values(row[None, :].astype(np.float32), storage), np.float64)[0]
        t = float(np.dot(np.abs(q), np.abs(x)))
        b = float(np.dot(q, x)) - t        # r = t > 0
        return np.array([b]), t / float(np.dot(q, q)) * q

    # binary32 sums of n products, b, r, the coefficient and its product:
    # each within 2^-24 of terms of at most 2 t
    tol = (n + 16) * 2.0 ** -22
    for first, second in ((plain, tiny), (tiny, plain)):
        b, want = system(first)
        with nsli.Solver(first[None, :].copy(), b, x, storage=storage) as s:
            y, h, _ = s.map_reduce()
            assert h == 1
            assert np.max(np.abs(y - want)) <= tol * np.max(np.abs(want))
            b, want = system(second)
            s.update_rows(0, second[None, :].copy(), b0=b)
            y, h, _ = s.map_reduce()
            assert h == 1
            assert np.max(np.abs(y - want)) <= tol * np.max(np.abs(want))
