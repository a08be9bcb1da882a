"""Every entry of a row counts once in the squared norm behind its record, at
lengths around the set-up and update kernels' steps (256 threads; two, four
and eight entries each), for rows created and rows replaced.

x has one non-zero entry and r = 1 exactly, so y = a / ||a||^2 with no rounding
but the record's and two products': an entry lost or taken twice shows, its
share of the norm being 5e-6 or more against a tolerance of 5e-7."""
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
        return oracle.quantize_e4m3_rows(A32)[0]
    return A32


# 1 / ||a||^2 rounded to binary32, times r (and FP8's scale, a power of two),
# times a: three roundings of 2^-24 relative each, and one for margin; the
# quick norm itself is good to about 1e-12
TOL = 4 * 2.0 ** -24


@pytest.mark.parametrize("storage", ["f32", "bf16", "fp8"])
@pytest.mark.parametrize("n", [1, 2, 3, 255, 256, 257, 511, 513, 767, 769, 1023, 1024, 1025, 1281, 1793, 2047, 2048,
                               2049, 2305, 4099])
def test_every_entry_counts_once(storage, n):
    rng = np.random.default_rng(n)
    plain = rng.uniform(0.5, 1.0, n).astype(np.float32)
    # entries on both sides of 2^-60, where the squares are taken in binary64
    tiny = plain * np.where(np.arange(n) % 3 == 0, np.float32(2.0 ** -58), np.float32(2.0 ** -60)).astype(np.float32)
    plain[0], tiny[0] = 1.0, 2.0 ** -58

    def system(row):
        q = np.asarray(stored_values(row[None, :], storage), np.float64)[0]
        assert q[0] == row[0]
        x = np.zeros(n)
        x[0] = 2.0 / row[0]             # a . x = 2, b = 1
        n2 = float(np.dot(q, q))
        assert (q * q).min() / n2 > 5e-6
        return x, q / n2

    one = np.ones(1)
    for first, second in ((plain, tiny), (tiny, plain)):
        x, want = system(second)
        with nsli.Solver(second[None, :].copy(), one, x, storage=storage) as s, \
                nsli.Solver(first[None, :].copy(), one, x, storage=storage) as t:
            t.update_rows(0, second[None, :].copy(), b0=one)
            (y, h, _), (z, k, _) = s.map_reduce(), t.map_reduce()
            assert h == k == 1
            assert np.all(np.abs(y - want) <= TOL * np.abs(want))
            np.testing.assert_array_equal(y, z)


@pytest.mark.parametrize("n", [1, 2, 255, 256, 257, 1793, 2047, 2048, 2049, 2305, 4099])
def test_every_entry_counts_once_in_the_batched_form(n):
    """The batched form's binary64 norms (eight entries per thread and step):
    one violated row; y within 16 roundings of 2^-23 (1 / ||a||^2, the weight's
    three bf16 terms and their products' sum), an entry's share 5e-5 or more."""
    rng = np.random.default_rng(n)
    m = 130
    A = oracle.quantize_bf16(rng.uniform(0.5, 1.0, (m, n)).astype(np.float32))
    A[:, 0] = 1.0
    q = A[7].astype(np.float64)
    assert (q * q).min() / np.dot(q, q) > 5e-5
    b = np.full(m, 100.0)
    b[7] = 1.0
    X = np.zeros((2, n))
    X[:, 0] = 2.0, 3.0
    with nsli.BatchSolver(A, b, X) as s:
        Y, h, _ = s.map_reduce()
    for k in range(2):
        want = (1.0 + k) * q / np.dot(q, q)
        assert h[k] == 1
        assert np.all(np.abs(Y[k] - want) <= 16 * 2.0 ** -23 * want)
