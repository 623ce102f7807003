"""The solution update of a restart cycle, x += Z H^-1 g, alone."""
import ctypes

import numpy as np
import pytest

from orth_harness import _ptr, compile_harness

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return compile_harness("update_harness.cu")


def _update(lib, f32, H, g, Z, x):
    k, n = Z.shape
    H, g, Z, x = (np.array(a, dtype=np.float64, order="C") for a in (H, g, Z, x))
    assert lib.update_x(int(f32), ctypes.c_int64(n), k, _ptr(H), _ptr(g), _ptr(Z), _ptr(x)) == 0
    return x


# FP64 bound of k products and sums: (k + 2) 2^-53 of the sum of their sizes,
# the triangle's solution (of condition below 4) likewise; FP32 results are
# rounded to 2^-24
@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("k,n", [(1, 1), (2, 33), (3, 2049), (4, 511), (17, 5000), (30, 2048)])
def test_update_against_extended_precision(lib, k, n, f32):
    r = np.random.RandomState(k)
    H = np.triu(r.uniform(-1, 1, (k, k)) / (2 * k)) + np.diag(r.uniform(1, 2, k))
    g, Z, x = r.standard_normal(k), r.standard_normal((k, n)), r.standard_normal(n)
    if f32:
        Z, x = Z.astype(np.float32).astype(np.float64), x.astype(np.float32).astype(np.float64)
    y = np.zeros(k, dtype=np.longdouble)
    for i in range(k - 1, -1, -1):
        y[i] = (np.longdouble(g[i]) - H[i, i + 1:].astype(np.longdouble) @ y[i + 1:]) / H[i, i]
    want = x.astype(np.longdouble) + y @ Z.astype(np.longdouble)
    size = np.abs(x) + np.abs(y).astype(np.float64) @ np.abs(Z)
    got = _update(lib, f32, H, g, Z, x)
    assert (np.abs(got - want) <= 16 * (k + 2) * 2.0 ** -53 * size
            + (2.0 ** -24 if f32 else 0) * np.abs(want)).all()


# two directions that cancel to 2^-46 of their size: FP64 sums are within
# 2 roundings of 2^-53, sums of FP32 pairs (48 bits) are not
def test_fp32_directions_are_added_in_fp64(lib):
    r = np.random.RandomState(1)
    n = 4000
    z = r.uniform(1, 2, n).astype(np.float32).astype(np.float64)
    y0 = 1 + r.randint(1, 2 ** 52) * 2.0 ** -52
    y = np.array([y0, -(y0 - 2.0 ** -46)])
    want = (z.astype(np.longdouble) * (np.longdouble(y[0]) + np.longdouble(y[1]))).astype(np.float64)
    got = _update(lib, True, np.eye(2), y, np.stack([z, z]), np.zeros(n))
    assert (np.abs(got - want) <= 2 * 2.0 ** -52 * z + 2.0 ** -24 * np.abs(want)).all()
    four = _update(lib, True, np.eye(4), np.array([y[0], y[1], 0.0, 0.0]),
                   np.stack([z, z, z, z]), np.zeros(n))
    assert (np.abs(four - want) <= 2 * 2.0 ** -52 * z + 2.0 ** -24 * np.abs(want)).all()


# entries whose bits are not those of a normal number, and coefficients beyond
# the range that the widened entries leave
def test_entries_and_coefficients_at_the_ends_of_their_range(lib):
    tiny, big = 2.0 ** -149, float(np.finfo(np.float32).max)
    z = np.array([0.0, -0.0, tiny, -7 * tiny, 2.0 ** -126, big, -big, np.inf, -np.inf, np.nan, 1.0])
    Z = np.stack([z, np.ones_like(z), np.ones_like(z), np.zeros_like(z), z])
    for y in ([2.0 ** 60, 0.5, 0.25, 1.0, 0.0], [2.0 ** 130, 0.0, 0.0, 3.0, 2.0 ** -40]):
        with np.errstate(invalid="ignore", over="ignore"):
            want = (np.array(y) @ Z).astype(np.float32)
        got = _update(lib, True, np.eye(5), y, Z, np.zeros_like(z))
        ok = np.isfinite(want)
        assert (np.isnan(got) == np.isnan(want)).all()
        assert (got[np.isinf(want)] == want[np.isinf(want)]).all()
        assert np.allclose(got[ok], want[ok].astype(np.float64), rtol=2.0 ** -23, atol=0)
