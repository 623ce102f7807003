"""The waits of the one-launch CG solve: blocks that never come end it at its
limit with the error mark, and a solve after it is clean."""
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
    return compile_harness("cg_harness.cu")


@pytest.mark.parametrize("lanes", [1, 8])
def test_a_wait_that_runs_out_is_reported(lib, lanes):
    n = 700  # 1D Laplacian plus a mass term: condition about 40
    rp = np.minimum(np.maximum(3 * np.arange(n + 1) - 1, 0), 3 * n - 2).astype(np.int32)
    ci = np.concatenate([[j for j in (i - 1, i, i + 1) if 0 <= j < n] for i in range(n)])
    ci = ci.astype(np.int32)
    v = np.where(ci == np.repeat(np.arange(n), np.diff(rp)), 2.1, -1.0)
    b = np.random.RandomState(1).standard_normal(n)
    A = np.zeros((n, n))
    A[np.repeat(np.arange(n), np.diff(rp)), ci] = v
    for absent, wait_ns in ((1, 2 * 10**6), (0, 10**9)):
        x, out, res = np.zeros(n), np.zeros(2, dtype=np.int32), np.zeros(2)
        rc = lib.cg_solve(ctypes.c_int64(n), _ptr(rp), _ptr(ci), _ptr(v), _ptr(b), _ptr(x), lanes,
                          7, absent, ctypes.c_uint64(wait_ns), ctypes.c_double(1e-12), 2000,
                          _ptr(out), _ptr(res))
        assert rc == 0
        if absent:
            assert out[1] == 1
        else:  # relative residual 1e-12, condition 40
            assert out[1] == 0 and res[0] <= 1e-23 * res[1]
            assert np.linalg.norm(x - np.linalg.solve(A, b)) <= 1e-10 * np.linalg.norm(x)
