"""The orthogonalisation kernels at the edges of their work-lists.

One block, a share of a few entries more than a block holds, odd vector
lengths (bulk copies start at padded rows), a batch whose instances end inside
a 16-byte unit, and a vector long enough for the streaming kernel.  Each
stepped state is compared with the oracle's steps, or (the long vectors, where
the oracle takes minutes) with the FP64 path, to the 1e-9 relative L2 that
every solution meets."""
import numpy as np
import pytest

import fs_workloads as W
from gpu_helpers import oracle_problem, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_25403_gb300 import build
    build.build()
    from paper_2605_25403_gb300 import fs as mod
    return mod


def _state(fs, wl, prec, steps):
    S = fs.Stepper.from_workload(wl, precision=prec)
    try:
        st = fs.fs_step(S.prob, steps)
        assert all(s["status"] == 0 for s in st)
        return S.state()[0]
    finally:
        S.close()


# (cells per axis): 59, 187 and 278 unknowns (one block in FP32), 514 (two
# blocks), 1,098 and 2,467 (ragged shares in both types)
@pytest.mark.parametrize("prec", ["FS_PREC_FP64", "FS_PREC_FP32_REFINE"])
@pytest.mark.parametrize("n", [(2, 2), (4, 4), (5, 5), (7, 7), (11, 10), (16, 16)])
def test_small_vectors(fs, n, prec):
    wl = W.unit_square(8, nu=0.05).with_(n=n)
    P = oracle_problem(wl)
    for _ in range(2):
        P.step()
    assert rel_l2(_state(fs, wl, getattr(fs, prec), 2), P.x) <= 1e-9


@pytest.mark.parametrize("prec", ["FS_PREC_FP64", "FS_PREC_FP32_REFINE"])
def test_batch_of_ragged_instances(fs, prec):
    wls = [W.unit_square(n, nu=nu, jitter=0.0) for n, nu in
           ((3, 1.0), (8, 0.01), (5, 0.1), (13, 0.02), (2, 1.0), (29, 0.005))]
    S = fs.Stepper.from_workloads(wls, precision=getattr(fs, prec))
    try:
        fs.fs_step(S.prob, 2)
        x, _ = S.state()
        for i, wl in enumerate(wls):
            P = oracle_problem(wl)
            for _ in range(2):
                P.step()
            assert rel_l2(S.instance_state(x, i), P.x) <= 1e-9
    finally:
        S.close()


# 739,027 unknowns in two dimensions (more than 4,096 per SM, odd length) and
# 709,971 in three
@pytest.mark.parametrize("wl", [W.unit_square(286, nu=0.01, dt=1e-3, jitter=0.0),
                                W.cube(30).with_(n=(30, 29, 31))])
def test_streamed_vectors(fs, wl):
    a = _state(fs, wl, fs.FS_PREC_FP32_REFINE, 2)
    b = _state(fs, wl, fs.FS_PREC_FP64, 2)
    assert rel_l2(a, b) <= 1e-9
