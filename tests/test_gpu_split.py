"""The kernels that share a row among the warps of a block against those of a
thread per row.

A schedule with explicit slot-group depths keeps the operator and the
smoothing passes at a thread per row; the default one shares rows on small
problems.  Sizes: less than one slice, slices that end inside a grid line,
both sides of the lines between eight and four warps, batches whose
instances converge at different times, both forms of the pressure block."""
import numpy as np
import pytest

import fs_workloads as W
from gpu_helpers import rel_l2

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


def _operator(fs, S, dt, x):
    fs.fs_assemble_step(S.prob, dt)
    y = torch.empty_like(x)
    torch.cuda.synchronize()
    fs.fs_apply_operator(S.prob, x, y)
    torch.cuda.synchronize()
    return y.cpu().numpy()


def _steps(fs, S, schedule):
    x0, t0 = S.state()
    fs.fs_set_schedule(S.prob, 0, 0, **schedule)
    st = fs.fs_step(S.prob, 2)
    assert all(s["status"] == 0 for s in st)
    x = S.state()[0]
    fs.fs_set_state(S.prob, x0, t0)
    return x, sum(s["iters"] for s in st)


SIZES = [W.unit_square(2), W.unit_square(8).with_(n=(3, 40)), W.unit_square(8).with_(n=(33, 7)),
         W.unit_square(40), W.unit_square(64), W.cube(3), W.cube(4).with_(n=(5, 4, 3)),
         W.cube(10), W.cube(13)]


# FP64 sums of at most 65 x 3 products in another order: 1e-13 of the largest
@pytest.mark.parametrize("wl", SIZES)
def test_operator(fs, wl):
    S = fs.Stepper.from_workload(wl)
    try:
        x = torch.from_numpy(np.random.RandomState(3).standard_normal(S.info["n_dof"])).cuda()
        y = _operator(fs, S, wl.dt, x)
        fs.fs_set_schedule(S.prob, 0, 0, spmv_group=4)
        z = _operator(fs, S, wl.dt, x)
        assert np.abs(y - z).max() <= 1e-13 * np.abs(z).max()
    finally:
        S.close()


# the same preconditioner up to rounding: the solutions agree to the solver's
# tolerance and the iteration counts to a few
@pytest.mark.parametrize("schur", [0, 1])
@pytest.mark.parametrize("precision", ["FS_PREC_FP64", "FS_PREC_FP32_REFINE"])
@pytest.mark.parametrize("wl", SIZES)
def test_steps(fs, wl, precision, schur):
    S = fs.Stepper.from_workload(wl, precision=getattr(fs, precision))
    try:
        x, n = _steps(fs, S, dict(schur=schur))
        y, m = _steps(fs, S, dict(schur=schur, spmv_group=4, smooth_group=4))
        assert rel_l2(x, y) <= 1e-9
        assert abs(n - m) <= 3 + 0.05 * m
    finally:
        S.close()


@pytest.mark.parametrize("precision", ["FS_PREC_FP64", "FS_PREC_FP32_REFINE"])
def test_batch(fs, precision):
    wls = [W.unit_square(n, nu=nu, dt=1e-3, jitter=0.0)
           for n, nu in ((3, 1.0), (17, 1e-3), (40, 0.1), (5, 1e-3))]
    S = fs.Stepper.from_workloads(wls, precision=getattr(fs, precision))
    try:
        x, n = _steps(fs, S, {})
        y, m = _steps(fs, S, dict(spmv_group=4, smooth_group=4))
        assert rel_l2(x, y) <= 1e-9
        assert abs(n - m) <= 3 + 0.05 * m
    finally:
        S.close()
