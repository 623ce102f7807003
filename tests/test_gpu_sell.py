"""The operator layout whose column indices are runs, and its padding.

The operator on meshes whose grid lines are shorter than, as long as and
longer than a 32-row slice (no run, several lines per slice, one or two lines),
against the oracle's assembled matrix; a batch whose instances end inside a
slice against the same instances alone; and a batch stepped after kernel
timings left non-finite values in the rows of the Krylov scratch that a
converged instance no longer writes."""
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


def _apply(fs, S, x):
    y = torch.empty_like(x)
    torch.cuda.synchronize()
    fs.fs_apply_operator(S.prob, x, y)
    torch.cuda.synchronize()  # the problem runs on a stream of its own
    return y.cpu().numpy()


# FP64 sums of at most 65 products: 1e-13 of the largest entry of the result
@pytest.mark.parametrize("wl", [
    W.unit_square(8).with_(n=(1, 1)), W.unit_square(8).with_(n=(3, 40)),
    W.unit_square(8).with_(n=(31, 5)), W.unit_square(8).with_(n=(32, 6)),
    W.unit_square(8).with_(n=(33, 7)), W.channel(70, 9), W.cube(1),
    W.cube(4).with_(n=(5, 4, 3)), W.cube(4).with_(n=(31, 3, 2)), W.cube(4).with_(n=(34, 2, 3))])
def test_operator_against_the_oracle(fs, wl):
    S = fs.Stepper.from_workload(wl, dofmap_arrays=True)
    try:
        n = S.info["n_dof"]
        val = torch.empty(S.info["nnz"], dtype=torch.float64, device="cuda")
        fs.fs_assemble_step(S.prob, wl.dt, val)
        torch.cuda.synchronize()
        x = torch.from_numpy(np.random.RandomState(1).standard_normal(n)).cuda()
        rp, col = S.info["rowptr"], S.info["col"]
        full = np.add.reduceat(val.cpu().numpy() * x.cpu().numpy()[col], rp[:-1])
        y = _apply(fs, S, x)
        assert np.abs(y - full).max() <= 1e-13 * np.abs(full).max()
    finally:
        S.close()
    if min(wl.n) < 2:
        return  # no interior vertex in a direction: the step's system is singular
    P = oracle_problem(wl)
    P.step()
    S = fs.Stepper.from_workload(wl, precision=fs.FS_PREC_FP32_REFINE)
    try:
        fs.fs_step(S.prob, 1)
        assert rel_l2(S.state()[0], P.x) <= 1e-9
    finally:
        S.close()


def test_batch_operator_matches_the_instances(fs):
    wls = [W.unit_square(n, nu=0.1, jitter=0.0) for n in (3, 17, 40, 2, 33, 5)]
    B = fs.Stepper.from_workloads(wls)
    try:
        fs.fs_assemble_step(B.prob, wls[0].dt)
        r = np.random.RandomState(2)
        xb = torch.from_numpy(r.standard_normal(B.info["n_dof"])).cuda()
        yb = _apply(fs, B, xb)
        for i, wl in enumerate(wls):
            S = fs.Stepper.from_workload(wl)
            fs.fs_assemble_step(S.prob, wl.dt)
            x = torch.from_numpy(B.instance_state(xb.cpu().numpy(), i)).cuda()
            y = _apply(fs, S, x)
            S.close()
            assert np.abs(B.instance_state(yb, i) - y).max() <= 1e-13 * np.abs(y).max()
    finally:
        B.close()


def test_converged_instances_do_not_reach_the_others(fs):
    # instance 0 converges first (a viscous square); its skipped rows keep
    # what the timings left there
    wls = [W.unit_square(4, nu=1.0, dt=1e-3, jitter=0.0)] + \
        [W.unit_square(n, nu=1e-3, dt=1e-3, jitter=0.0) for n in (23, 37, 18)]
    S = fs.Stepper.from_workloads(wls, precision=fs.FS_PREC_FP32_REFINE)
    try:
        fs.fs_step(S.prob, 1)
        for k in (fs.FS_KERNEL_CGS, fs.FS_KERNEL_CGS_UPD, fs.FS_KERNEL_CGS_FIN):
            fs.fs_profile_kernel(S.prob, k, 60)
        st = fs.fs_step(S.prob, 3)
        assert all(s["status"] == 0 for s in st)
        assert np.isfinite(S.state()[0]).all()
    finally:
        S.close()
