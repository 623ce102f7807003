"""The bytes fs_profile_kernel counts for the operator kernels: values and
vectors once, and the offsets and columns the layout has the kernels read, 8
bytes per slot of 32 rows where the columns are runs (nearly all slices of a
mesh whose grid lines are longer than a slice)."""
import numpy as np
import pytest

import fs_workloads as W

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


@pytest.mark.parametrize("wl", [W.unit_square(120), W.channel(200, 40), W.cube(34)],
                         ids=lambda w: w.name)
def test_operator_bytes(fs, wl):
    S = fs.Stepper.from_workload(wl, precision=fs.FS_PREC_FP32_REFINE, dofmap_arrays=True)
    try:
        d, nv, n2, n = (S.info[k] for k in ("dim", "n_vert", "n_p2", "n_dof"))
        nnzb = (np.diff(S.info["rowptr"])[d * n2:].sum() - nv) // d
        nnza = (S.info["nnz"] - 2 * d * nnzb - nv) // d
        for kernel, size in ((fs.FS_KERNEL_SPMV, 4), (fs.FS_KERNEL_SPMV_FP64, 8)):
            by = fs.fs_profile_kernel(S.prob, kernel, 3)[1]
            index = by - size * (nnza + 2 * d * nnzb + nv + 2 * n)
            assert 0 < index <= 0.4 * 4 * (nnza + 2 * nnzb)
        index = fs.fs_profile_kernel(S.prob, fs.FS_KERNEL_CHEB, 3)[1] - 4 * (nnza + n2 + 5 * d * n2)
        assert 0 < index <= 0.4 * 4 * nnza
    finally:
        S.close()


# one segment in one block's reach, streamed, and a batch
@pytest.mark.parametrize("wls", [[W.unit_square(40)], [W.unit_square(290, nu=0.01, dt=1e-3)],
                                 [W.unit_square(n, jitter=0.0) for n in (30, 7, 41)]],
                         ids=["one", "streamed", "batch"])
def test_orthogonalisation_as_a_step_runs_it(fs, wls):
    S = fs.Stepper.from_workloads(wls, precision=fs.FS_PREC_FP32_REFINE) if len(wls) > 1 else \
        fs.Stepper.from_workload(wls[0], precision=fs.FS_PREC_FP32_REFINE)
    try:
        fs.fs_step(S.prob, 1)
        x0, t0 = S.state()
        ms, by = fs.fs_profile_kernel(S.prob, fs.FS_KERNEL_ORTH, 20)
        both = fs.fs_profile_kernel(S.prob, fs.FS_KERNEL_CGS, 20)[0]
        assert by == (2 * 15 + 5) * S.info["n_dof"] * 4 and 0 < ms < both
        x, t = S.state()
        assert (x == x0).all() and t == t0
        assert fs.fs_step(S.prob, 1)[0]["status"] == 0
    finally:
        S.close()
