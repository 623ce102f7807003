"""fs_autotune leaves an explicit slot depth: on a small FP64 problem the
shared-row kernels, which only depth 0 selects, take about half the time."""
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


@pytest.mark.parametrize("group", [4, 6, 8])
def test_back_to_shared_rows(fs, group):
    S = fs.Stepper.from_workload(W.cube(12), precision=fs.FS_PREC_FP64)
    try:
        fs.fs_set_schedule(S.prob, 0, 0, spmv_group=group)
        r = fs.fs_autotune(S.prob, reps=30)
        assert r["best"]["spmv_group"] == 0
        assert fs.fs_get_schedule(S.prob)["spmv_group"] == 0
        assert r["spmv_best_ms"] < 0.8 * r["spmv_default_ms"]
    finally:
        S.close()
