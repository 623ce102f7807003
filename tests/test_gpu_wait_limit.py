"""Waits that run out, through the public calls: with a limit of 0 a solve ends
in FS_ERR_TIMEOUT (launched directly and as a graph with a loop node), and with
the limit back the problem steps as one that never timed out."""
import pytest

import fs_workloads as W
from gpu_helpers import rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
SQUARE = W.unit_square(96, nu=0.02, dt=1e-3, jitter=0.0)


@pytest.fixture(scope="module")
def fs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_25403_gb300 import build
    build.build()
    from paper_2605_25403_gb300 import fs as mod
    return mod


def _problem(fs, kind, precision):
    if kind == "batch":
        return fs.Stepper.from_workloads([SQUARE.with_(n=(n, n)) for n in (60, 71, 33, 90)],
                                         precision=precision)
    wl = W.unit_square(290, nu=0.01, dt=1e-3, jitter=0.0) if kind == "streamed" else SQUARE
    return fs.Stepper.from_workload(wl, precision=precision)


@pytest.mark.parametrize("graph", [0, 1])
@pytest.mark.parametrize("kind,precision", [("one", "FS_PREC_FP32_REFINE"), ("one", "FS_PREC_FP64"),
                                            ("streamed", "FS_PREC_FP32_REFINE"),
                                            ("batch", "FS_PREC_FP32_REFINE"),
                                            ("batch", "FS_PREC_FP64")])
def test_a_step_times_out_and_the_next_is_clean(fs, kind, precision, graph):
    opts = fs.fs_default_solve_opts(use_graph=graph)
    S, T = (_problem(fs, kind, getattr(fs, precision)) for _ in range(2))
    try:
        x0, t0 = S.state()
        fs.fs_set_wait_limit(S.prob, 0.0)
        st = fs.fs_step(S.prob, 1, opts, raise_on_error=False)
        assert st[0]["status"] == 7
        with pytest.raises(fs.FsError, match="limit"):
            fs.fs_set_state(S.prob, x0, t0)
            fs.fs_step(S.prob, 1, opts)
        fs.fs_set_wait_limit(S.prob, 1.0)
        fs.fs_set_state(S.prob, x0, t0)
        for P in (S, T):
            assert fs.fs_step(P.prob, 1, opts)[0]["status"] == 0
        assert rel_l2(S.state()[0], T.state()[0]) <= 1e-9
    finally:
        S.close()
        T.close()


def test_ipcs_times_out_and_the_next_is_clean(fs):
    S, T = (fs.Stepper.from_workload(SQUARE) for _ in range(2))
    try:
        x0, t0 = S.state()
        fs.fs_set_wait_limit(S.prob, 0.0)
        assert fs.fs_step_ipcs(S.prob, 1, raise_on_error=False)[0]["status"] == 7
        fs.fs_set_wait_limit(S.prob, 1.0)
        fs.fs_set_state(S.prob, x0, t0)
        for P in (S, T):
            assert fs.fs_step_ipcs(P.prob, 1)[0]["status"] == 0
        assert rel_l2(S.state()[0], T.state()[0]) <= 1e-9
    finally:
        S.close()
        T.close()


def test_limits_out_of_range_are_refused(fs):
    S = fs.Stepper.from_workload(W.unit_square(4))
    try:
        for bad in (-1.0, 61.0):
            with pytest.raises(fs.FsError):
                fs.fs_set_wait_limit(S.prob, bad)
    finally:
        S.close()
