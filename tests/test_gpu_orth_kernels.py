"""The orthogonalisation kernels alone, on vectors and work-lists made for one
property each."""
import numpy as np
import pytest

import orth_harness as H

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ONE = H.one(500, 128, 3)                       # four blocks
MANY = H.many([700, 301, 5, 2049], 256, 6, 3)  # segments end inside 16-byte units


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return H.compile_harness("orth_harness.cu")


@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("case", [ONE, MANY], ids=["one", "many"])
def test_the_loop_ends_when_every_segment_is_done(lib, case, f32):
    # the condition was left set behind a wait that ran out
    assert H.loop_passes(lib, f32, case, max_pass=6) == 1


# blocks that never come: every block's wait ends at its limit, the segments
# are marked, and a launch with its counters reset is clean
@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("many", [False, True])
def test_a_wait_that_runs_out_is_reported(lib, many, f32):
    r = np.random.RandomState(1)
    for absent in (1, 0):
        kw = dict(wait_ns=2 * 10**6 if absent else 10**9, absent=absent)
        case = H.many([700, 301, 5, 2049], 256, 6, 3, **kw) if many else H.one(500, 128, 3, **kw)
        c, seg0 = case
        V = np.concatenate([H.basis(r, 3, k) for k in np.diff(seg0)], axis=1)
        out = H.step(lib, f32, case, V)
        if absent:
            assert (out["seg"][:, :2] == [2, 1]).all() and out["ctl"][1] == 1
        else:
            assert (out["seg"][:, :2] == 0).all() and out["ctl"][:2].tolist() == [4, 0]
