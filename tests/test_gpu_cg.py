"""The one-launch CG solves of the pressure-correction stages at the edges of
their dispatch: one block, rows short of a warp, eight lanes per row against
one (P3/P2, 19,456 rows on a 152-SM chip), several sweeps of the chip, three
components, and an iteration cap; every state against the oracle's step of the
scheme, to the 1e-9 relative L2 that every solution meets."""
import pytest

import fs_workloads as W
from gpu_helpers import oracle_problem, rel_l2
from oracle import oracle as O
from oracle import p3p2 as Q

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


def _stepped(fs, S, steps):
    try:
        st = fs.fs_step_ipcs(S.prob, steps)
        assert all(s["status"] == 0 and max(s["rel_res"]) <= 1e-11 for s in st)
        return S.state()[0]
    finally:
        S.close()


@pytest.mark.parametrize("wl", [
    W.unit_square(8, nu=0.05).with_(n=(2, 2)), W.unit_square(8, nu=0.05).with_(n=(3, 9)),
    W.unit_square(8, nu=0.05).with_(n=(70, 3)),
    W.unit_square(8, nu=0.02, dt=5e-3).with_(n=(142, 140)),
    W.cube(2, nu=0.1, dt=0.01), W.cube(4, nu=0.1, dt=0.01).with_(n=(5, 4, 3))],
    ids=lambda w: "x".join(map(str, w.n)))
def test_p2_steps_match_the_oracle(fs, wl):
    steps = 1 if wl.ndof > 10000 else 2
    P = oracle_problem(wl)
    for _ in range(steps):
        O.ipcs_step(P)
    assert rel_l2(_stepped(fs, fs.Stepper.from_workload(wl), steps), P.x) <= 1e-9


@pytest.mark.parametrize("n", [(2, 2), (3, 5), (46, 46), (47, 47)],
                         ids=lambda n: "x".join(map(str, n)))
def test_p3_steps_match_the_oracle(fs, n):
    wl = W.unit_square(8, nu=0.02, dt=5e-3, jitter=0.05, seed=4).with_(n=n)
    P = Q.Problem3(n=wl.n, problem=wl.problem, nu=wl.nu, dt=wl.dt, jitter=wl.jitter,
                   seed=wl.seed, wconst=wl.wconst)
    for _ in range(2):
        P.ipcs_step()
    assert rel_l2(_stepped(fs, fs.Stepper.from_workload_p3(wl), 2), P.x) <= 1e-9


def test_iteration_cap(fs):
    S = fs.Stepper.from_workload(W.unit_square(12, nu=0.02, dt=5e-3))
    try:
        st = fs.fs_step_ipcs(S.prob, 1, max_iter=5, raise_on_error=False)[0]
        assert st["status"] == 5 and st["iters"][0] == 5
    finally:
        S.close()
