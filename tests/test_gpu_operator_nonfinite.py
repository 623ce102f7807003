"""fs_apply_operator on vectors with entries that are not finite: the rows that
couple to them, by the matrix' pattern, and no others."""
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


def _apply(fs, S, x):
    x = torch.from_numpy(x).cuda()
    y = torch.empty_like(x)
    torch.cuda.synchronize()
    fs.fs_apply_operator(S.prob, x, y)
    torch.cuda.synchronize()
    return y.cpu().numpy()


def _rows(rp, col, entries):
    row = np.repeat(np.arange(len(rp) - 1), np.diff(rp))
    hit = np.zeros(len(rp) - 1, dtype=bool)
    hit[row[np.isin(col, entries)]] = True
    return hit


# slices of several grid lines, of one or two, and in 3D; problems whose rows
# are shared by the warps of a block (the default) and a thread per row
@pytest.mark.parametrize("group", [0, 4])
@pytest.mark.parametrize("wl", [W.unit_square(8).with_(n=(3, 40)), W.unit_square(8).with_(n=(33, 7)),
                                W.channel(70, 9), W.cube(4).with_(n=(5, 4, 3)),
                                W.cube(4).with_(n=(34, 3, 2))],
                         ids=lambda w: w.name + "_" + "x".join(map(str, w.n)))
def test_rows_reached(fs, wl, group):
    S = fs.Stepper.from_workload(wl, dofmap_arrays=True)
    try:
        if group:
            fs.fs_set_schedule(S.prob, 0, 0, spmv_group=group)
        fs.fs_assemble_step(S.prob, wl.dt)
        n, rp, col = S.info["n_dof"], S.info["rowptr"], S.info["col"]
        r = np.random.RandomState(1)
        base = r.standard_normal(n)
        y0 = _apply(fs, S, base)
        assert np.isfinite(y0).all()
        nv = S.info["n_vert"]
        # one entry at a time: velocity nodes of every kind, pressures
        picks = list(r.randint(0, n - nv, 12)) + list(r.randint(n - nv, n, 6)) + [0, n - 1]
        for k, bad in zip(picks, [np.nan, np.inf, -np.inf] * 7):
            x = base.copy()
            x[k] = bad
            y = _apply(fs, S, x)
            hit = _rows(rp, col, [k])
            assert (np.isfinite(y) == ~hit).all()
            assert (y[~hit] == y0[~hit]).all()
    finally:
        S.close()


def test_instances_of_a_batch_stay_apart(fs):
    wls = [W.unit_square(n, nu=0.1, jitter=0.0) for n in (3, 17, 40, 2, 33, 5)]
    B = fs.Stepper.from_workloads(wls)
    try:
        fs.fs_assemble_step(B.prob, wls[0].dt)
        n = B.info["n_dof"]
        x = np.random.RandomState(2).standard_normal(n)
        y0 = _apply(fs, B, x)
        owner = np.arange(n, dtype=np.float64)
        for i in range(len(wls)):
            mine = B.instance_state(owner, i).astype(np.int64)
            z = x.copy()
            z[mine] = np.nan
            y = _apply(fs, B, z)
            rest = np.setdiff1d(np.arange(n), mine)
            assert (y[rest] == y0[rest]).all()
    finally:
        B.close()
