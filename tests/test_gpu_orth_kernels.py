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


# a limit of 0: the waits for bulk copies run out while the copies are under
# way; the blocks end behind their copies and a launch after them is clean
def test_expired_ring_waits_end_behind_their_copies(lib):
    r = np.random.RandomState(2)
    lens = [20001, 7, 30002]
    V = np.concatenate([H.basis(r, 3, k) for k in lens], axis=1)
    for wait_ns in (0, 10**9):
        out = H.step(lib, True, H.many(lens, 2048, 8, 3, wait_ns=wait_ns), V)
        if wait_ns == 0:
            assert (out["seg"][:, :2] == [2, 1]).all() and out["ctl"][1] == 1
        else:
            assert (out["seg"][:, :2] == 0).all() and out["ctl"][:2].tolist() == [4, 0]
            w, q = out["w"], V[:4]
            for s, e in zip(np.cumsum([0] + lens[:-1]), np.cumsum(lens)):
                # FP32 rows of norm 1: entries rounded to 6e-8, a few operations each
                assert np.abs(q[:, s:e] @ w[s:e]).max() <= 1e-6
                assert abs(np.linalg.norm(w[s:e]) - 1) <= 1e-6


# from the first step to the longest basis the kernels hold; FP32 rows carry
# 6e-8 per entry, and a sum of 31 products of such entries 31 times that
@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("j", [0, 7, 29, 30])
@pytest.mark.parametrize("many", [False, True])
def test_step_against_extended_precision(lib, many, j, f32):
    r = np.random.RandomState(3)
    case = H.many([700, 301, 33, 2049], 256, 6, j) if many else H.one(1501, 512, j, LU=1)
    V = np.concatenate([H.basis(r, j, k) for k in np.diff(case[1])], axis=1)
    new, h, E = H.reference(V, case[1], np.float32 if f32 else np.float64)
    out = H.step(lib, f32, case, V, E)
    u = 6e-8 if f32 else 1.2e-16
    assert (out["seg"][:, 0] == 0).all() and out["ctl"][0] == j + 1
    assert np.abs(out["h"] - h).max() <= 20 * u
    assert np.abs(out["w"] - new).max() <= 100 * u


# FP32 sums run over 128 products and are added in FP64: entries whose sums of
# up to 128 are exact in FP32 (1 + 2^-22 times powers of two) give an exact
# projection, where a lane's longer FP32 sum drops the 2^-22
@pytest.mark.parametrize("T", [512, 256, 64])
def test_fp32_sums_are_short(lib, T):
    n = 4096
    case = H.one(n, 4096, 0, T=T, LU=4)
    w = np.repeat([1.0, 2.0], n // 2) * (1 + 2.0 ** -22) / 64
    out = H.step(lib, True, case, np.stack([np.full(n, 1.0 / 64), w]))
    want = (w / 64).sum()
    assert abs(out["h"][0, 0] - want) <= 1e-13 * want


# FP64 vectors: the Gram correction and its product with the sums carry FP64;
# the column is that of the unit vectors
# (rows that have lost 1e-6 of their orthogonality; one FP64 rounding each of
# some 30 products and sums of size 1)
@pytest.mark.parametrize("many", [False, True])
def test_fp64_correction_is_fp64(lib, many):
    r = np.random.RandomState(4)
    j = 12
    case = H.many([700, 2049], 256, 6, j) if many else H.one(1501, 512, j)
    V = np.concatenate([H.basis(r, j, k) for k in np.diff(case[1])], axis=1)
    for a, b in zip(case[1][:-1], case[1][1:]):
        V[:j + 1, a:b] += 1e-6 * r.uniform(-1, 1, (j + 1, j + 1)) @ V[:j + 1, a:b]
    X = V.astype(np.longdouble)
    _, _, E = H.reference(V, case[1], np.float64)
    out = H.step(lib, False, case, V, E)
    for s, (a, b) in enumerate(zip(case[1][:-1], case[1][1:])):
        Q, p = X[:j + 1, a:b], X[:j + 1, a:b] @ X[j + 1, a:b]
        G = Q @ Q.T - np.eye(j + 1, dtype=np.longdouble)
        nu = np.sqrt(1 + np.diag(G))
        assert np.abs(out["h"][s, :j + 1] - nu * (p - G @ p)).max() <= 30 * 1.2e-16
        assert np.abs(out["E"][s, j, :j + 1] - G[j]).max() <= 30 * 1.2e-16


# The norm by Pythagoras loses the digits that cancel; a step later the dot
# pass finds the norm itself and the rotation is brought up to date: tangent
# hn |v_{j+1}| / (h_j |v_j|), to the 2 x 128 products' rounding of the sums
# (FP32: 9 operations of 6e-8 on partial sums, averaged over n / 128 of them)
@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("many", [False, True])
def test_rotation_takes_the_norm_of_the_stored_vector(lib, many, f32):
    j, n = 11, 2000
    worst = 0.0
    for seed in range(6):
        r = np.random.RandomState(seed)
        first = H.many([n], 256, 6, j) if many else H.one(n, 512, j)
        V = H.basis(r, j, n, inside=0.012)
        _, _, E = H.reference(V, first[1], np.float32 if f32 else np.float64)
        out = H.step(lib, f32, first, V, E)
        assert out["seg"][0, 2] != 2  # no second pass
        c, s = out["h"][0, j], out["h"][0, j + 1]
        x = out["w"].astype(np.longdouble)
        norm = np.sqrt(x @ x)
        worst = max(worst, abs(float(norm) - 1))
        then = H.many([n], 256, 6, j + 1) if many else H.one(n, 512, j + 1)
        W = np.concatenate([V[:j + 1], out["w"][None], r.standard_normal((1, n)) / np.sqrt(n)])
        rot = H.step(lib, f32, then, W, state=out["state"])["rot"][0]
        want = s / c * float(norm)
        assert abs(rot[1] / rot[0] / want - 1) <= (9 * 6e-8 / np.sqrt(n / 128) if f32 else 3e-15)
    assert worst > (1e-7 if f32 else 1e-15)  # the norms were off


def _check_segments(V, seg0, out, u, redo):
    """Arnoldi relation, norm and orthogonality of every segment; a sum of up to
    31 products of rows with entries rounded by u."""
    j = len(V) - 2
    for s, (a, b) in enumerate(zip(seg0[:-1], seg0[1:])):
        Q, w, x, h = V[:j + 1, a:b], V[j + 1, a:b], out["w"][a:b], out["h"][s]
        assert np.linalg.norm(h[:j + 1] @ Q + h[j + 1] * x - w) <= 60 * u
        # one pass: the sums' rounding over hn; two: that of the second alone
        grow = 1.0 if redo[s] else np.sqrt(1 / 0.01)
        assert abs(np.linalg.norm(x) - 1) <= 20 * u * grow
        assert np.abs(Q @ x).max() <= 20 * u * grow


# the second pass: taken by a segment whose first cancels most of the vector,
# in a batch by some segments and not by others, and by blocks with more pieces
# than their list holds (three rounds of it)
@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("lens,piece,blocks,inside", [
    ([1501], 0, 3, [1e-4]),
    ([1501], 0, 1, [1e-6]),
    ([3000], 256, 5, [1e-4]),
    ([700, 301, 33, 2049, 64], 256, 6, [0.5, 1e-4, 0.3, 1e-5, 0.02]),
    ([9000, 37, 8000, 2963], 4, 2, [0.5, 0.4, 1e-4, 0.3]),
    ([9000, 37, 8000, 2963], 4, 2, [0.5, 0.4, 0.1, 0.3])],
    ids=["one", "one_block", "streamed", "some", "rounds", "rounds_single_pass"])
def test_second_pass(lib, lens, piece, blocks, inside, f32):
    r = np.random.RandomState(5)
    j = 9
    ty = np.float32 if f32 else np.float64
    case = H.many(lens, piece, blocks, j) if piece else \
        H.one(lens[0], (-(-lens[0] // blocks) + 31) // 32 * 32, j)
    V = np.concatenate([H.basis(r, j, n, inside=q) for n, q in zip(lens, inside)], axis=1)
    V = V.astype(ty).astype(np.float64)
    _, _, E = H.reference(V, case[1], ty)
    out = H.step(lib, f32, case, V, E)
    redo = [q < 0.01 for q in inside]
    assert (out["seg"][:, 0] == 0).all() and out["ctl"][0] == j + 1 and out["ctl"][2] == 0
    if piece:
        assert out["seg"][:, 2].tolist() == [2 if q else 1 for q in redo]
        assert out["ctl"][3] == case[0].blocks * (4 if any(redo) else 2)
    else:
        assert out["ctl"][3] == (2 * case[0].blocks if case[0].blocks > 1 else 0)
    _check_segments(V, case[1], out, 6e-8 if f32 else 1.2e-16, redo)
