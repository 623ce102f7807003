"""Binding of tests/cuda/orth_harness.cu: the orthogonalisation kernels alone."""
import ctypes
import os
import subprocess

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))


class Case(ctypes.Structure):
    _fields_ = [(k, ctypes.c_int32) for k in
                ("many", "nseg", "j", "T", "LU", "blocks", "piece", "absent")] + \
               [("n", ctypes.c_int64), ("share", ctypes.c_int64), ("wait_ns", ctypes.c_uint64)]


def compile_harness(source):
    """The harness' shared library, compiled with the library's own flags."""
    from paper_2605_25403_gb300 import build
    out_dir = os.path.join(HERE, "_build")
    os.makedirs(out_dir, exist_ok=True)
    src = os.path.join(HERE, "cuda", source)
    lib = os.path.join(out_dir, source.replace(".cu", ".so"))
    deps = [src] + [os.path.join(build.CSRC, f) for f in os.listdir(build.CSRC)]
    if build._stale(lib, deps):
        tmp = f"{lib}.{os.getpid()}.tmp"
        subprocess.run([build._nvcc()] + build._flags() + ["-I", build.CSRC, "-shared", src, "-o",
                                                           tmp], check=True)
        os.replace(tmp, lib)
    return ctypes.CDLL(lib)


def _ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def one(n, share, j, T=512, LU=1, wait_ns=10**9, absent=0):
    """A single segment, `share` entries per block (a multiple of 32)."""
    return Case(many=0, nseg=1, j=j, T=T, LU=LU, blocks=-(-n // share), piece=0, absent=absent,
                n=n, share=share, wait_ns=wait_ns), np.array([0, n], dtype=np.int64)


def many(lens, piece, blocks, j, T=512, wait_ns=10**9, absent=0):
    """Segments of the given lengths in pieces of at most `piece` entries."""
    seg0 = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    return Case(many=1, nseg=len(lens), j=j, T=T, LU=1, blocks=blocks, piece=piece, absent=absent,
                n=int(seg0[-1]), share=0, wait_ns=wait_ns), seg0


def step(lib, f32, case, V, E=None, state=None):
    """One step on the rows V (j + 2 of them): the new vector, per segment the
    Hessenberg column, the Gram correction, (bad, done, act, k), the rotation
    before this step's and the segments' records (a later step's `state`, which
    then holds E); and (j, all_done, nredo, barrier arrivals)."""
    c, seg0 = case
    V = np.ascontiguousarray(V, dtype=np.float64)
    assert V.shape == (c.j + 2, c.n)
    E = np.zeros((c.nseg, 32, 32)) if E is None else np.array(E, dtype=np.float64)
    w, h = np.empty(c.n), np.zeros((c.nseg, 33))
    seg, ctl = np.zeros((c.nseg, 4), dtype=np.int32), np.zeros(4, dtype=np.int32)
    resume = state is not None
    state = state.copy() if resume else np.zeros(c.nseg * lib.orth_state_size(), dtype=np.uint8)
    rot = np.zeros((c.nseg, 2))
    rc = lib.orth_step(int(f32), ctypes.byref(c), _ptr(seg0), _ptr(V), _ptr(E), _ptr(w), _ptr(h),
                       _ptr(seg), _ptr(ctl), _ptr(state), int(resume), _ptr(rot))
    assert rc == 0, rc
    return dict(w=w, h=h[:, :c.j + 2], E=E, seg=seg, ctl=ctl, rot=rot, state=state)


def loop_passes(lib, f32, case, max_pass):
    c, seg0 = case
    n = ctypes.c_int(0)
    rc = lib.orth_loop(int(f32), ctypes.byref(c), _ptr(seg0), max_pass, ctypes.byref(n))
    assert rc == 0, rc
    return n.value


def basis(r, j, n, wnorm=1.0, inside=None):
    """j + 1 orthonormal rows and a row w of the given norm; `inside`: the
    share of w^2 outside the span of the others."""
    q = np.linalg.qr(r.standard_normal((n, j + 2)))[0].T
    w = r.standard_normal(j + 1) @ q[:j + 1]
    if inside is None:
        inside = 0.5
    w = w / np.linalg.norm(w) * np.sqrt(1 - inside) + q[j + 1] * np.sqrt(inside)
    return np.concatenate([q[:j + 1], wnorm * w[None]])


def reference(V, seg0, dtype):
    """The step on rows of the given type in extended precision: per segment
    the projection of w onto the others' span, the norm of what is left and
    that vector normalised; and the Gram correction the earlier steps left
    (rows and columns below j)."""
    X = V.astype(dtype).astype(np.longdouble)
    j = len(V) - 2
    new, h, E = np.empty_like(X[0]), [], np.zeros((len(seg0) - 1, 32, 32))
    for s, (a, b) in enumerate(zip(seg0[:-1], seg0[1:])):
        Q, w = X[:j + 1, a:b], X[j + 1, a:b]
        G = Q @ Q.T - np.eye(j + 1, dtype=np.longdouble)
        E[s, :j, :j] = G[:j, :j]
        c = p = Q @ w
        for _ in range(12):
            c = p - G @ c  # (I + G) c = p, G of rounding size
        r = w - c @ Q
        nrm = np.sqrt(r @ r)
        new[a:b] = r / nrm
        h.append(np.append(c, nrm))
    return new, np.array(h), E
