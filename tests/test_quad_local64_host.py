"""Local coordinates of the FP64 form on quadrilaterals, on the host: cells of every shape, place and direction, thin ones oblique to
the axes and cells far from the origin among them, against Newton's method in extended precision."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

import hostcheck as H
from paper_2002_04353_gb300 import build, inputs as I

SRC = os.path.join(H.HERE, "hostcheck_local64.cu")
OUT = os.path.join(H.HERE, "_build", "libalelb_hostcheck_local64.so")


@pytest.fixture(scope="module")
def lib():
    if not os.path.exists(OUT) or any(os.path.getmtime(d) > os.path.getmtime(OUT) for d in build.DEPS + [SRC]):
        os.makedirs(os.path.dirname(OUT), exist_ok=True)
        tmp = OUT + f".{os.getpid()}.tmp"
        subprocess.run(["nvcc", "-O2", "-std=c++17", "-Xcompiler", "-fPIC,-ffp-contract=off", "-shared", "-I",
                        os.path.join(build.ROOT, "include"), "-I", build.CSRC, "-o", tmp, SRC], check=True)
        os.replace(tmp, OUT)
    L = C.CDLL(OUT)
    L.alelb_hostcheck_local64.argtypes = [C.c_int, C.c_void_p, C.c_void_p]
    return L


def _newton(w, p, iters=14):
    """xi, eta of points p in cells w, and the inverse Jacobians, in extended precision (an error far below FP64's)."""
    q = np.longdouble
    c = w.astype(q) - p.astype(q)[:, None]
    a, b = np.zeros(len(w), q), np.zeros(len(w), q)
    for _ in range(iters):
        n = np.stack([(1 - a) * (1 - b), (1 + a) * (1 - b), (1 + a) * (1 + b), (1 - a) * (1 + b)], 1)[:, :, None] / 4
        da = np.stack([-(1 - b), 1 - b, 1 + b, -(1 + b)], 1)[:, :, None] / 4
        db = np.stack([-(1 - a), -(1 + a), 1 + a, 1 - a], 1)[:, :, None] / 4
        r, A, B = (n * c).sum(1), (da * c).sum(1), (db * c).sum(1)
        det = A[:, 0] * B[:, 1] - B[:, 0] * A[:, 1]
        inv = np.stack([B[:, 1], -B[:, 0], -A[:, 1], A[:, 0]], 1) / det[:, None]
        a, b = a - (inv[:, 0] * r[:, 0] + inv[:, 1] * r[:, 1]), b - (inv[:, 2] * r[:, 0] + inv[:, 3] * r[:, 1])
    return a, b, inv


def _cells(kind):
    rng = np.random.default_rng(4)
    if kind in ("box", "omesh", "channel"):
        m = {"box": lambda: I.periodic_box(24, 48.0, 0.2, seed=1, elem="q2"), "channel": lambda: I.wall_channel(elem="q2"),
             "omesh": lambda: I.naca_omesh(96, 36, chord=1000.0, R=20000.0, first=1.0, elem="q2")}[kind]()
        w = m.X[m.conn[:, :4]].copy()
        for d, L in enumerate(m.period):
            if L > 0:
                w[:, :, d] -= np.round((w[:, :, d] - w[:, :1, d]) / L) * L
        return w
    aspect, far = kind
    t = rng.uniform(0, 2 * np.pi, 2000)
    w = np.array([[0, 0], [1, 0], [1, 1], [0, 1]])[None] + rng.uniform(-0.12, 0.12, (len(t), 4, 2))
    w[:, :, 0] *= aspect
    R = np.stack([np.stack([np.cos(t), -np.sin(t)], 1), np.stack([np.sin(t), np.cos(t)], 1)], 1)
    return np.einsum("kij,kcj->kci", R, w) + far * rng.uniform(-1, 1, (len(t), 1, 2))


@pytest.mark.parametrize("kind", ["box", "omesh", "channel", (1, 1.0), (1, 1e3), (1, 3e6), (30, 1e3), (1e3, 1e3), (1e4, 1e4)], ids=str)
def test_local_coordinates(lib, kind):
    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("no extended precision")
    w = _cells(kind)
    rng = np.random.default_rng(5)
    w = w[rng.integers(0, len(w), 20000)]
    a, b = rng.uniform(-1, 1, (2, len(w)))
    n = np.stack([(1 - a) * (1 - b), (1 + a) * (1 - b), (1 + a) * (1 + b), (1 - a) * (1 + b)], 1) / 4
    p = (n[:, :, None] * w).sum(1)
    buf = np.ascontiguousarray(np.concatenate([w.reshape(-1, 8), p], 1))
    out = np.empty((len(w), 2))
    assert lib.alelb_hostcheck_local64(len(w), buf.ctypes.data, out.ctypes.data) == 0
    x, y, inv = _newton(w, p)
    # The residual: the differences from the corner and the centre, three fused operations on terms of at most the cell's extent
    # in each direction, the coefficients' own rounding: some eight roundings of 2^-53 of the extent; the inverse Jacobian carries it
    # into the coordinates (rounded themselves: 2^-52), and FP32's part of a further correction (at most twice as much).
    ext = np.abs(w - w[:, :1]).max(1) + np.abs(p - w[:, 0])
    tol = 2.0 ** -52 + 16 * 2.0 ** -53 * (np.abs(inv.reshape(-1, 2, 2)) * ext[:, None, :]).sum(2)
    err = np.abs(np.stack([x, y], 1) - out)
    assert np.all(err <= tol), float((err / tol).max())


@pytest.mark.parametrize("size", [1e-25, 1e-19, 1e10, 1e18, 1e20, 1e45])
def test_cells_beyond_fp32(lib, size):
    """Where FP32 does not hold a cell's edges or their products the point is left to Newton's method in FP64, or is right."""
    w = _cells((1, 1.0))[:500] * size
    p = w.mean(1) + 0.3 * (w[:, 1] - w[:, 0])
    buf = np.ascontiguousarray(np.concatenate([w.reshape(-1, 8), p], 1))
    out = np.empty((1, 2))
    q = np.longdouble
    x, y, _ = _newton((w / size).astype(q), (p / size).astype(q))
    for k in range(len(w)):
        if lib.alelb_hostcheck_local64(1, buf[k].ctypes.data, out.ctypes.data) == 0:
            assert abs(out[0, 0] - x[k]) < 1e-12 and abs(out[0, 1] - y[k]) < 1e-12
