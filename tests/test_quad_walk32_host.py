"""The quadrilaterals' exact path on the host: the walk on certified FP32 signs names the element the exact FP64 walk names, for every
map and across periods, at ties (lattice), walls and the far field; and the exterior cone never certifies a population that is
not missing."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

import hostcheck as H
from paper_2002_04353_gb300 import build, inputs as I
from test_walk_host import CASES

SRC = os.path.join(H.HERE, "hostcheck_walk32.cu")
OUT = os.path.join(H.HERE, "_build", "libalelb_hostcheck_walk32.so")


@pytest.fixture(scope="module")
def lib():
    deps = build.DEPS + [SRC, H.SRC]
    if not os.path.exists(OUT) or any(os.path.getmtime(d) > os.path.getmtime(OUT) for d in deps):
        os.makedirs(os.path.dirname(OUT), exist_ok=True)
        tmp = OUT + f".{os.getpid()}.tmp"
        subprocess.run(["nvcc", "-O2", "-std=c++17", "-Xcompiler", "-fPIC,-ffp-contract=off", "-shared", "-I",
                        os.path.join(build.ROOT, "include"), "-I", build.CSRC, "-I", H.HERE, "-o", tmp, SRC], check=True)
        os.replace(tmp, OUT)
    L = C.CDLL(OUT)
    L.alelb_hostcheck_walk32_q2.argtypes = [C.c_void_p, C.c_double, C.c_void_p]
    return L


MORE = {
    "q2_static_omesh": (lambda: I.naca_omesh(64, 20, chord=200.0, R=4000.0, first=1.0, elem="q2"),
                        lambda: I.Motion.make(I.MOTION_NONE), [1]),
    "q2_tiny_box": (lambda: I.periodic_box(4, 8.0, 0.2, seed=1, elem="q2"),
                    lambda: I.Motion.make(I.MOTION_SINE, 0.3, 8.0, 40.0, 0.0), [1, 9]),
    "q2_pitch": (lambda: I.naca_omesh(64, 20, chord=200.0, R=4000.0, first=1.0, elem="q2"),
                 lambda: I.Motion.make(I.MOTION_PITCH, 0.05, 0.05, 0.003, 50.0, 0.0), [3, 400]),
}


@pytest.mark.parametrize("name", sorted([k for k in CASES if k.startswith("q2")] + list(MORE)))
def test_fp32_walk_names_the_exact_walks_element(lib, name):
    mk_mesh, mk_mot, times = MORE[name] if name in MORE else CASES[name]
    mesh, mot = mk_mesh(), mk_mot()
    d, keep = H._desc(mesh, mot)
    for t in times:
        out = np.zeros(4, dtype=np.int64)
        bad = lib.alelb_hostcheck_walk32_q2(C.byref(d), float(t), out.ctypes.data)
        assert bad == 0, f"{name} t={t}: {bad} locations differ"
        assert out[0] > 7 * mesh.n_nodes and out[3] == 0
        if "omesh" in name or "plunge" in name or "pitch" in name:
            assert out[2] > 0  # the cone is used
