"""FP64 batches with the transformed velocities as printed (LITERAL_VG): batches in which every case runs them take the plain pass,
mixed ones the two passes; both give what each case gives alone, and the same count of located populations."""
import dataclasses

import numpy as np
import pytest

import oracle as O
from paper_2002_04353_gb300 import alelb
from test_batch import TOL64, _cases, _rel, _solvers

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("which", [(0, 1, 2, 3), (0, 2), ()])
@pytest.mark.parametrize("tune", [False, True])
def test_batch_equals_the_oracle(which, tune):
    cases = [(m, mo, dataclasses.replace(fl, flags=fl.flags | (O.FLAG_LITERAL_VG if k in which else 0)))
             for k, (m, mo, fl) in enumerate(_cases())]
    ss, alone = _solvers(cases, alelb.PREC_FP64), _solvers(cases, alelb.PREC_FP64)
    b = alelb.Batch(ss)
    if tune:
        b.tune(1)  # one step
    b.step(5 - tune)
    b.sync()
    for k, ((mesh, motion, flow), s, a) in enumerate(zip(cases, ss, alone)):
        o = O.Oracle(mesh, motion, flow)
        o.step(5)
        a.lb_step(5)
        st = o.state()
        f, g = s.get_pops()
        assert _rel(f, st["f"]) < TOL64 and _rel(g, st["g"]) < TOL64, f"case {k}"
        assert s.info()["walks"] == a.info()["walks"], f"case {k}"
        assert np.all(np.isfinite(f))
