"""The two-pass propagation of the FP64 form: a population's value does not depend on which pass settles it, so a solver with a
warm element cache and one with an empty cache give the same bits; and the step agrees with the oracle on both sides of the
node counts at which the launch changes."""
import dataclasses

import numpy as np
import pytest

from paper_2002_04353_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _case(kind, n, elem):
    if kind == "box":
        return I.uniform_flow_case(n=n, L=2.0 * n, period_steps=40.0, elem=elem)
    ni, nj = I.omesh_size_for(n)
    if kind == "plunge":
        c = I.plunge_case(ni=ni, nj=nj, elem=elem)
    else:
        c = I.pitch_case(ni=ni, nj=nj, Ma=0.3, blended=kind == "blended", plunge_frac=0.0 if kind == "blended" else 0.05,
                         elem=elem)
    return dataclasses.replace(c, flow=dataclasses.replace(c.flow, flags=256))


def _start(case, seed):
    from paper_2002_04353_gb300 import alelb
    s = alelb.Solver(alelb.Mesh(case.mesh, case.motion), case.flow, alelb.PREC_FP64)
    f, g = s.get_pops()
    rng = np.random.default_rng(seed)
    f = f * (1.0 + 1e-3 * rng.uniform(-1, 1, f.shape))
    g = g * (1.0 + 1e-3 * rng.uniform(-1, 1, g.shape))
    s.set_pops(f, g, t=17.0)
    return s


@pytest.mark.parametrize("kind,n", [("box", 7), ("box", 46), ("box", 130), ("plunge", 9000), ("pitch", 6000), ("blended", 21000),
                                    ("blended", 66000)])
@pytest.mark.parametrize("elem", ["p2", "q2"])
def test_values_do_not_depend_on_the_cache(kind, n, elem):
    from paper_2002_04353_gb300 import alelb
    case = _case(kind, n, elem)
    warm = _start(case, 1)
    warm.lb_step(3)
    f, g = warm.get_pops()
    m = warm.moments()
    cold = alelb.Solver(alelb.Mesh(case.mesh, case.motion), case.flow, alelb.PREC_FP64)
    cold.set_pops(f, g, m["rho"], m["ux"], m["uy"], m["T"], t=warm.time()[0])
    w0 = warm.info()["walks"]
    warm.lb_step(2)
    cold.lb_step(2)
    for a, b in zip(warm.get_pops(), cold.get_pops()):
        np.testing.assert_array_equal(a, b)
    assert warm.info()["walks"] - w0 == cold.info()["walks"]


@pytest.mark.parametrize("kind,n", [("box", 45), ("box", 46), ("box", 129), ("pitch", 8000)])
@pytest.mark.parametrize("elem", ["p2", "q2"])
def test_against_the_oracle(kind, n, elem):
    import oracle as O
    case = _case(kind, n, elem)
    s = _start(case, 2)
    f, g = s.get_pops()
    m = s.moments()
    o = O.Oracle(case.mesh, case.motion, case.flow)
    o.set_state(f, g, m["rho"], m["ux"], m["uy"], m["T"], s.time()[0])
    s.lb_step(2)
    o.step(2)
    st = o.state()
    for a, b in zip(s.get_pops(), (st["f"], st["g"])):
        assert np.abs(a - b).max() <= 1e-12 * np.abs(b).max()
