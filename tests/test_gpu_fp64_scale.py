"""The FP64 step is linear in the density: a run at a power of two of it, down to where the populations are barely normal numbers and up
to where they nearly overflow, gives that multiple of the same run at one."""
import numpy as np
import pytest

from paper_2002_04353_gb300 import alelb, inputs as I

pytestmark = pytest.mark.gpu


def _run(k, elem):
    r = 2.0 ** k
    mesh = I.periodic_box(6, 12.0, 0.2, seed=3, elem=elem)
    flow = I.Flow(mu=0.02 * r, rho_inf=r, T_inf=0.3, u_inf=(0.05, 0.02))
    s = alelb.Solver(alelb.Mesh(mesh, I.Motion.make(I.MOTION_SINE, 0.6, 12.0, 40.0, 0.0)), flow, alelb.PREC_FP64)
    f, g = s.get_pops()
    rng = np.random.default_rng(2)
    d = 1.0 + 1e-2 * rng.uniform(-1, 1, (2, *f.shape))
    s.set_pops(f * d[0], g * d[1], t=0.0)
    s.lb_step(4)
    m = s.moments()
    return [v * 2.0 ** -(k // 2) * 2.0 ** -(k - k // 2) for v in (*s.get_pops(), m["rho"])] + [m["ux"], m["uy"], m["T"]]


@pytest.mark.parametrize("elem", ["p2", "q2"])
@pytest.mark.parametrize("k", [-1012, -1006, -895, -300, 300, 900, 1012])
def test_linear_in_the_density(k, elem):
    # a population of 2^-1012 / 50 keeps 48 bits at least where terms a hundred times smaller are below the normal range
    for a, b in zip(_run(k, elem), _run(0, elem)):
        assert np.all(np.isfinite(a)) and np.abs(a - b).max() <= 1e-12 * np.abs(b).max()
