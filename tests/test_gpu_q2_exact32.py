"""FP32 quadrilaterals on the exact path: the local coordinates come from the FP64 departure point and corners, also across a period
that FP32 does not hold.  One propagation (no collision) from a cold cache, against the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_2002_04353_gb300 import alelb, inputs as I
from test_gpu_q2 import _pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,L", [(16, 32.0), (200, 400.0 + 2.0 ** -16)])
def test_propagation_from_a_cold_cache(n, L):
    mesh = I.periodic_box(n, L, 0.2, seed=1, elem="q2")
    motion = I.Motion.make(I.MOTION_SINE, 0.05 * L, L, 100.0, 0.0)
    flow = I.Flow(mu=0.02, T_inf=0.3, u_inf=(0.05, 0.02), flags=O.FLAG_COLLIDE_OFF)
    o, s = _pair(mesh, motion, flow, alelb.PREC_FP32_DEV)
    z = np.zeros((9, s.nn), dtype=np.float32)
    s.set_pops_stored(z, z)
    cf, cg = s.get_pops()
    rng = np.random.default_rng(2)
    amp = 1e-2
    df, dg = (amp * rng.uniform(-1, 1, (9, s.nn)).astype(np.float32) for _ in range(2))
    s.set_pops_stored(df, dg, t=3.0)
    m = s.moments()
    o.set_state(df + cf, dg + cg, m["rho"], m["ux"], m["uy"], m["T"], 3.0)
    o.step(1)
    s.lb_step(1)
    st = o.state()
    # Local coordinates: corners relative to the point, rounded once (2^-24 of up to three half cells), the residual's four products
    # and sums and the last FP32 step: some 16 roundings of 2^-24 each times the inverse Jacobian (2 half cells): 2^-19.  The nine
    # shape functions' derivatives sum to at most 9 in modulus; then their own 27 FP32 roundings.
    tol = amp * (9 * 2.0 ** -19 + 27 * 2.0 ** -24)
    for got, ref in zip(s.get_pops(), (st["f"], st["g"])):
        assert np.abs(got - ref).max() <= tol
