"""Import of populations into the FP32 deviation form at free-stream densities and temperatures far from one, and of populations that
lie close to the reference: a stored deviation is the exact difference rounded once, and the fields are FP32 roundings, at every
scale.  (16-bit forms store the same difference, rounded further.)"""
import numpy as np
import pytest

from paper_2002_04353_gb300 import alelb, inputs as I

pytestmark = pytest.mark.gpu


def _solver(rho, T):
    mesh = I.periodic_box(6, 12.0, 0.2, seed=3)
    flow = I.Flow(mu=0.02 * rho, rho_inf=rho, T_inf=T, u_inf=(0.05, 0.02))
    s = alelb.Solver(alelb.Mesh(mesh, I.Motion.make(I.MOTION_NONE)), flow, alelb.PREC_FP32_DEV)
    z = np.zeros((9, s.nn), dtype=np.float32)
    s.set_pops_stored(z, z)
    return s, s.get_pops()  # the reference populations


@pytest.mark.parametrize("amp", [0.3, 1e-3, 1e-9])
@pytest.mark.parametrize("how", ["host", "device", "stored"])
@pytest.mark.parametrize("rho,T", [(1e-22, 0.3), (1e-18, 0.3), (1e-15, 0.3), (1e-12, 0.2), (1e-9, 0.3), (1e-6, 0.3), (2.0 ** -19, 0.3), (0.02, 0.05),
                                   (1.0, 0.05), (1.0, 0.3), (7.0, 0.2), (1e5, 0.3), (1e25, 0.3)])
def test_import_is_relative_to_the_density(rho, T, how, amp):
    import torch
    s, (cf, cg) = _solver(rho, T)
    rng = np.random.default_rng(7)
    f, g = (c * (1.0 + amp * rng.uniform(-1, 1, c.shape)) for c in (cf, cg))
    if how == "stored":
        df, dg = ((v - c).astype(np.float32) for v, c in ((f, cf), (g, cg)))
        s.set_pops_stored(df, dg)
        f, g = df.astype(np.float64) + cf, dg.astype(np.float64) + cg
    elif how == "device":
        s.set_pops_dev(torch.from_numpy(f).cuda(), torch.from_numpy(g).cuda(), t=0.0)
    else:
        s.set_pops(f, g, t=0.0)
    got = s.get_pops_stored()
    if how == "stored":
        assert np.array_equal(got[0], df) and np.array_equal(got[1], dg)
    for d, v, c in zip(got, (f, g), (cf, cg)) if how != "stored" else ():
        # one rounding of the difference (exact in FP64 at these amplitudes) and 2^-30 of it on the way there
        assert np.all(np.abs(d.astype(np.float64) - (v - c)) <= (2.0 ** -24 + 2.0 ** -30) * np.abs(v - c)), "deviations"
    m = s.moments()
    cx, cy = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1.0]), np.array([0, 0, 1, 0, -1, 1, 1, -1, -1.0])
    r = f.sum(0)
    ux, uy = cx @ f / r, cy @ f / r
    E = g.sum(0) / r
    Tr = 0.4 * 0.5 * (E - ux * ux - uy * uy)
    # one FP32 rounding; the FP64 sums before it against what cancels in u and T
    a = 16 * 2.0 ** -52
    for k, v, e in (("rho", r, a * r), ("ux", ux, a), ("uy", uy, a), ("T", Tr, a * E)):
        assert np.all(np.abs(m[k] - v) <= 2.0 ** -24 * np.abs(v) + e), k
