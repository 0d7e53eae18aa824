"""Export to device arrays agrees bit for bit with the export to the host, also for deviations below FP32's normal range where the
reference population is zero (at T = 1 the lattice's axis populations vanish) and cannot absorb them."""
import numpy as np
import pytest

from paper_2002_04353_gb300 import alelb, inputs as I

pytestmark = pytest.mark.gpu


def test_small_deviations_reach_the_device_arrays():
    import torch
    mesh = I.periodic_box(4, 8.0, 0.2, seed=3)
    flow = I.Flow(mu=0.02, rho_inf=1.0, T_inf=1.0)
    s = alelb.Solver(alelb.Mesh(mesh, I.Motion.make(I.MOTION_NONE)), flow, alelb.PREC_FP32_DEV)
    d = np.zeros((9, s.nn), dtype=np.float32)
    d[:, 0::4], d[:, 1::4], d[:, 2::4] = 1e-40, -3e-42, 2e-38
    s.set_pops_stored(d, d)
    hf, hg = s.get_pops()
    f, g = (torch.empty((9, s.nn), dtype=torch.float64, device="cuda") for _ in range(2))
    s.get_pops_dev(f, g)
    assert np.count_nonzero((np.abs(hf) < 1e-37) & (hf != 0)) > 0  # some are seen
    assert np.array_equal(f.cpu().numpy(), hf) and np.array_equal(g.cpu().numpy(), hg)
