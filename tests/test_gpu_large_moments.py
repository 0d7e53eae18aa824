"""Meshes large enough for the propagation that takes the moments along (FP32, a turning or deforming map), a ragged last block, walls
whose nodes wait for the exact path: against the batched step with the moments in a kernel of their own."""
import dataclasses

import numpy as np
import pytest

from paper_2002_04353_gb300 import alelb, inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("blended", [True, False])
def test_moments_along_with_the_propagation(blended):
    c = I.pitch_case(ni=450, nj=168, Ma=0.3, blended=blended)
    assert c.mesh.n_nodes >= 300000 and c.mesh.n_nodes % 128
    flow = dataclasses.replace(c.flow, flags=alelb.FLAG_OFFWALL_VG)
    m = alelb.Mesh(c.mesh, c.motion)
    one, other = alelb.Solver(m, flow, alelb.PREC_FP32_DEV), alelb.Solver(m, flow, alelb.PREC_FP32_DEV)
    b = alelb.Batch([other])
    b.set_choice([128, 128, 128, 256, 256, 128, 64, 9])
    for _ in range(2):  # a second call: the lists were emptied
        one.lb_step(2)
        b.step(2)
    b.sync()
    # the two forms fuse their multiply-adds differently: FP32 roundings of four steps
    for x, y in zip(one.get_pops(), other.get_pops()):
        assert np.abs(x - y).max() <= 1e-5 * np.abs(y).max()
    mx, my = one.moments(), other.moments()
    for k in mx:
        assert np.abs(mx[k] - my[k]).max() <= 1e-5 * max(np.abs(my[k]).max(), 0.1), k
    assert one.info()["walks"] == other.info()["walks"]
