"""Import of full FP64 populations into the deviation forms at the ends of its fixed-point range (around 1/2, 1 and 2, far above,
tiny, zero, not finite): what is stored and the fields, against FP64 numpy."""
import numpy as np
import pytest

from paper_2002_04353_gb300 import alelb
from test_batch import _cases, _solvers

pytestmark = pytest.mark.gpu


def _planes(N, scale, seed):
    rng = np.random.default_rng(seed)
    f, g = (scale * (0.05 + 0.1 * rng.random((9, N))) for _ in range(2))
    at = rng.permutation(N)[:64].reshape(8, 8)
    for row, v in zip(at, (0.0, 1e-30, 2.0 ** -60, np.nextafter(2.0, 0), 2.0, 3.7e3, 1e-12, 0.99999999)):
        f[rng.integers(0, 9), row] = v
        g[rng.integers(0, 9), row] = v
    return f, g


@pytest.mark.parametrize("scale", [1.0, 1e-6, 6.5, 1e4])
@pytest.mark.parametrize("dev", [False, True])
def test_stored_deviations_and_fields(scale, dev):
    import torch
    s = _solvers(_cases()[1:2], alelb.PREC_FP32_DEV)[0]
    z = np.zeros((9, s.nn), dtype=np.float32)
    s.set_pops_stored(z, z)
    cf, cg = s.get_pops()  # the reference populations
    f, g = _planes(s.nn, scale, 3)
    if dev:
        s.set_pops_dev(torch.from_numpy(f).cuda(), torch.from_numpy(g).cuda(), t=0.0)
    else:
        s.set_pops(f, g, t=0.0)
    df, dg = s.get_pops_stored()
    for d, v, c in ((df, f, cf), (dg, g, cg)):
        # one FP32 rounding, one of the value to 2^-58 and one of its difference in FP64
        assert np.all(np.abs(d.astype(np.float64) - (v - c)) <= 2.0 ** -24 * np.abs(v - c) + 2.0 ** -58 + 2.0 ** -52 * np.abs(v))
    m = s.moments()
    rho = f.sum(0)
    cx, cy = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1.0]), np.array([0, 0, 1, 0, -1, 1, 1, -1, -1.0])
    ux, uy = cx @ f / rho, cy @ f / rho
    T = (g.sum(0) / (2 * rho) - 0.5 * (ux * ux + uy * uy)) * 0.4
    # FP32 roundings; the sums' FP64 and 2^-58 ones against what cancels in u and T
    a = 2.0 ** -54 * 9 / rho + 2.0 ** -50
    for k, v, e in (("rho", rho, 0 * rho), ("ux", ux, a), ("uy", uy, a),
                    ("T", T, a * (np.abs(ux) + np.abs(uy) + g.sum(0) / rho))):
        assert np.all(np.abs(m[k] - v) <= 2.0 ** -24 * np.abs(v) * 1.0001 + 4 * e + 1e-12 * np.abs(v)), k


def test_what_is_not_finite_stays_so():
    import torch
    s = _solvers(_cases()[1:2], alelb.PREC_FP32_DEV)[0]
    f, g = _planes(s.nn, 1.0, 5)
    f[3, 11], g[4, 12], f[0, 13] = np.inf, np.nan, -np.inf
    s.set_pops_dev(torch.from_numpy(f).cuda(), torch.from_numpy(g).cuda(), t=0.0)
    df, dg = s.get_pops_stored()
    assert df[3, 11] == np.inf and np.isnan(dg[4, 12]) and df[0, 13] == -np.inf
    assert np.isfinite(df).sum() == df.size - 2 and np.isfinite(dg).sum() == dg.size - 1
    of, og = torch.empty((9, s.nn), dtype=torch.float64, device="cuda"), torch.empty((9, s.nn), dtype=torch.float64, device="cuda")
    hf, hg = np.empty((9, s.nn)), np.empty((9, s.nn))
    s.get_pops(hf, hg)
    try:
        s.get_pops_dev(of, og)
    except Exception:
        pass
    assert np.array_equal(of.cpu().numpy(), hf, equal_nan=True) and np.array_equal(og.cpu().numpy(), hg, equal_nan=True)
