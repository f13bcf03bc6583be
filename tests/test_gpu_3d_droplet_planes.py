"""The 3D droplet kernel with one, two, four and eight planes per CTA (it takes as many as
leave every SM two CTAs) against the profile: boxes whose planes are not a multiple of
any, a droplet cut by the periodic seams, one that overlaps another. phi is max(field,
1/2 + 1/2 tanh(2 (R - r) / W)) at fluid nodes, the profile evaluated in the precision
of the solve from distances in 64 bits: to 1e-13 in FP64 (sums of a few roundings), to
1e-6 in FP32 (2 ulp in each of two tanh, 1e-7 each, and seven roundings of 6e-8).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-13), ("fp32", 1e-6)])
@pytest.mark.parametrize("nx,ny,nz,R", [(24, 24, 20, 5.0), (33, 47, 25, 9.0), (40, 96, 37, 14.0), (96, 64, 51, 22.0),
                                        (130, 70, 45, 40.0), (200, 160, 43, 60.0)])
def test_droplet_equals_profile(nx, ny, nz, R, precision, tol):
    from paper_2312_00369_gb300 import workloads as wl
    from paper_2312_00369_gb300.pflbm import Solver3D
    solid, zw = wl.box3d(nx, ny, nz)
    W = 2.0
    drops = [(nx / 3.0, 0.8, zw, R), (nx - 0.7, ny / 2.0, 0.6 * nz, 0.7 * R)]
    s = Solver3D(solid, precision=precision, W=W)
    for d in drops:
        s.init_droplet(*d)
    phi = s.get()[0]
    s.close()
    z, y, x = np.mgrid[:nz, :ny, :nx].astype(np.float64)
    want = np.zeros((nz, ny, nx))
    c = np.float64 if precision == "fp64" else np.float32
    for x0, y0, z0, r0 in drops:
        dx, dy = np.abs(x - x0), np.abs(y - y0)
        dx, dy = np.minimum(dx, nx - dx), np.minimum(dy, ny - dy)
        r2 = dx * dx + dy * dy + (z - z0) ** 2
        want = np.maximum(want, c(0.5) + c(0.5) * np.tanh(c(2) * (c(r0) - np.sqrt(r2.astype(c))) / c(W)))
    err = np.max(np.abs(phi - want)[solid == 0])
    assert err < tol, err
