"""A droplet added to a given field (init_phi, then init_droplet) combines with it
by maximum within |R| + 10 W of its centre and leaves every other node alone,
also those in the corners of its bounding box: a field that is negative there
stays negative. Beyond the reach and its stencils the state is that of the
field alone, bit for bit; at the nodes themselves phi of the FP64 and FP32 states
is max(field, profile) to 1e-6 (the FP32 tanh; a 16-bit state's phi also holds the
rounding of its neighbours' g_i). A replacing
call whose centre and radius overflow FP32 clears the field (the profile is
undefined there in FP32, and a comparison with NaN never wins).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision", ["fp64", "fp32", "bf16", "fp16"])
@pytest.mark.parametrize("nx,ny,x0,R", [(128, 96, 64.0, 10.0), (131, 97, 3.0, 12.0), (80, 70, 40.0, -2.0)])
def test_negative_field_beyond_a_droplet_is_kept(precision, nx, ny, x0, R):
    from paper_2312_00369_gb300.pflbm import Solver
    W, y0 = 2.0, ny / 2.0
    solid = np.zeros((ny, nx), np.uint8)
    solid[:2] = solid[-2:] = 1
    y, x = np.mgrid[:ny, :nx].astype(np.float64)
    field = -0.05 - 0.02 * np.cos(2 * np.pi * x / nx)
    got = []
    for drop in (False, True):
        s = Solver(solid, precision=precision, W=W)
        s.init_phi(field)
        if drop:
            s.init_droplet(x0, y0, R)
        got.append(s.get())
        s.close()
    dx = np.abs(x - x0)
    dx = np.minimum(dx, nx - dx)
    r = np.sqrt(dx * dx + (y - y0) ** 2)
    fluid = solid == 0
    # three stencils reach out from a changed node: mu, phi (a 16-bit state's g_0
    # holds the rounding of its neighbours' mu) and the gradient in u
    far = fluid & (r > abs(R) + 10 * W + 3 * np.sqrt(2.0))
    box = (dx <= abs(R) + 10 * W) & (np.abs(y - y0) <= abs(R) + 10 * W)
    assert (far & box).sum() > 20              # corners of the box
    for a, b in zip(*got):
        assert np.array_equal(a[far], b[far])
    if precision in ("bf16", "fp16"):
        return
    profile = 0.5 + 0.5 * np.tanh(2 * (R - r) / W)
    want = np.where(r > abs(R) + 10 * W, field, np.maximum(field, profile))
    edge = np.abs(r - abs(R) - 10 * W) < 1e-6  # within rounding of the reach
    assert np.max(np.abs(got[1][0] - want)[fluid & ~edge]) < 1e-6


def test_replacing_droplet_past_fp32_clears_the_field():
    from paper_2312_00369_gb300.pflbm import Solver
    solid = np.zeros((50, 100), np.uint8)
    solid[:2] = solid[-2:] = 1
    s = Solver(solid, precision="fp32")
    s.init_droplet(50.0, 1e40, 1e40)
    assert np.array_equal(s.get()[0], np.zeros((50, 100)))
    s.close()
