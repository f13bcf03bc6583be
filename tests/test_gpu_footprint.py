"""pflbm_footprint_bytes bounds what a handle takes through its allocator, the
exchange memory of resident runs and the FP64 read-back's scratch included, for
any mask; and the runs that use that memory equal single steps bit for bit.
Masks: open channel, disc, dense blocks (whose exchange lists overflow shared
memory), one-node slits and pores (the most links), a corridor that fills a
corner of a large lattice.
"""
import numpy as np
import pytest

from tests.test_gpu_resident_members import dense

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _frame(nx, ny):
    return dense(nx, ny, 1, 10 * (nx + ny))


def _disc(nx, ny):
    from paper_2312_00369_gb300 import workloads as wl
    return wl.cylinder(nx, ny, nx / 2.0, ny / 2.0, 0.3 * ny)[0]


def _slits(nx, ny):
    s = _frame(nx, ny)
    s[:, ::5] = 1
    return s


def _corner(nx, ny):
    s = np.ones((ny, nx), np.uint8)
    s[2:ny // 3, : nx // 3] = 0
    return s


def _pores(nx, ny):
    s = np.ones((ny, nx), np.uint8)
    s[3:-3:4, 1::4] = 0
    return s


MASKS = {"frame": _frame, "disc": _disc, "dense3": lambda a, b: dense(a, b, 3, 6),
         "dense5": lambda a, b: dense(a, b, 5, 8), "slits": _slits, "pores": _pores, "corner": _corner}
SIZES = [(3, 5), (64, 32), (100, 50), (129, 65), (256, 128), (400, 200), (512, 512), (1000, 700)]


@pytest.mark.parametrize("precision", ["fp64", "fp32", "bf16", "fp16"])
@pytest.mark.parametrize("mask", sorted(MASKS))
def test_footprint_bounds_what_a_handle_takes(precision, mask, monkeypatch):
    from paper_2312_00369_gb300 import pflbm
    taken = []

    def alloc(nbytes, ctx):
        taken.append(nbytes)
        return pflbm._torch_alloc(nbytes, ctx)

    monkeypatch.setattr(pflbm, "_TORCH_ALLOC", pflbm._ALLOC(alloc))
    for nx, ny in SIZES:
        got = []
        for kernel in ("default", "global"):
            taken.clear()
            s = pflbm.Solver(MASKS[mask](nx, ny), theta_deg=70.0, precision=precision, step_kernel=kernel, dgdt_mode=1)
            s.init_droplet(0.3 * nx, 0.4 * ny, 0.3 * min(nx, ny))
            for n in (300, 17) if nx * ny < 100_000 else (260,):
                s.step(n)
            got.append(s.get() + (s.mass(),))
            s.check()
            s.close()
            assert sum(taken) <= pflbm.pflbm_footprint_bytes(nx, ny, precision), (nx, ny, kernel, sum(taken))
        for a, b in zip(*got):
            assert np.array_equal(a, b), (nx, ny)
