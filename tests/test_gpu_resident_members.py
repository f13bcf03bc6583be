"""Batches whose members change between resident runs (waves of k_resident), against
the same lattices stepped alone by the global-load kernel, bit for bit.

The members are lattices of dense obstacles: solid blocks every few nodes give a
patch more exchange entries and bounce-back copies than its lists in shared
memory hold, so the lists overflow to global memory. Sets of members large,
small, then large again move everything that is laid out per set.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def dense(nx, ny, block, period):
    """Square blocks every `period` nodes between the walls."""
    s = np.zeros((ny, nx), np.uint8)
    s[:2] = s[-2:] = 1
    for y in range(5, ny - 5 - block, period):
        for x in range(1, nx - block, period):
            s[y:y + block, x:x + block] = 1
    return s


SIZES = [(256, 128, 3, 6), (256, 128, 5, 8), (192, 96, 3, 6), (128, 64, 3, 6), (128, 64, 5, 8), (96, 40, 3, 6)]


def _make(precision, kernel, stream):
    from paper_2312_00369_gb300.pflbm import Solver
    out = []
    for i, (nx, ny, block, period) in enumerate(SIZES):
        s = Solver(dense(nx, ny, block, period), theta_deg=60.0 + 10 * i, precision=precision, step_kernel=kernel,
                   stream=stream, dgdt_mode=1)
        s.init_droplet(0.4 * nx, 0.5 * ny, 0.3 * ny)
        out.append(s)
    return out


@pytest.mark.parametrize("precision", ["fp32", "bf16", "fp16"])
def test_members_large_small_large(precision):
    from paper_2312_00369_gb300.pflbm import Batch
    stream = torch.cuda.Stream()
    many, one = _make(precision, "default", stream), _make(precision, "global", stream)
    sets = [range(6), [5], [3, 4], range(6), [4], range(6), [2, 5], [0, 1, 3]]
    b = Batch([many[i] for i in sets[0]])
    assert b.debug(16, route=1) >= 1               # waves, whatever the estimate says
    for k, members in enumerate(sets):
        if k:
            b.set([many[i] for i in members])
        n = (16, 17, 40, 16, 300, 19, 16, 33)[k]
        b.step(n)
        for i in members:
            one[i].step(n)
        for i in members:
            for p, q, what in zip(many[i].get() + (many[i].mass(),), one[i].get() + (one[i].mass(),), "phi u p mass".split()):
                assert np.array_equal(p, q), (k, SIZES[i], what)
            many[i].check()
    b.close()
    for s in many + one:
        s.close()


@pytest.mark.parametrize("refuse_after", [0, 1, 2, 3])
@pytest.mark.parametrize("before", [0, 3])
def test_refused_launch_falls_back(refuse_after, before):
    """A refused cooperative launch: before any, after one wave's first launch of
    1024 steps, between waves, in a later wave, from either phase. The batch takes
    the launches for what is left and stays with them."""
    from paper_2312_00369_gb300.pflbm import Batch, Solver
    stream = torch.cuda.Stream()
    sizes = [(192, 96), (192, 96), (320, 160), (256, 256), (100, 50), (300, 200), (256, 256), (256, 256), (256, 256)]
    def make(kernel):
        out = []
        for i, (nx, ny) in enumerate(sizes):
            s = Solver(dense(nx, ny, 3, 40), theta_deg=50.0 + 10 * i, precision="fp16", step_kernel=kernel, stream=stream,
                       dgdt_mode=1)
            s.init_droplet(0.4 * nx, 0.5 * ny, 0.3 * ny)
            out.append(s)
        return out
    many, one = make("default"), make("global")
    b = Batch(many)
    n = 1029
    b.step(before)
    assert b.debug(n, route=1, refuse_after=refuse_after) >= 2
    b.step(n)
    assert b.debug(n, route=1) == 0
    b.step(17)
    b.set(many[:3])
    b.step(20)
    for s in one:
        s.step(before + n + 17)
    for s in one[:3]:
        s.step(20)
    for x, y, size in zip(many, one, sizes):
        assert x.steps == y.steps
        for p, q, what in zip(x.get() + (x.mass(),), y.get() + (y.mass(),), "phi u p mass".split()):
            assert np.array_equal(p, q), (size, what)
        x.check()
    b.close()
    for s in many + one:
        s.close()
