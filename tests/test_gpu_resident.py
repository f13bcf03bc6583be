"""Runs of many steps on a lattice that fits the chip's shared memory (one
cooperative launch, csrc/resident.cu) against the same steps taken one launch
each with the global-load kernel. Both round alike, so the fields agree bit for
bit: there is no tolerance. The sizes are the edges of the path: one patch that
is its own periodic neighbour, patches of one or two nodes, odd widths, several
patches with unequal parts, the largest patches, lattices with solid patches
left out, walls and ghosts at patch borders, step counts of either parity and
beyond one launch.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _frame(nx, ny):
    s = np.zeros((ny, nx), np.uint8)
    s[:2] = s[-2:] = 1
    return s


def _blocks(nx, ny, seed=5):
    """Solid blocks and single solid nodes all over: links and ghosts everywhere."""
    rng = np.random.default_rng(seed)
    s = _frame(nx, ny)
    for _ in range(max(2, nx * ny // 300)):
        x, y, w, h = rng.integers(nx), rng.integers(2, ny - 2), rng.integers(1, 7), rng.integers(1, 7)
        s[y:y + h, x:x + w] = 1
    return s


def _slope(nx, ny):
    from paper_2312_00369_gb300 import workloads as wl
    return wl.inclined(nx, ny, 30.0)[0]


def _disc(nx, ny):
    from paper_2312_00369_gb300 import workloads as wl
    return wl.cylinder(nx, ny, nx / 2.0, ny / 2.0, 0.3 * ny)[0]


CASES = [  # mask, nx, ny, steps, options
    (_frame, 3, 5, 16, {}),
    (_frame, 4, 9, 17, {}),
    (_frame, 7, 12, 40, dict(chi_case=1)),
    (_frame, 33, 18, 33, dict(dgdt_mode=1)),
    (_frame, 64, 32, 1030, {}),
    (_blocks, 65, 33, 48, {}),
    (_frame, 100, 50, 101, dict(nu_l=0.3, nu_g=0.05, gx=2e-6, gy=-1e-6)),
    (_blocks, 131, 70, 37, dict(chi_case=3)),
    (_slope, 150, 90, 64, {}),
    (_disc, 301, 203, 35, dict(dgdt_mode=1)),
    (_blocks, 400, 200, 32, {}),
    (_disc, 512, 512, 20, {}),
    (_slope, 513, 400, 21, dict(nu_l=0.2, nu_g=0.1)),
]


def _solver(mask, nx, ny, precision, kernel, options):
    from paper_2312_00369_gb300.pflbm import Solver
    rng = np.random.default_rng(nx + ny)
    theta = rng.uniform(40.0, 140.0, (ny, nx)).astype(np.float32)
    s = Solver(mask(nx, ny), theta_field=theta, precision=precision, step_kernel=kernel, **options)
    s.init_droplet(0.4 * nx, 0.3 * ny, 0.25 * min(nx, ny))
    s.init_droplet(0.9 * nx, 0.6 * ny, 0.2 * min(nx, ny))     # across the periodic seam
    return s


def _state(s):
    return (*s.get(), s.mass())


@pytest.mark.parametrize("precision", ["fp64", "fp32", "bf16", "fp16"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: f"{c[0].__name__[1:]}{c[1]}x{c[2]}")
def test_resident_equals_single_steps(case, precision):
    mask, nx, ny, steps, options = case
    many = _solver(mask, nx, ny, precision, "default", options)
    one = _solver(mask, nx, ny, precision, "global", options)
    try:
        # a run, a few single steps from the copy it ended in, a run again
        for n in (steps, 3, 17):
            many.step(n)
            one.step(n)
            assert many.steps == one.steps
            for a, b, what in zip(_state(many), _state(one), ("phi", "u", "p", "mass")):
                assert np.array_equal(a, b), (n, what, np.max(np.abs(np.asarray(a) - b)))
        many.check()
    finally:
        many.close()
        one.close()


def test_resident_runs_from_a_checkpoint_and_new_angles():
    a = _solver(_frame, 100, 50, "fp32", "default", {})
    b = _solver(_frame, 100, 50, "fp32", "global", {})
    a.step(40)
    blob = a.save()
    a.step(25)
    a.load(blob)                       # back to step 40: other data in the copies
    b.step(40)
    theta = np.full((50, 100), 75.0, np.float32)
    for s in (a, b):
        s.set_theta_field(theta)
        s.step(31)
    for x, y in zip(_state(a), _state(b)):
        assert np.array_equal(x, y)
    a.close()
    b.close()


def test_captured_steps_replay():
    # a stream under capture takes single steps: the graph replays them
    from paper_2312_00369_gb300.pflbm import Solver
    stream = torch.cuda.Stream()
    pair = [Solver(_frame(100, 50), precision="fp32", stream=stream, step_kernel=k) for k in ("default", "global")]
    for s in pair:
        s.init_droplet(50.0, 0.5, 20.0)
        s.step(20)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        pair[0].step(20)               # an even count: the copies end as they began
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    pair[1].step(60)
    for x, y in zip(_state(pair[0]), _state(pair[1])):
        assert np.array_equal(x, y)
    del graph
    for s in pair:
        s.close()


BOUNDS_SCRIPT = """
import numpy as np
from tests import test_gpu_resident as t
from paper_2312_00369_gb300 import pflbm
assert pflbm.debug_bounds()[0]
for mask, nx, ny, steps, options in t.CASES:
    for precision in ("fp64", "fp32", "bf16"):
        s = t._solver(mask, nx, ny, precision, "default", options)
        s.step(min(steps, 64))
        s.check()
        assert np.isfinite(s.get()[0]).all()
        s.close()
print("violations", pflbm.debug_bounds()[1])
"""


def test_no_index_outside_its_buffer():
    import os
    import subprocess
    import sys
    from paper_2312_00369_gb300 import pflbm
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, PFLBM_LIBRARY=pflbm.BOUNDS_LIB_PATH, PYTHONPATH=root)
    r = subprocess.run([sys.executable, "-c", BOUNDS_SCRIPT], cwd=root, env=env, capture_output=True, text=True,
                       timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    assert r.stdout.strip().endswith("violations 0"), r.stdout


BATCH = [  # mask, nx, ny, options: 1 to 100 patches, odd widths, one lattice that does not fit
    (_frame, 64, 32, {}), (_slope, 128, 64, {}), (_blocks, 65, 33, dict(chi_case=1)),
    (_disc, 256, 128, dict(nu_l=0.3, nu_g=0.05, gx=2e-6, gy=-1e-6)), (_frame, 3, 9, {}), (_slope, 512, 256, {}),
    (_frame, 301, 203, {}), (_frame, 1200, 400, {}), (_disc, 512, 256, dict(dgdt_mode=1)),
]


@pytest.mark.parametrize("precision", ["fp32", "bf16", "fp16"])
def test_resident_batch_equals_single_steps(precision):
    from paper_2312_00369_gb300.pflbm import Batch
    stream = torch.cuda.Stream()
    many = [_solver(*c[:3], precision, "default", dict(c[3], stream=stream)) for c in BATCH]
    one = [_solver(*c[:3], precision, "global", dict(c[3], stream=stream)) for c in BATCH]
    b = Batch(many)
    # resident runs of either parity, single steps between, a member stepped
    # alone, a change of members
    for n in (16, 3, 37):
        b.step(n)
        for s in one:
            s.step(n)
    many[1].step(5)
    one[1].step(5)
    b.step(20)
    for s in one:
        s.step(20)
    b.set(many[:4])
    b.step(17)
    for s in one[:4]:
        s.step(17)
    for c, x, y in zip(BATCH, many, one):
        assert x.steps == y.steps
        for p, q, what in zip(_state(x), _state(y), ("phi", "u", "p", "mass")):
            assert np.array_equal(p, q), (c[1:3], what)
        x.check()
    b.close()
    for s in many + one:
        s.close()


@pytest.mark.parametrize("nx,ny", [(1024, 640), (1021, 643)])
@pytest.mark.parametrize("visc", [{}, dict(nu_l=0.3, nu_g=0.05)])
def test_alternating_rows_equal_the_staged_kernel(visc, nx, ny):
    """Single steps of lattices larger than the alternation's lower line take the
    tile rows up and down in turn; the staged kernel, which never does, gives
    the same bits (the per-node arithmetic is shared and a step only reads the
    other copy, so no order can matter)."""
    from paper_2312_00369_gb300 import workloads as wl
    from paper_2312_00369_gb300.pflbm import Solver
    c = wl.many_droplets_flat(nx, ny, 4)
    got = []
    for k in ("default", "staged32x8"):
        s = Solver(c.solid, theta_deg=c.theta_deg, theta_field=c.theta_field, precision="fp32", step_kernel=k,
                   **{**c.physical(), **visc})
        for d in c.droplets:
            s.init_droplet(*d)
        for n in (1, 2, 7, 1):
            s.step(n)
        got.append(s.get() + (s.mass(),))
        s.close()
    for a, b in zip(*got):
        assert np.array_equal(a, b)
