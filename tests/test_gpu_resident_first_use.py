"""A handle's first resident run: when it plans and takes its exchange memory,
that a capture in global mode elsewhere survives it, and the index-checked build
over both runs of a handle. The fields equal those of single steps bit for bit.
"""
import os
import subprocess
import sys

import numpy as np
import pytest

from tests import test_gpu_resident as res

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


RUNS = [  # nx, ny, precision, (steps of a run, whether it takes the memory)
    (131, 70, "fp64", [(15, False), (16, True)]),
    (131, 70, "fp32", [(16, False), (15, False), (17, True)]),
    (131, 70, "fp16", [(39, False), (16, True)]),
    (131, 70, "fp32", [(40, True)]),
    (131, 70, "bf16", [(16, False), (3, False), (500, True)]),
    (400, 300, "fp32", [(63, False), (16, True)]),
    (400, 300, "fp16", [(64, True)]),
]


@pytest.mark.parametrize("nx,ny,precision,runs", RUNS, ids=str)
def test_when_a_handle_takes_exchange_memory(nx, ny, precision, runs, monkeypatch):
    """Short first runs cost what single steps cost: nothing is planned or allocated
    before a first run long enough or a second one (steps in between do not count)."""
    from paper_2312_00369_gb300 import pflbm
    taken = []

    def alloc(nbytes, ctx):
        taken.append(nbytes)
        return pflbm._torch_alloc(nbytes, ctx)

    monkeypatch.setattr(pflbm, "_TORCH_ALLOC", pflbm._ALLOC(alloc))
    many = res._solver(res._blocks, nx, ny, precision, "default", {})
    one = res._solver(res._blocks, nx, ny, precision, "global", {})
    for n, resident in runs:
        taken.clear()
        many.step(n)
        assert (len(taken) > 0) == resident, (n, taken)
        one.step(n)
    for a, b in zip(res._state(many), res._state(one)):
        assert np.array_equal(a, b)
    many.close()
    one.close()


def test_capture_elsewhere_survives_first_use():
    """The first resident run of a handle with cudaMalloc memory, while another stream
    is captured in global mode by the same thread: steps never allocated before resident
    runs, so such a capture was never disturbed by them."""
    from paper_2312_00369_gb300.pflbm import Solver
    mine, other = torch.cuda.Stream(), torch.cuda.Stream()
    pair = [Solver(res._frame(100, 50), precision="fp32", stream=mine, step_kernel=k, torch_memory=False)
            for k in ("default", "global")]
    for s in pair:
        s.init_droplet(50.0, 0.5, 20.0)
        s.step(1)
    x = torch.zeros(1 << 20, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=other, capture_error_mode="global"):
        x += 1
        pair[0].step(200)
        x += 2
    pair[1].step(200)
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    assert bool((x == 9).all())
    for a, b in zip(res._state(pair[0]), res._state(pair[1])):
        assert np.array_equal(a, b)
    del graph
    for s in pair:
        s.close()


BOUNDS_SCRIPT = """
import numpy as np
from tests import test_gpu_resident as t
from tests.test_gpu_resident_members import dense
from paper_2312_00369_gb300 import pflbm
assert pflbm.debug_bounds()[0]
masks = t.CASES + [(lambda a, b: dense(a, b, 3, 6), 256, 128, 40, {}), (lambda a, b: dense(a, b, 5, 8), 400, 300, 40, {})]
for mask, nx, ny, steps, options in masks:
    for precision in ("fp64", "fp32", "bf16"):
        s = t._solver(mask, nx, ny, precision, "default", options)
        s.step(16)
        s.step(max(17, min(steps, 64)))
        s.check()
        assert np.isfinite(s.get()[0]).all()
        s.close()
print("violations", pflbm.debug_bounds()[1])
"""


def test_no_index_outside_its_buffer_in_a_second_run():
    from paper_2312_00369_gb300 import pflbm
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, PFLBM_LIBRARY=pflbm.BOUNDS_LIB_PATH, PYTHONPATH=root)
    r = subprocess.run([sys.executable, "-c", BOUNDS_SCRIPT], cwd=root, env=env, capture_output=True, text=True,
                       timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    assert r.stdout.strip().endswith("violations 0"), r.stdout
