"""Graph replays of a batch's launches: the captured graph holds 8 steps, each size
group's steps back to back on its own forked stream. Runs of fewer than 16 steps, and
longer ones kept off the resident path, from even and odd phases, against each
lattice stepped alone by the global-load kernel, bit for bit.
"""
import numpy as np
import pytest

from tests.test_gpu_batch import mix

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("use_graph", [0, 1])
@pytest.mark.parametrize("precision", ["fp32", "bf16"])
@pytest.mark.parametrize("runs,route", [([3, 15, 14, 8, 9, 1, 10], 0), ([3, 21, 16, 40, 33], 2)], ids=str)
def test_replays_of_several_size_groups(runs, route, precision, use_graph):
    from paper_2312_00369_gb300.pflbm import Batch, Solver, schedule
    stream = torch.cuda.Stream()
    cases = mix(seed=11, n=10)

    def make(kernel):
        out = []
        for c in cases:
            s = Solver(c.solid, theta_deg=c.theta_deg, precision=precision, stream=stream, step_kernel=kernel, **c.physical())
            for d in c.droplets:
                s.init_droplet(*d)
            out.append(s)
        return out

    together, alone = make("default"), make("global")
    b = Batch(together, schedule(use_graph=use_graph))
    assert b.kernel == 3 and b.info()["grid"] > 1            # launches per step: several size groups
    for n in runs:
        assert b.debug(n, route=route) == 0                  # no waves
        b.step(n)
    for s in alone:
        s.step(sum(runs))
    for x, y in zip(together, alone):
        assert x.steps == y.steps
        for p, q in zip(x.get(), y.get()):
            assert np.array_equal(p, q)
    b.close()
    for s in together + alone:
        s.close()
