"""Which way a batch takes a run of many steps, waves of members held in shared memory or
launches per size group, and that both give what the members give alone, bit for bit.

The routes are those that were measured to be faster by a wide margin (a step of
either is in csrc/batch.cu), on both sides of the line; the bit comparison forces
the waves where the estimate may choose the launches.
"""
import numpy as np
import pytest

from tests import test_gpu_resident as res

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _members(sizes, precision, stream):
    from paper_2312_00369_gb300 import workloads as wl
    from paper_2312_00369_gb300.pflbm import Solver
    out = []
    for i, (nx, ny, wall) in enumerate(sizes):
        c = wl.batch_instance(None, nx, ny, wall, 60.0 + i % 60, 200)
        s = Solver(c.solid, theta_deg=c.theta_deg, precision=precision, stream=stream, dgdt_mode=1, **c.physical())
        for d in c.droplets:
            s.init_droplet(*d)
        out.append(s)
    return out


def _uneven(n, wall=None):
    from paper_2312_00369_gb300 import workloads as wl
    return [(c.nx, c.ny, i % 3 if wall is None else wall) for i, c in enumerate(wl.batched_instances()[:n])]


def _requests(n):
    from paper_2312_00369_gb300 import workloads as wl
    return [(d["nx"], d["ny"], d["wall_type"]) for d in wl.request_stream(n_max=n)]


ROUTES = [  # members, precision, steps, waves?
    (lambda: _requests(16), "fp16", 200, True),
    (lambda: _requests(8), "fp32", 200, True),
    (lambda: _requests(8), "fp32", 16, False),          # the set-up of the waves outweighs 16 steps
    (lambda: _uneven(256), "bf16", 200, True),
    (lambda: _uneven(256, wall=0), "bf16", 200, False),
    (lambda: _uneven(16), "fp32", 200, False),
    (lambda: [(400, 200, 0)] * 31, "fp32", 200, False),
    (lambda: [(528, 264, 0)] * 18, "fp16", 200, False),
    (lambda: [(528, 264, 0)] * 18, "fp16", 10**9, False),
    (lambda: [(128, 64, 0)] * 4, "fp16", 200, True),
    (lambda: [(128, 64, 0)] * 4, "fp16", 15, False),
    (lambda: [(128, 64, 0)] * 4, "fp64", 200, False),
]


@pytest.mark.parametrize("k", range(len(ROUTES)))
def test_route_is_the_faster_one(k):
    from paper_2312_00369_gb300.pflbm import Batch
    members, precision, steps, waves = ROUTES[k]
    solvers = _members(members(), precision, torch.cuda.Stream())
    b = Batch(solvers)
    assert (b.debug(steps) > 0) == waves
    b.close()
    for s in solvers:
        s.close()


@pytest.mark.parametrize("route", [1, 2])
@pytest.mark.parametrize("precision", ["fp32", "bf16", "fp16"])
def test_both_routes_equal_single_steps(precision, route):
    from paper_2312_00369_gb300.pflbm import Batch
    stream = torch.cuda.Stream()
    many, one = ([res._solver(*c[:3], precision, kernel, dict(c[3], stream=stream)) for c in res.BATCH]
                 for kernel in ("default", "global"))
    b = Batch(many)
    assert (b.debug(16, route=route) > 0) == (route == 1)
    # runs of either parity, single steps between, a member stepped alone, a change
    # of members
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
    for c, x, y in zip(res.BATCH, many, one):
        assert x.steps == y.steps
        for p, q, what in zip(res._state(x), res._state(y), ("phi", "u", "p", "mass")):
            assert np.array_equal(p, q), (c[1:3], what)
        x.check()
    b.close()
    for s in many + one:
        s.close()
