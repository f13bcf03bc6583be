"""The autotuner times runs as long as those it tunes for, so that a schedule is not
chosen by runs of fewer than 16 steps and then used for hundreds: on a few small
lattices, whose runs of many steps go through shared memory with the two-node
schedule (3.5 us a step, any other schedule above 6), it chooses that one.
"""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_default_search_sees_runs_of_many_steps(monkeypatch, tmp_path):
    from paper_2312_00369_gb300 import autotune, pflbm, workloads as wl
    monkeypatch.setenv("PFLBM_TUNE_CACHE", str(tmp_path / "sched.json"))
    cases = [wl.batch_instance(None, 128, 64, i % 3, 60.0 + i, 200) for i in range(4)]
    runs = []
    step = pflbm.Batch.step
    monkeypatch.setattr(pflbm.Batch, "step", lambda self, n=1: (runs.append(n), step(self, n))[1])
    best, timings = autotune.tune(cases, "fp16")
    assert min(runs) >= 16 and max(runs) >= 100
    assert best["kernel"] == 3, timings
