"""The autotuner times the kernel that the tuned system will run: a plain system
capped above 128 sweeps solves by dataflow, one capped at 128 or less behind
barriers, so a trial has its sweeps on the same side (no GPU needed: the systems
are stood in for)."""
import pytest

from paper_1104_3516_gb300 import autotune, workloads as W


class Recorder:
    made = []

    def __init__(self, wl, **kw):
        self.sweeps = kw["max_sweeps"]
        self.fast = kw["sweep_threads"] == 512
        Recorder.made.append(self.sweeps)

    def step(self, n):
        # the dataflow of the default shape against barriers, where the narrow shape is 2% faster
        per = 1.0 if self.fast and self.sweeps > 128 else 2.04 if self.fast else 2.0
        return {"phase_ms": {"sweep": n * self.sweeps * per}, "last": {"sweeps": self.sweeps}}


@pytest.mark.parametrize("cap, sweeps, threads", [(1000, 40, 512), (129, 40, 512), (129, 300, 512), (128, 40, 256),
                                                  (50, 40, 256), (100, 300, 256)])
@pytest.mark.parametrize("given", [False, True])
def test_trials_run_the_schedule_of_the_tuned_system(monkeypatch, cap, sweeps, threads, given):
    monkeypatch.setattr(autotune.cd, "CDSystem", Recorder)
    Recorder.made.clear()
    wl = W.settling_discs(seed=1, n=4)
    wl.max_sweeps = 7 if given else cap
    best, table = autotune.tune(wl, sweeps=sweeps, max_sweeps=cap if given else None)
    assert len(table) == len(autotune.BLOCK_SHAPES)
    assert all((s > 128) == (cap > 128) for s in Recorder.made)
    assert best["sweep_threads"] == threads
