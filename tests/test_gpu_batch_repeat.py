"""A batch repeats itself: which block solves which packing depends on timing,
what comes out does not, to the last bit of the statistics."""
import numpy as np
import pytest

from gpu_common import gpu_system, needs_gpu
from paper_1104_3516_gb300 import cd, workloads as W

pytestmark = [pytest.mark.gpu, needs_gpu]


def result(g):
    per = g.packing_stats()
    s = g.state()
    return [np.array([p[k] for p in per]) for k in ("sweeps", "converged", "residual", "r_avg", "wall_force")] + \
           [s["x"], s["v"], s["w"], g.contacts()["impulse"]]


@pytest.mark.parametrize("m, nmin, nmax", [(150, 50, 4000), (40, 2000, 6000), (400, 20, 600)])
@pytest.mark.parametrize("precision", [0, 1])
def test_a_batch_repeats_itself(m, nmin, nmax, precision):
    packs = [W.settled_pile(seed=77 + b, n=int(n), mu=0.3)
             for b, n in enumerate(W.batch_sizes(n_packings=m, nmin=nmin, nmax=nmax))]
    g = gpu_system(packs[0], batch=packs, precision=precision, criterion=cd.CD_CONV_GLOBAL_REL, max_sweeps=400,
                   max_contacts=4 * sum(p.n for p in packs))
    start = g.save_checkpoint()
    runs = []
    for _ in range(4):
        g.load_checkpoint(start)
        g.step(2)
        runs.append(result(g))
    for other in runs[1:]:
        for a, b in zip(runs[0], other):
            assert np.array_equal(a, b)
