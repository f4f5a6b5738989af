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


def small(n, spacing, seed):
    """n discs on a jittered lattice: at spacing 1 they have 16 contacts each."""
    k = int(np.ceil(np.sqrt(n)))
    x = np.stack(np.meshgrid(np.arange(k), np.arange(k), indexing="ij"), -1).reshape(-1, 2)[:n] * spacing + 1.5
    r = W.uniform(seed, n, 0.8, 1.2)
    inv_m, inv_I = W.masses(2, r)
    return W.Workload(name="small", dim=2, x=x + W.normal(seed, 2 * n, 0.05).reshape(n, 2), v=np.zeros((n, 2)),
                      w=np.zeros(n), r=r, inv_m=inv_m, inv_I=inv_I, gravity=(0.0, -1.0, 0.0),
                      box_hi=(k * spacing + 3.0,) * 2 + (1.0,), wall_mask=0b0100, seed=seed)


# few packings: by dataflow; very many, and many crowded ones: left to the barriers;
# among many one that is crowded, or very large
@pytest.mark.parametrize("packs", [
    lambda: [small(300, 1.9, b) for b in range(3)], lambda: [small(20, 1.9, b % 5) for b in range(1500)],
    lambda: [small(1500, 1.0, b % 5) for b in range(90)], lambda: [small(2000, 1.9, b % 5) for b in range(60)] + [small(300, 1.0, 1)],
    lambda: [small(20, 1.9, b % 5) for b in range(900)] + [small(30000, 1.9, 1)]])
@pytest.mark.parametrize("precision", [0, 1])
def test_either_schedule_solves_each_packing_as_alone(packs, precision):
    packs = packs()
    kw = dict(precision=precision, criterion=cd.CD_CONV_NONE, max_sweeps=25)
    per = 10
    g = gpu_system(packs[0], batch=packs, max_contacts=per * sum(p.n for p in packs), **kw)
    g.step(1)
    s = g.state()
    for b in {0, len(packs) // 2, len(packs) - 1}:
        alone = gpu_system(packs[b], max_contacts=per * packs[b].n, **kw)
        alone.step(1)
        at = slice(g.offsets[b], g.offsets[b + 1])
        for k in ("x", "v", "w"):
            assert np.array_equal(s[k][at], alone.state()[k]), (b, k)
