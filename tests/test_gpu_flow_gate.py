"""FP32 dataflow of systems so small that a block has no more warp items than warps
(and a little larger), against the barrier schedule: the same impulses, velocities
and sweeps, bit for bit.  Another block shape than the default keeps the barriers."""
import numpy as np
import pytest

from gpu_common import gpu_system, needs_gpu
from paper_1104_3516_gb300 import cd, workloads as W

pytestmark = [pytest.mark.gpu, needs_gpu]


def lattice(n, spacing):
    k = int(np.ceil(n ** (1.0 / 3.0)))
    x = np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n] * spacing + 1.5
    x = x + W.normal(6, 3 * n, 0.05).reshape(n, 3)
    r = W.uniform(6, n, 0.8, 1.2)
    inv_m, inv_I = W.masses(3, r)
    hi = (k * spacing + 3.0,) * 3
    return W.Workload(name="lattice", dim=3, x=x, v=W.normal(7, 3 * n, 0.1).reshape(n, 3), w=np.zeros((n, 3)), r=r,
                      inv_m=inv_m, inv_I=inv_I, gravity=(0.0, 0.0, -1.0), box_hi=hi, wall_mask=0b010000)


CASES = {f"spheres {n} {s}": (lambda n=n, s=s: lattice(n, s)) for n, s in ((7, 2.0), (400, 1.6), (3000, 1.6), (6000, 2.0),
                                                                        (20000, 2.0))}
CASES.update({f"discs {n}": (lambda n=n: W.dense_biaxial_discs(seed=2, n=n)) for n in (30, 3000, 20000)})


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("domains", [False, True])
def test_small_single_precision_systems(name, domains):
    wl = CASES[name]()
    kw = dict(precision=cd.CD_FP32, max_sweeps=150, max_contacts=8 * wl.n + 64,
              domains=(2,) * wl.dim + (1,) * (3 - wl.dim) if domains else (1, 1, 1))
    a, b = gpu_system(wl, **kw), gpu_system(wl, sweep_threads=256, sweep_blocks_per_sm=2, **kw)
    for _ in range(2):
        sa, sb = a.step(1), b.step(1)
        for k in ("sweeps", "n_contacts", "n_colours", "converged"):
            assert sa["last"][k] == sb["last"][k], k
        ca, cb = a.contacts(), b.contacts()
        for k in ca:
            assert np.array_equal(ca[k], cb[k]), k
        xa, xb = a.state(), b.state()
        for k in ("x", "v", "w"):
            assert np.array_equal(xa[k], xb[k]), k
