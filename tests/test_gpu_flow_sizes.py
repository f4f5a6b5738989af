"""Systems on both sides of the particle counts up to which the solve runs by
dataflow, against the barriers that another block shape keeps: the same impulses,
velocities and sweeps, bit for bit, and a phase for each colour on either side."""
import numpy as np
import pytest
import torch

from gpu_common import gpu_system, needs_gpu
from paper_1104_3516_gb300 import cd, workloads as W

pytestmark = [pytest.mark.gpu, needs_gpu]


def lattice(dim, n):
    k = int(np.ceil(n ** (1.0 / dim)))
    x = np.stack(np.meshgrid(*[np.arange(k)] * dim, indexing="ij"), -1).reshape(-1, dim)[:n] * 2.0 + 1.5
    x = x + W.normal(6, dim * n, 0.05).reshape(n, dim)
    r = W.uniform(6, n, 0.8, 1.2)
    inv_m, inv_I = W.masses(dim, r)
    hi = (k * 2.0 + 3.0,) * dim + (1.0,) * (3 - dim)
    return W.Workload(name="lattice", dim=dim, x=x, v=W.normal(7, dim * n, 0.1).reshape(n, dim),
                      w=np.zeros(n) if dim == 2 else np.zeros((n, 3)), r=r, inv_m=inv_m, inv_I=inv_I,
                      gravity=(0.0, -1.0, 0.0) if dim == 2 else (0.0, 0.0, -1.0), box_hi=hi,
                      wall_mask=0b0100 if dim == 2 else 0b010000)


@pytest.mark.parametrize("dim, precision, per_sm", [(2, 1, 2300), (3, 1, 1100), (2, 0, 6000)])
@pytest.mark.parametrize("more", [0, 1])
@pytest.mark.parametrize("domains", [False, True])
def test_around_the_line(dim, precision, per_sm, more, domains):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    wl = lattice(dim, per_sm * sms + more)
    kw = dict(precision=precision, max_sweeps=130, max_contacts=4 * wl.n, criterion=cd.CD_CONV_NONE,
              domains=(2,) * dim + (1,) * (3 - dim) if domains else (1, 1, 1))
    a = gpu_system(wl, **kw)
    b = gpu_system(wl, sweep_threads=256, sweep_blocks_per_sm=2, merge_last_colour=0, **kw)
    sa, sb = a.step(1)["last"], b.step(1)["last"]
    assert sa["sweeps"] == sb["sweeps"] == 130 and sa["n_phases"] == sa["n_colours"] == sb["n_phases"]
    assert abs(sa["r_avg"] - sb["r_avg"]) <= (1e-12 if precision == 0 else 1e-5) * sb["r_avg"]
    ca, cb = a.contacts(), b.contacts()
    for k in ca:
        assert np.array_equal(ca[k], cb[k]), k
    xa, xb = a.state(), b.state()
    for k in ("x", "v", "w"):
        assert np.array_equal(xa[k], xb[k]), k
