"""Few particles in a large box, whose cells outnumber them: a grid of up to 2^17
cells is prepared by one cluster, up to 2^22 by all SMs, a larger one by the
separate kernels (which systems created with timing = 1 run anyway).  Contact
sets, colours, impulses and states are bit-equal on both sides of each line."""
import numpy as np
import pytest

from gpu_common import gpu_system, needs_gpu
from paper_1104_3516_gb300 import workloads as W

pytestmark = [pytest.mark.gpu, needs_gpu]


def corner(dim, n, cells):
    """n touching particles in the corner of a box of `cells` cells per axis."""
    r = W.uniform(3, n, 0.8, 1.2)
    k = int(np.ceil(n ** (1.0 / dim)))
    x = np.stack(np.meshgrid(*[np.arange(k)] * dim, indexing="ij"), -1).reshape(-1, dim)[:n] * 2.1 + 1.2
    inv_m, inv_I = W.masses(dim, r)
    side = (2.0 * float(r.max()) + 0.24) * (1.0 + 1e-8)
    hi = tuple(c * side for c in cells) + (1.0,) * (3 - dim)
    down = (0.0, -1.0, 0.0) if dim == 2 else (0.0, 0.0, -1.0)
    return W.Workload(name="corner", dim=dim, x=x, v=W.normal(2, dim * n, 0.1).reshape(n, dim),
                      w=np.zeros(n) if dim == 2 else np.zeros((n, 3)), r=r, inv_m=inv_m, inv_I=inv_I, gravity=down,
                      box_hi=hi, wall_mask=0b0100 if dim == 2 else 0b010000)


@pytest.mark.parametrize("dim, cells, fused", [(2, (512, 256), True), (2, (513, 256), True), (2, (2048, 2048), True),
                                               (2, (2049, 2048), False), (2, (3000, 3000), False),
                                               (3, (64, 64, 32), True), (3, (65, 64, 32), True),
                                               (3, (256, 128, 128), True), (3, (257, 128, 128), False)])
@pytest.mark.parametrize("n", [600, 8000])
def test_large_boxes(dim, cells, fused, n):
    wl = corner(dim, n, cells)
    a, b = gpu_system(wl, timing=1, max_sweeps=40), gpu_system(wl, max_sweeps=40)
    assert a.detect_contacts() == b.detect_contacts() > n // 2
    for _ in range(2):
        sa, sb = a.step(1), b.step(1)
        assert (sb["kernel_launches"] < sa["kernel_launches"] - 15) == fused
        ca, cb = a.contacts(), b.contacts()
        for k in ca:
            assert np.array_equal(ca[k], cb[k]), k
        xa, xb = a.state(), b.state()
        for k in ("x", "v", "w"):
            assert np.array_equal(xa[k], xb[k]), k
