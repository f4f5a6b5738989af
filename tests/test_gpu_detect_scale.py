"""The contact set does not depend on the unit of length: with every length times
a power of two (which FP64 does without rounding) the pairs and normals are the
same bits and the gaps times that power.  At 2^-74 the squares of distances
leave the range of single precision, in which far pairs are sorted out first."""
import copy

import numpy as np
import pytest

from gpu_common import gpu_system, needs_gpu
from paper_1104_3516_gb300 import workloads as W
from test_zz_no_alloc import _noalloc, _periodic_gas_3d

pytestmark = [pytest.mark.gpu, needs_gpu]


def scaled(wl, s):
    wl = copy.deepcopy(wl)
    wl.x, wl.r, wl.delta = wl.x * s, wl.r * s, wl.delta * s
    wl.box_lo = tuple(a * s for a in wl.box_lo)
    wl.box_hi = tuple(a * s for a in wl.box_hi)
    wl.wall_pos = np.asarray(wl.wall_pos) * s
    return wl


def by_system(wl, **kw):
    g = gpu_system(wl, max_contacts=60000, **kw)
    g.detect_contacts()
    c = g.contacts()
    return c["pairs"], c["normal"], c["gap"]


WAYS = {"without workspace": lambda wl: _noalloc(wl, 60000), "one kernel": by_system,
        "separate kernels": lambda wl: by_system(wl, timing=1)}


@pytest.mark.parametrize("make", [lambda: W.dense_biaxial_discs(seed=1, n=3000), _periodic_gas_3d])
@pytest.mark.parametrize("way", list(WAYS))
@pytest.mark.parametrize("e", [-74, -70, -60, 60, 70])
def test_lengths_times_a_power_of_two(make, way, e):
    wl = make()
    pairs, normal, gap = WAYS[way](wl)
    p, n, g = WAYS[way](scaled(wl, 2.0 ** e))
    assert len(pairs) > wl.n // 2
    assert np.array_equal(p, pairs) and np.array_equal(n, normal) and np.array_equal(g, gap * 2.0 ** e)
