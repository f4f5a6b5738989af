"""cd_detect_contacts_noalloc lays its cell grid out on the device: the contact
set against cd_detect_contacts (grid on the host) at one particle, around a
warp, at the largest count of one cluster and past it, and at the limit; and
what it refuses for the grid's sake is refused as before, with the next call
unharmed."""
import copy

import numpy as np
import pytest

from gpu_common import gpu_system, needs_gpu
from paper_1104_3516_gb300 import cd, workloads as W
from test_zz_no_alloc import _noalloc

pytestmark = [pytest.mark.gpu, needs_gpu]


def same(wl):
    s = gpu_system(wl, max_contacts=65536)
    s.detect_contacts()
    c = s.contacts()
    pairs, normal, gap = _noalloc(wl, 65536)
    assert np.array_equal(pairs, c["pairs"])
    assert np.array_equal(normal, c["normal"])
    assert np.array_equal(gap, c["gap"])


@pytest.mark.parametrize("n", [1, 2, 31, 33, 1000, 7000, 7001, 16384])
def test_discs(n):
    same(W.settling_discs(seed=n, n=n) if n < 40 else W.dense_biaxial_discs(seed=n, n=n))


@pytest.mark.parametrize("n", [1000, 5000, 5001, 16384])
def test_spheres(n):
    same(W.sphere_gas(seed=n, n=n, floor=40.0))


def test_few_contacts():
    same(W.dilute_discs(seed=3, n=700, width=60.0))


def test_refusals():
    good = W.dense_biaxial_discs(seed=1, n=500)
    for change, words in ((lambda w: w.r.__setitem__(7, 0.0), "radius"), (lambda w: w.r.__setitem__(7, np.inf), "radius"),
                          (lambda w: w.r.__setitem__(7, np.nan), "radius"),
                          (lambda w: (w.r.__setitem__(slice(None), 1e-4), setattr(w, "delta", 1e-4)), "65536 cells")):
        wl = copy.deepcopy(good)
        change(wl)
        with pytest.raises(cd.CDError, match=words):
            _noalloc(wl, 10000)
    wl = W.sphere_gas(n=200, floor=12.0)
    wl.periodic = (1, 1, 0)
    wl.wall_mask = 0b010000
    wl.r[:] = 3.0
    with pytest.raises(cd.CDError, match="at least 3 cells"):
        _noalloc(wl, 10000)
    same(good)
