"""The one-kernel preparation (detection, colouring, order and free flight of
plain systems) against the separate kernels, which systems created with
timing = 1 run: contact sets, colours, impulses and states are bit-equal."""
import numpy as np
import pytest

from gpu_common import gpu_system, needs_gpu
from paper_1104_3516_gb300 import workloads as W

pytestmark = [pytest.mark.gpu, needs_gpu]


def periodic_gas(n, floor):
    wl = W.sphere_gas(n=n, floor=floor, vsig=0.5)
    wl.periodic = (1, 1, 0)
    wl.wall_mask = 0b010000
    return wl


# 2D up to 7,000 and 3D up to 5,000 particles run as one cluster, larger ones
# as a grid; counts around a warp and a block's share of particles; a pile whose
# highest colour is repaired, an axis that wraps, a lid that is a body
CASES = {
    "1 disc": lambda: W.settling_discs(seed=1, n=1),
    "33 discs": lambda: W.settling_discs(seed=1, n=33, vsig=0.5),
    "513 discs": lambda: W.settling_discs(seed=1, n=513, vsig=0.5),
    "7000 discs": lambda: W.settling_discs(seed=1, n=7000, vsig=0.5),
    "7001 discs": lambda: W.settling_discs(seed=1, n=7001, vsig=0.5),
    "pile 3000": lambda: W.dense_biaxial_discs(seed=1, n=3000),
    "pile 20011": lambda: W.dense_biaxial_discs(seed=1, n=20011),
    "lid 700": lambda: W.pressure_column(seed=1, n=700),
    "gas 777": lambda: W.sphere_gas(seed=1, n=777, floor=14.0, vsig=0.5),
    "gas 12000": lambda: W.sphere_gas(seed=1, n=12000, floor=40.0, vsig=0.5),
    "periodic gas 3000": lambda: periodic_gas(3000, 20.0),
}


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("precision", [0, 1])
def test_prepared_steps_are_bit_identical(name, precision):
    wl = CASES[name]()
    kw = dict(precision=precision, max_sweeps=20, f_ext=0.01 * np.arange(wl.n * wl.dim) / (wl.n * wl.dim))
    a, b = gpu_system(wl, timing=1, **kw), gpu_system(wl, **kw)
    assert a.detect_contacts() == b.detect_contacts()
    for _ in range(3):   # the second and third are warm-started from the set before
        sa, sb = a.step(1), b.step(1)
        for k in ("sweeps", "n_contacts", "n_colours", "n_phases", "wall_force"):
            assert sa["last"][k] == sb["last"][k], k
        ca, cb = a.contacts(), b.contacts()
        for k in ca:
            assert np.array_equal(ca[k], cb[k]), k
        xa, xb = a.state(), b.state()
        for k in ("x", "v", "w"):
            assert np.array_equal(xa[k], xb[k]), k


def test_overflow_leaves_the_state_and_reports_the_need():
    from paper_1104_3516_gb300 import cd
    wl = W.dense_biaxial_discs(seed=1, n=500)
    need = gpu_system(wl).detect_contacts()
    g = gpu_system(wl, max_contacts=need - 1)
    before = g.state()
    for _ in range(2):
        with pytest.raises(cd.CDError) as e:
            g.step(2)
        assert e.value.status == cd.CD_ERR_CAPACITY and str(need) in e.value.message
    after = g.state()
    assert np.array_equal(before["x"], after["x"]) and np.array_equal(before["v"], after["v"])
    g = gpu_system(wl, max_contacts=need)
    assert g.detect_contacts() == need


def test_more_partners_than_the_counting_pass_keeps():
    """One large disc among many small ones: 30 partners (16 are kept), which
    the emitting pass walks for again."""
    small = 30
    ang = np.linspace(0.0, 2.0 * np.pi, small, endpoint=False)
    r = np.concatenate([[5.0], np.full(small, 0.4)])
    x = np.concatenate([[[10.0, 10.0]], 10.0 + 5.41 * np.stack([np.cos(ang), np.sin(ang)], 1)])
    inv_m, inv_I = W.masses(2, r)
    wl = W.Workload(name="ring", dim=2, x=x, v=np.zeros_like(x), w=np.zeros(small + 1), r=r, inv_m=inv_m, inv_I=inv_I,
                    box_hi=(60.0, 60.0, 1.0), max_sweeps=10)
    a, b = gpu_system(wl, timing=1, max_contacts=200), gpu_system(wl, max_contacts=200)
    a.step(2), b.step(2)
    ca, cb = a.contacts(), b.contacts()
    assert len(ca["pairs"]) >= small
    for k in ca:
        assert np.array_equal(ca[k], cb[k]), k
