"""What the one-kernel preparation cannot take ends the step before the solve:
more than 64 candidates at a disc, more than 64 colours, on one cluster of blocks
and on the grid.  The state stays as it was, on the first step and after a good
one, and the system steps on, equal to the separate kernels (timing = 1).  A solve
by itself refuses the set that was left without a colour order."""
import numpy as np
import pytest

from gpu_common import gpu_system, needs_gpu
from paper_1104_3516_gb300 import cd, workloads as W

pytestmark = [pytest.mark.gpu, needs_gpu]


def ringed(n, large_first):
    """n - 71 small discs apart from each other, and a large one (the first or
    the last disc) in a ring of 70: on it in the second set of positions."""
    ring = 70
    ang = np.linspace(0.0, 2.0 * np.pi, ring, endpoint=False)
    circle = np.stack([np.cos(ang), np.sin(ang)], 1)
    side = int(np.ceil(np.sqrt(n)))
    k = np.arange(n - ring - 1)
    field = np.stack([30.0 + 1.3 * (k % side), 1.0 + 1.3 * (k // side)], 1)
    centre = np.array([[12.0, 12.0]])
    sets = [np.concatenate([centre, 12.0 + rad * circle, field]) for rad in (6.5, 5.3)]
    r = np.concatenate([[5.0], np.full(ring, 0.2), np.full(len(field), 0.4)])
    if not large_first:
        sets, r = [np.roll(x, -1, axis=0) for x in sets], np.roll(r, -1)
    inv_m, inv_I = W.masses(2, r)
    wl = W.Workload(name="ringed", dim=2, x=sets[0], v=W.normal(1, 2 * n, 0.1).reshape(n, 2), w=np.zeros(n), r=r,
                    inv_m=inv_m, inv_I=inv_I, box_hi=(1.3 * side + 40.0, 1.3 * side + 40.0, 1.0), wall_mask=0b0100)
    return wl, sets


def put(g, x, v):
    import torch
    for dst, a in ((g.pos, x), (g.vel, v)):
        dst.copy_(torch.as_tensor(np.ascontiguousarray(a).reshape(-1), device=dst.device))


def whole(g):
    s = g.state()
    return [s["x"], s["v"], s["w"], g.walls()]


@pytest.mark.parametrize("n", [500, 20000])
@pytest.mark.parametrize("large_first", [True, False])
@pytest.mark.parametrize("kw", [{"max_sweeps": 20}, {"max_sweeps": 200}, {"max_sweeps": 200, "domains": (2, 2, 1)}])
@pytest.mark.parametrize("good_first", [False, True])
def test_a_step_that_cannot_be_prepared_leaves_the_state(n, large_first, kw, good_first):
    wl, (good, bad) = ringed(n, large_first)
    words = "64 contact candidates" if large_first else "64 colours"
    one, apart = gpu_system(wl, **kw), gpu_system(wl, timing=1, **kw)
    for g in (one, apart):
        if good_first:
            g.step(1)
        put(g, bad, wl.v)
        before = whole(g)
        for _ in range(2):
            with pytest.raises(cd.CDError, match=words) as e:
                g.step(2)
            assert e.value.status == cd.CD_ERR_CAPACITY
        for a, b in zip(before, whole(g)):
            assert np.array_equal(a, b)
        put(g, good, wl.v)
        g.step(2)
    for a, b in zip(whole(one), whole(apart)):
        assert np.array_equal(a, b)
    a, b = one.contacts(), apart.contacts()
    for k in a:
        assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("n", [500, 20000])
@pytest.mark.parametrize("timing", [0, 1])
@pytest.mark.parametrize("max_sweeps", [20, 200])
def test_a_set_without_a_colour_order_is_not_solved(n, timing, max_sweeps):
    wl, (good, bad) = ringed(n, large_first=False)
    g = gpu_system(wl, timing=timing, max_sweeps=max_sweeps)
    put(g, bad, wl.v)
    for fail in (lambda: g.step(1), g.detect_contacts):
        with pytest.raises(cd.CDError, match="64 colours"):
            fail()
    before = whole(g)
    g.load_checkpoint(g.save_checkpoint())   # counts as a set, and has no order either
    with pytest.raises(cd.CDError, match="colour order") as e:
        g.solve_contacts()
    assert e.value.status == cd.CD_ERR_STATE
    for a, b in zip(before, whole(g)):
        assert np.array_equal(a, b)
    # a checkpoint with more contacts than the set that was ordered last
    put(g, good, wl.v)
    more = g.detect_contacts()
    saved = g.save_checkpoint()
    put(g, np.concatenate([[[3.0, 25.0]], good[1:]]), wl.v)   # a disc of the ring alone
    assert 0 < g.detect_contacts() < more
    g.load_checkpoint(saved)
    with pytest.raises(cd.CDError, match="colour order"):
        g.solve_contacts()
    assert g.detect_contacts() == more
    g.solve_contacts()
    g.load_checkpoint(saved)   # of the set that is in order
    g.solve_contacts()


@pytest.mark.parametrize("n", [500, 16000])
def test_detection_without_workspace_counts_what_it_refuses(n):
    from test_zz_no_alloc import _noalloc
    wl, (good, bad) = ringed(n, large_first=True)
    wl.x = bad
    for _ in range(3):
        with pytest.raises(cd.CDError, match="64 contact candidates") as e:
            _noalloc(wl, 1000)
        assert e.value.status == cd.CD_ERR_CAPACITY and e.value.needed == 140   # 70 on the large disc, 70 along the ring
    wl.x = good
    assert len(_noalloc(wl, 1000)[0]) == 70


@pytest.mark.parametrize("kw", [{}, {"max_sweeps": 50}, {"domains": (2, 2, 1)}, {"timing": 1}])
def test_an_empty_set_from_a_checkpoint_is_solved(kw):
    wl, (good, _) = ringed(500, large_first=True)
    g = gpu_system(wl, **kw)
    empty = g.save_checkpoint()
    for detected in (False, True):
        if detected:
            g.detect_contacts()
        g.load_checkpoint(empty)
        before = whole(g)
        st = g.solve_contacts()
        assert st["converged"] and st["sweeps"] == 0 and st["n_contacts"] == 0
        for a, b in zip(before, whole(g)):
            assert np.array_equal(a, b)


def test_a_batch_solves_what_it_has_ranges_for():
    packs = [W.settling_discs(seed=s, n=60, vsig=0.5) for s in (1, 2)]
    g = gpu_system(packs[0], batch=packs, max_sweeps=200)
    empty = g.save_checkpoint()
    assert g.detect_contacts() > 0
    g.solve_contacts()
    full = g.save_checkpoint()
    g.load_checkpoint(empty)
    with pytest.raises(cd.CDError, match="colour order"):
        g.solve_contacts()
    g.load_checkpoint(full)
    g.solve_contacts()


@pytest.mark.parametrize("timing", [0, 1])
@pytest.mark.parametrize("domains", [(1, 1, 1), (2, 2, 1)])
def test_a_set_that_outlives_a_failed_step(timing, domains):
    """More contacts than room: the set before stays, and is solved with its colour
    order; not where its domain records went."""
    wl, (good, _) = ringed(500, large_first=True)
    more = good.copy()
    more[71:106] = good[1:36] + 0.05   # 35 discs of the field into the ring
    kw = dict(timing=timing, domains=domains, max_sweeps=200, max_contacts=100)
    g, twin = gpu_system(wl, **kw), gpu_system(wl, **kw)
    for s in (g, twin):
        assert s.detect_contacts() == 70
    put(g, more, wl.v)
    with pytest.raises(cd.CDError, match="capacity 100 exceeded"):
        g.step(1)
    put(g, good, wl.v)
    if domains == (1, 1, 1):
        assert g.solve_contacts()["n_contacts"] == 70
        twin.solve_contacts()
        for a, b in zip(whole(g), whole(twin)):
            assert np.array_equal(a, b)
    else:
        with pytest.raises(cd.CDError, match="colour order"):
            g.solve_contacts()
        assert g.detect_contacts() == 70
        g.solve_contacts()
