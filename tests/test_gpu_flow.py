"""The dataflow solve (batches, and plain systems whose sweep cap exceeds 128, without an
asked-for merge) against the barrier schedule on the same system: the order of
the updates is the same, so impulses, velocities and positions are bit-equal,
and the stopping sweep is the same (a solve that stops after sweeps that were
started before their test was known takes them back).  merge_last_colour = 1
keeps the barrier schedule."""
import numpy as np
import pytest

from gpu_common import gpu_system, needs_gpu
from paper_1104_3516_gb300 import workloads as W

pytestmark = [pytest.mark.gpu, needs_gpu]


def both(wl, steps=2, **kw):
    a = gpu_system(wl, merge_last_colour=1, **kw)
    b = gpu_system(wl, merge_last_colour=4, **kw)
    sa = [a.step(1) for _ in range(steps)]
    sb = [b.step(1) for _ in range(steps)]
    for x, y in zip(sa, sb):
        for k in ("sweeps", "converged", "n_contacts", "n_colours"):
            assert x["last"][k] == y["last"][k], k
        # the sums of |P| over the contacts differ in their order only
        assert abs(x["last"]["r_avg"] - y["last"]["r_avg"]) <= 1e-13 * x["last"]["r_avg"]
        assert np.allclose(x["last"]["wall_force"], y["last"]["wall_force"], rtol=1e-13, atol=0)
        assert y["last"]["n_phases"] == y["last"]["n_colours"]
    ca, cb = a.contacts(), b.contacts()
    for k in ("pairs", "colour", "impulse"):
        assert np.array_equal(ca[k], cb[k]), k
    xa, xb = a.state(), b.state()
    for k in ("x", "v", "w"):
        assert np.array_equal(xa[k], xb[k]), k
    return sb


# discs per block of 152 from one lane pair (a few contacts a colour in some
# blocks, none in others) over whole warps to several items a warp; 300,000
# exceed what the blocks' shared memory holds
@pytest.mark.parametrize("n", [3, 40, 700, 4999, 20011, 40000, 300000])
@pytest.mark.parametrize("precision", [0, 1])
def test_pile_is_bit_identical(n, precision):
    from paper_1104_3516_gb300 import cd
    wl = W.dense_biaxial_discs(seed=5, n=n) if n > 3 else W.settling_discs(seed=5, n=3)
    both(wl, steps=1 if n > 100000 else 2, criterion=cd.CD_CONV_NONE, max_sweeps=131, precision=precision,
         max_contacts=4 * n + 64)


@pytest.mark.parametrize("precision", [0, 1])
def test_spheres_are_bit_identical(precision):
    from paper_1104_3516_gb300 import cd
    for wl in (W.sphere_gas(n=3000, floor=20.0, vsig=0.5), W.sphere_gas(seed=3, n=20011, floor=40.0, vsig=0.5)):
        both(wl, criterion=cd.CD_CONV_NONE, max_sweeps=131, precision=precision)


# thresholds whose stopping sweep falls before, at and after the sweeps from
# which on one and two sweeps are started ahead of their test
@pytest.mark.parametrize("criterion", [0, 1])
@pytest.mark.parametrize("alpha", [1e-1, 3e-2, 1e-2, 5e-3, 2e-3, 1e-3, 3e-4, 1e-4])
def test_stops_at_the_same_sweep(alpha, criterion):
    wl = W.dense_biaxial_discs(seed=9, n=2000)
    sb = both(wl, steps=3, criterion=criterion, alpha=alpha if criterion == 0 else alpha * alpha, max_sweeps=5000)
    assert sb[0]["last"]["converged"]


def test_cap_reached_and_few_contacts():
    wl = W.dense_biaxial_discs(seed=2, n=1000)
    sb = both(wl, criterion=0, alpha=0.0, max_sweeps=129)
    assert sb[0]["last"]["sweeps"] == 129 and not sb[0]["last"]["converged"]
    both(W.dilute_discs(seed=4, n=200, width=20.0), steps=4)   # a handful of contacts, most colours empty in most blocks


@pytest.mark.parametrize("precision", [0, 1])
def test_force_controlled_lid_is_bit_identical(precision):
    """The lid is a body of many colours (its contacts conflict)."""
    both(W.pressure_column(seed=6, n=600), steps=3, precision=precision)


@pytest.mark.parametrize("count", [2, 7, 40, 200])
@pytest.mark.parametrize("precision", [0, 1])
def test_batches_are_bit_identical(count, precision):
    """Packings solved by teams of blocks (one round of teams, several rounds,
    packings without a contact among them) against the barrier schedule, which
    another block shape keeps."""
    batch = [W.settled_pile(seed=50 + b, n=int(n), mu=0.1 + 0.5 * b / count)
             for b, n in enumerate(W.batch_sizes(seed=3, n_packings=count, nmin=20, nmax=3000))]
    batch[1] = W.dilute_discs(seed=1, n=5, width=40.0)
    kw = dict(batch=batch, precision=precision, alpha=1e-3, max_sweeps=150, max_contacts=4 * sum(b.n for b in batch))
    a = gpu_system(batch[0], sweep_threads=256, sweep_blocks_per_sm=2, **kw)
    b = gpu_system(batch[0], **kw)
    for _ in range(2):
        sa, sb = a.step(1), b.step(1)
        for k in ("total_sweeps", "total_contact_updates", "max_sweeps_in_step", "n_not_converged"):
            assert sa[k] == sb[k], k
        for p, q in zip(a.packing_stats(), b.packing_stats()):
            for k in ("sweeps", "converged", "n_contacts", "wall_pos"):
                assert p[k] == q[k], k
            assert abs(p["r_avg"] - q["r_avg"]) <= 1e-13 * p["r_avg"]
            assert np.allclose(p["wall_force"], q["wall_force"], rtol=1e-13, atol=0)
        ca, cb = a.contacts(), b.contacts()
        for k in ("pairs", "colour", "impulse"):
            assert np.array_equal(ca[k], cb[k]), k
        xa, xb = a.state(), b.state()
        for k in ("x", "v", "w"):
            assert np.array_equal(xa[k], xb[k]), k


def test_batch_of_sphere_gases_is_bit_identical():
    batch = [W.sphere_gas(seed=b, n=300 + 900 * b, floor=16.0, vsig=0.5) for b in range(4)]
    a = gpu_system(batch[0], batch=batch, sweep_threads=256, sweep_blocks_per_sm=2)
    b = gpu_system(batch[0], batch=batch)
    for _ in range(3):
        assert a.step(1)["total_sweeps"] == b.step(1)["total_sweeps"]
    ca, cb = a.contacts(), b.contacts()
    for k in ca:
        assert np.array_equal(ca[k], cb[k]), k
    xa, xb = a.state(), b.state()
    for k in ("x", "v", "w"):
        assert np.array_equal(xa[k], xb[k]), k


def test_residual_magnitudes_match_64_bits():
    """R_avg against the mean of sqrt(P_n^2 + P_t^2) of the impulses, for
    magnitudes over many decades (the masses scale the impulses): within the
    rounding of the integer root (7.3e-15 a contact) and of the sum."""
    for scale in (1e-30, 1e-3, 1.0, 1e25):
        wl = W.dense_biaxial_discs(seed=4, n=3000)
        wl.inv_m, wl.inv_I = wl.inv_m / scale, wl.inv_I / scale
        g = gpu_system(wl, criterion=-1, max_sweeps=200)
        r = g.step(1)["last"]["r_avg"]
        P = g.contacts()["impulse"].astype(np.longdouble)
        exact = np.sqrt((P * P).sum(1)).mean()
        assert abs(np.longdouble(r) - exact) <= 2e-14 * exact


# a particle with two records, corners with four (eight in 3D), and cuts so
# fine that most particles have several
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("make,domains", [
    (lambda: W.dense_biaxial_discs(seed=5, n=40), (2, 1, 1)),
    (lambda: W.dense_biaxial_discs(seed=5, n=4999), (4, 2, 1)),
    (lambda: W.dense_biaxial_discs(seed=5, n=20011), (70, 70, 1)),
    (lambda: W.sphere_gas(seed=3, n=4000, floor=20.0, vsig=0.5), (3, 2, 5)),
])
def test_domains_are_bit_identical(make, domains, precision):
    """The domain-wise update, also of short solves (a sweep's tests against
    the ones started ahead: sweeps 1, 17 and 40), against the barrier schedule,
    which another block shape keeps."""
    wl = make()
    for kw in (dict(criterion=-1, max_sweeps=1), dict(criterion=-1, max_sweeps=17), dict(alpha=1e-2, max_sweeps=400),
               dict(alpha=1e-5, max_sweeps=40)):
        kw.update(precision=precision, domains=domains, max_contacts=4 * wl.n + 64)
        a = gpu_system(wl, sweep_threads=256, sweep_blocks_per_sm=2, **kw)
        b = gpu_system(wl, **kw)
        for _ in range(2):
            x, y = a.step(1)["last"], b.step(1)["last"]
            for k in ("sweeps", "converged", "n_contacts", "n_colours"):
                assert x[k] == y[k], k
            assert abs(x["r_avg"] - y["r_avg"]) <= 1e-13 * x["r_avg"]
        ca, cb = a.contacts(), b.contacts()
        for k in ("pairs", "colour", "impulse"):
            assert np.array_equal(ca[k], cb[k]), k
        xa, xb = a.state(), b.state()
        for k in ("x", "v", "w"):
            assert np.array_equal(xa[k], xb[k]), k


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("value", [0.0, 3e38, np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("dim", [2, 3])
def test_open_contacts_next_to_a_wild_velocity(dim, value, precision):
    """Items whose contacts are all open and stay so are passed by; one with an
    infinite or undefined rate is not."""
    wl = (W.settling_discs(seed=2, n=40000, vsig=0.1) if dim == 2 else
          W.sphere_gas(seed=2, n=20000, floor=40.0, vsig=0.1))
    kw = dict(precision=precision, criterion=-1, max_sweeps=131, max_contacts=4 * wl.n)
    a, b = gpu_system(wl, merge_last_colour=1, **kw), gpu_system(wl, **kw)
    for s in (a, b):
        s.detect_contacts()
        s.vel.reshape(wl.n, dim)[::977] = value
        s.solve_contacts()
    ca, cb = a.contacts(), b.contacts()
    assert len(ca["impulse"]) > 1000
    assert np.array_equal(ca["impulse"], cb["impulse"], equal_nan=True)
    xa, xb = a.state(), b.state()
    for k in ("v", "w"):
        assert np.array_equal(xa[k], xb[k], equal_nan=True), k


@pytest.mark.parametrize("count", [100, 230])
def test_batches_of_many_colours_are_bit_identical(count):
    """A large disc among small ones: more than 16 colours.  230 packings
    (5,000,000 contacts) are then left to the barrier schedule, 100 are not."""
    wl = W.dense_biaxial_discs(seed=3, n=10000)
    wl.r[5000] = 6.0
    kw = dict(batch=[wl] * count, alpha=1e-6, max_sweeps=30, max_contacts=24000 * count)
    a = gpu_system(wl, sweep_threads=256, sweep_blocks_per_sm=2, **kw)
    b = gpu_system(wl, **kw)
    sa, sb = a.step(1), b.step(1)
    assert sb["last"]["n_colours"] > 16 and (sb["last"]["n_contacts"] > 30000 * 152) == (count == 230)
    for k in ("total_sweeps", "total_contact_updates", "max_sweeps_in_step", "n_not_converged"):
        assert sa[k] == sb[k], k
    ca, cb = a.contacts(), b.contacts()
    assert np.array_equal(ca["impulse"], cb["impulse"])
    xa, xb = a.state(), b.state()
    for k in ("x", "v", "w"):
        assert np.array_equal(xa[k], xb[k]), k
