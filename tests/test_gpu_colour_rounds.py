"""The colouring on both sides of the line from which it runs in rounds (more than
nine contacts a thread of the grid, 700,000 on 152 SMs, with three a body or more):
the oracle's greedy colouring and repair, contact for contact, by the one-kernel
preparation, the separate kernels and in a batch, whose packings have their own."""
import numpy as np
import pytest

import oracle as O
from gpu_common import gpu_system, needs_gpu
from paper_1104_3516_gb300 import workloads as W

pytestmark = [pytest.mark.gpu, needs_gpu]


def squeezed(n, spacing, seed=4):
    """n discs on a jittered lattice: 16 contacts each at spacing 1, 4 at 1.9."""
    k = int(np.ceil(np.sqrt(n)))
    x = np.stack(np.meshgrid(np.arange(k), np.arange(k), indexing="ij"), -1).reshape(-1, 2)[:n] * spacing + 1.5
    x = x + W.normal(seed, 2 * n, 0.05).reshape(n, 2)
    r = W.uniform(seed, n, 0.8, 1.2)
    inv_m, inv_I = W.masses(2, r)
    return W.Workload(name="squeezed", dim=2, x=x, v=np.zeros((n, 2)), w=np.zeros(n), r=r, inv_m=inv_m, inv_I=inv_I,
                      box_hi=(k * spacing + 3.0, k * spacing + 3.0, 1.0), wall_mask=0b0100, seed=seed)


def check(pairs, colour, n, seed, want):
    assert (len(pairs) > 700416) == want
    ref, K = O.colour_greedy(n, pairs, seed)
    assert np.array_equal(colour, ref)


@pytest.mark.parametrize("n, spacing, rounds", [(80000, 1.0, False), (100000, 1.0, True), (420000, 1.9, True)])
@pytest.mark.parametrize("timing", [0, 1])
def test_plain_systems(n, spacing, rounds, timing):
    wl = squeezed(n, spacing)
    g = gpu_system(wl, timing=timing, max_contacts=10 * n)
    g.detect_contacts()
    c = g.contacts()
    check(c["pairs"], c["colour"], n, wl.seed, rounds)


def test_a_batch():
    from test_gpu_batch import split
    packs = [squeezed(n, 1.0, seed=s) for n, s in ((60000, 4), (300, 5), (45000, 6))]
    total = sum(p.n for p in packs)
    g = gpu_system(packs[0], batch=packs, max_contacts=10 * total)
    g.detect_contacts()
    c = g.contacts()
    assert len(c["pairs"]) > 700416
    for wl, part in zip(packs, split(c, g.offsets, len(packs), total)):
        assert np.array_equal(part["colour"], O.colour_greedy(wl.n, part["pairs"], wl.seed)[0])
