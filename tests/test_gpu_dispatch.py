"""Both sides of the dispatch rules on sizes, against the oracle (needs a
GB300): grids, thread counts and passes that differ by size only."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from oracle import CLOCK, ISING, POTTS

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sw():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1403_7560_gb300 import build, sw as swmod
    build.build()
    return swmod


@pytest.mark.parametrize("dim,L,q", [
    # row words: one wave of CTAs up to 98304 of them, then 4096 CTAs; above
    # 2^20 sites the flip has a compression (N mod 4 = 0, 1, 0, 3, 1)
    (2, 1024, 512), (2, 1025, 6), (3, 102, 37), (3, 139, 6), (2, 2005, 512)])
def test_clock_sweeps_on_both_sides_of_the_grid_rule(sw, dim, L, q):
    T = 0.9 if dim == 2 else 2.2
    h, o = sw.sw_create(CLOCK, dim, L, q, T, 21 + L), oracle.Oracle(CLOCK, dim, L, q, T, 21 + L)
    try:
        sw.sw_sweep(h, 2)
        sw.sw_discard(h, 1)
        o.sweep(2)
        o.sweep(1, measure=False)
        assert np.array_equal(sw.sw_get_bonds(h), o.planes)
        assert np.array_equal(sw.sw_get_labels(h), o.labels)
        assert np.array_equal(sw.sw_get_spins(h), o.spins)
        got, ref = sw.sw_measure(h), o.take_acc()
        assert all(got[f] == ref[f] for f in ref)
    finally:
        sw.sw_destroy(h)
        o.close()


def same_as_alone(sw, specs, seed, calls):
    """Every member of a batch against the same lattice advanced alone."""
    b = sw.sw_batch_create(specs[0][1])
    inb = [sw.sw_create(*s, seed + k) for k, s in enumerate(specs)]
    alone = [sw.sw_create(*s, seed + k) for k, s in enumerate(specs)]
    try:
        for h in inb:
            sw.sw_batch_add(b, h)
        for n in calls:
            sw.sw_batch_sweep(b, n)
        total = sum(calls)
        for x, y in zip(inb, alone):
            sw.sw_sweep(y, total)
            assert np.array_equal(sw.sw_get_spins(x), sw.sw_get_spins(y))
            assert np.array_equal(sw.sw_get_labels(x), sw.sw_get_labels(y))
            assert sw.sw_get_series(x, 1, total) == sw.sw_get_series(y, 1, total)
            mx, my = sw.sw_measure(x), sw.sw_measure(y)
            assert all(mx[f] == my[f] for f in mx)
    finally:
        sw.sw_batch_destroy(b)
        for h in inb + alone:
            sw.sw_destroy(h)


@pytest.mark.parametrize("dim,large", [(2, None), (2, 112), (3, None), (3, 22)])
def test_more_small_members_than_sms(sw, dim, large):
    """One-CTA members by the pair on an SM, and one to an SM where the largest
    leaves no room for two."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(31 + dim)
    specs = []
    for k in range(sms + 9):
        L = int(rng.integers(4, 60 if dim == 2 else 17))
        model, q = ((ISING, 2), (POTTS, 2), (POTTS, 3), (POTTS, 5))[k % 4]
        specs.append((model, dim, L, q, 2.3 if model == ISING and dim == 2 else 4.5 if model == ISING else 0.9))
    if large:
        specs[5] = (ISING, dim, large, 2, 2.3 if dim == 2 else 4.5)
        specs[6] = (POTTS, dim, large, 3, 1.0 if dim == 2 else 1.8)
    same_as_alone(sw, specs, 3000, (3, 2))
