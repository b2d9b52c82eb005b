"""Both sides of the dispatch rules on sizes, against the oracle (needs a
GB300): grids, thread counts and passes that differ by size only."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from oracle import CLOCK

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
