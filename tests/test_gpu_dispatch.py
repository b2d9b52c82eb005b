"""Both sides of the dispatch rules on sizes, against the oracle (needs a
GB300): grids, thread counts and passes that differ by size only."""
from __future__ import annotations

import os
import re

import numpy as np
import pytest

import oracle
from oracle import CLOCK, ISING, POTTS, XY
from test_gpu_parity import ANGLE_TOL, ang_diff, xy_borderline

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


def same_as_alone(sw, specs, seed, calls, config=None):
    """Every member of a batch against the same lattice advanced alone."""
    b = sw.sw_batch_create(specs[0][1])
    inb = [sw.sw_create(*s, seed + k) for k, s in enumerate(specs)]
    alone = [sw.sw_create(*s, seed + k) for k, s in enumerate(specs)]
    try:
        for h in inb:
            sw.sw_batch_add(b, h)
        if config:
            sw.sw_batch_set_config(b, *config)
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


def one_cta_sites(dim):
    """The library's largest lattice that runs whole in one CTA."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    text = open(os.path.join(root, "paper_1403_7560_gb300", "csrc", "sw_internal.h")).read()
    return int(re.search(rf"\bkSmallSites{dim}D = (\d+)", text).group(1))


TILED = {2: [(ISING, 2, 300, 2, 2.269185), (POTTS, 2, 131, 3, 1.0), (ISING, 2, 161, 2, 2.2), (POTTS, 2, 146, 17, 0.7),
             (POTTS, 2, 128, 4, 0.91)],
         3: [(ISING, 3, 40, 2, 4.4), (POTTS, 3, 27, 3, 1.8), (ISING, 3, 33, 2, 4.5), (POTTS, 3, 30, 17, 1.2),
             (POTTS, 3, 32, 4, 1.6)]}


@pytest.mark.parametrize("shape", [0, 1, 2])
@pytest.mark.parametrize("schedule", list(range(8)))
@pytest.mark.parametrize("dim", [2, 3])
def test_tiled_members_of_both_models_in_every_configuration(sw, dim, shape, schedule):
    """Every tile shape, label layout (apart and combined), grid form and merge
    form, on tiled members of both models with L a multiple of 4 or not."""
    specs = TILED[dim]
    assert all(s[2] ** dim > one_cta_sites(dim) for s in specs)
    for model in (ISING, POTTS):
        assert {s[2] % 4 == 0 for s in specs if s[0] == model} == {True, False}
    same_as_alone(sw, specs, 4100, (3, 2), config=(shape, schedule))


@pytest.mark.parametrize("dim,L", [
    # fewer blocks of 32 x 128 (2D) or 32 x 16 x 8 sites than SMs: four sets of warps a block
    (2, 90), (2, 256), (3, 33), (3, 64),
    # more: one set, whole and ragged blocks
    (2, 1000), (2, 1001), (3, 97), (3, 128)])
def test_xy_bonds_on_both_sides_of_the_split(sw, dim, L):
    """The bond kernel that measures the state before (sweep 2), and the one
    that does not (sweep 3)."""
    T, seed, N = 0.89 if dim == 2 else 2.2, 61 + L, L ** dim
    h, first = sw.sw_create(XY, dim, L, 2, T, seed), sw.sw_create(XY, dim, L, 2, T, seed)
    try:
        sw.sw_sweep(first, 1)
        theta = sw.sw_get_spins(first)
        ref = oracle.moments(XY, dim, L, 2, theta)
        sw.sw_sweep(h, 2)
        mismatches = 0
        for k in (2, 3):
            if k == 3:
                sw.sw_discard(h, 1)
            mask, labels, new = sw.sw_get_bonds(h), sw.sw_get_labels(h), sw.sw_get_spins(h)
            mismatches += xy_borderline(T, dim, L, seed, k, theta, mask, oracle.bonds(XY, dim, L, 2, T, seed, k, theta))
            assert np.array_equal(labels, oracle.labels(dim, L, mask)), k
            assert ang_diff(new, oracle.flip(XY, dim, L, 2, seed, k, labels, theta)[0]).max() < ANGLE_TOL, k
            theta = new
        assert mismatches <= max(2, N * dim * 2 // 100000)
        # sums of N float terms of a few 1e-7 each
        rec, tol = sw.sw_get_series(h, 1, 1)[0], 2e-6 * N * (dim + 1) + 1e-3
        assert all(abs(rec[f] - ref[f]) < tol for f in ("mx", "my", "e_xy"))
    finally:
        sw.sw_destroy(h)
        sw.sw_destroy(first)
