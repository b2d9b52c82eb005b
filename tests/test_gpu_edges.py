"""Sizes at which the kernels' branches change (edges of words, rows and
tiles, lattices no longer than a tile), against the oracle (needs a GB300)."""
from __future__ import annotations

import numpy as np
import pytest

import inputs
import oracle
from oracle import ISING, POTTS

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sw():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1403_7560_gb300 import build, sw as swmod
    build.build()
    return swmod


@pytest.mark.parametrize("dim,L", [(2, L) for L in (4, 5, 31, 32, 36, 63, 127, 128, 129, 132, 257)]
                         + [(3, L) for L in (4, 5, 8, 15, 16, 17, 20, 33, 36)])
def test_tile_labels_at_tile_edges(sw, dim, L):
    """Hooked runs, unions around the torus inside a tile, and both forest
    layouts of the last phase (L a multiple of 4 or not)."""
    h = sw.sw_create(ISING, dim, L, 2, 2.0, 1)
    try:
        for density in (0.15, 0.25, 0.5, 0.9):
            m = inputs.random_mask(dim, L, density, seed=7 * L + int(100 * density))
            assert np.array_equal(sw.sw_label_from_bonds(h, m), oracle.labels(dim, L, m)), density
    finally:
        sw.sw_destroy(h)


@pytest.mark.parametrize("model,dim,L,q", [
    (ISING, 2, 4, 2), (ISING, 2, 5, 2), (ISING, 2, 31, 2), (ISING, 2, 32, 2), (ISING, 2, 33, 2), (ISING, 2, 65, 2),
    (ISING, 2, 90, 2), (ISING, 3, 4, 2), (ISING, 3, 7, 2), (ISING, 3, 16, 2),
    (POTTS, 2, 6, 2), (POTTS, 2, 33, 3), (POTTS, 2, 90, 5), (POTTS, 2, 64, 16), (POTTS, 2, 37, 17),
    (POTTS, 2, 90, 256), (POTTS, 3, 5, 4), (POTTS, 3, 16, 3)])
def test_one_cta_sweeps(sw, model, dim, L, q):
    """Whole sweeps in shared memory: calls longer than the record ring (64
    sweeps), bonds, labels, states, records and accumulators."""
    T = 2.3 if model == ISING and dim == 2 else 4.5 if model == ISING else 0.9
    h = sw.sw_create(model, dim, L, q, T, 77 + L)
    o = oracle.Oracle(model, dim, L, q, T, 77 + L)
    try:
        sw.sw_sweep(h, 130)
        sw.sw_discard(h, 3)
        sw.sw_sweep(h, 64)
        recs = []
        for k in range(197):
            o.sweep(1, measure=not 130 <= k < 133)
            recs.append(o.last_record())
        assert np.array_equal(sw.sw_get_spins(h), o.spins)
        assert np.array_equal(sw.sw_get_bonds(h), o.planes)
        assert np.array_equal(sw.sw_get_labels(h), o.labels)
        for first, n in ((1, 130), (134, 64)):
            for r, ref in zip(sw.sw_get_series(h, first, n), recs[first - 1:]):
                assert all(r[f] == ref[f] for f in ref if f in r), (r, ref)
        got, ref = sw.sw_measure(h), o.take_acc()
        assert all(got[f] == ref[f] for f in ref)
    finally:
        sw.sw_destroy(h)
        o.close()


def test_small_members_over_several_launches(sw):
    """More sweeps in a batch call than one launch of the small members takes,
    with members that stop early, beside a tiled member."""
    spec = [(ISING, 2, 8, 2, 2.3, 1, 0), (POTTS, 2, 13, 3, 1.0, 2, 300), (ISING, 2, 33, 2, 2.2, 3, 10),
            (ISING, 2, 100, 2, 2.27, 4, 5)]
    b = sw.sw_batch_create(2)
    hs = [sw.sw_create(*s[:6]) for s in spec]
    try:
        for h, s in zip(hs, spec):
            sw.sw_batch_add(b, h)
            if s[6]:
                sw.sw_set_sweep_target(h, s[6])
        sw.sw_batch_sweep(b, 600)
        for h, s in zip(hs, spec):
            n = s[6] or 600
            o = oracle.Oracle(*s[:6])
            o.sweep(n)
            assert sw.sw_sweep_counter(h) == n
            assert np.array_equal(sw.sw_get_spins(h), o.spins)
            got, ref = sw.sw_measure(h), o.take_acc()
            assert all(got[f] == ref[f] for f in ref), s
            o.close()
    finally:
        sw.sw_batch_destroy(b)
        for h in hs:
            sw.sw_destroy(h)


@pytest.mark.parametrize("model,dim,L,q", [
    # four threads a row word: rows at every alignment, whole and half words
    (ISING, 2, 113, 2), (ISING, 2, 114, 2), (POTTS, 2, 115, 5), (ISING, 2, 144, 2), (POTTS, 2, 176, 17),
    (ISING, 3, 23, 2), (POTTS, 3, 26, 4), (ISING, 3, 48, 2),
    # two
    (POTTS, 2, 1185, 3), (ISING, 3, 99, 2), (POTTS, 3, 100, 3),
    # one
    (ISING, 2, 1801, 2), (POTTS, 3, 161, 3)])
def test_tiled_sweeps_split_and_ragged(sw, model, dim, L, q):
    T = 2.27 if model == ISING and dim == 2 else 4.5 if model == ISING else 0.95 if dim == 2 else 1.8
    h = sw.sw_create(model, dim, L, q, T, 5 + L)
    o = oracle.Oracle(model, dim, L, q, T, 5 + L)
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


@pytest.mark.parametrize("model,dim,L,q", [
    # one tile (no merge), tiles merged and walked without a compression, the
    # last size that walks and the first that does not
    (oracle.CLOCK, 2, 32, 37), (oracle.CLOCK, 3, 16, 512), (oracle.CLOCK, 2, 33, 6), (ISING, 2, 1024, 2),
    (ISING, 2, 1025, 2), (POTTS, 3, 101, 3), (POTTS, 3, 102, 3)])
def test_flip_paths(sw, model, dim, L, q):
    T = 2.27 if model == ISING else 0.9 if model == oracle.CLOCK and dim == 2 else 2.2 if model == oracle.CLOCK else 1.8
    h = sw.sw_create(model, dim, L, q, T, 11 + L)
    o = oracle.Oracle(model, dim, L, q, T, 11 + L)
    try:
        sw.sw_sweep(h, 3)
        o.sweep(3)
        assert np.array_equal(sw.sw_get_labels(h), o.labels)
        assert np.array_equal(sw.sw_get_spins(h), o.spins)
        got, ref = sw.sw_measure(h), o.take_acc()
        assert all(got[f] == ref[f] for f in ref)
    finally:
        sw.sw_destroy(h)
        o.close()


@pytest.mark.parametrize("dim,shape", [(2, 0), (2, 1), (2, 2), (3, 0), (3, 1), (3, 2)])
def test_batch_records_measured_together(sw, dim, shape):
    """A call of many sweeps measures its members' last records in one launch
    (rows at every alignment, q on both sides of the per-warp histogram), and
    a short call leaves them to the next one."""
    spec = [(ISING, dim, 120 if dim == 2 else 24, 2, 2.3 if dim == 2 else 4.5, 1),
            (POTTS, dim, 131 if dim == 2 else 27, 3, 1.0, 2), (POTTS, dim, 146 if dim == 2 else 30, 17, 0.7, 3),
            (ISING, dim, 161 if dim == 2 else 33, 2, 2.2 if dim == 2 else 4.4, 4)]
    b = sw.sw_batch_create(dim)
    hs = [sw.sw_create(*s) for s in spec]
    try:
        for h in hs:
            sw.sw_batch_add(b, h)
        sw.sw_batch_set_config(b, shape, 0)
        sw.sw_set_sweep_target(hs[3], 12)
        for n in (17, 3, 16):
            sw.sw_batch_sweep(b, n)
        for h, s in zip(hs, spec):
            n = 12 if h is hs[3] else 36
            o = oracle.Oracle(*s)
            o.sweep(n)
            assert sw.sw_sweep_counter(h) == n
            assert np.array_equal(sw.sw_get_spins(h), o.spins)
            ref, last = o.take_acc(), o.last_record()
            r = sw.sw_get_series(h, n, 1)[0]
            assert all(r[f] == last[f] for f in last if f in r), (r, last)
            got = sw.sw_measure(h)
            assert all(got[f] == ref[f] for f in ref), s
            o.close()
    finally:
        sw.sw_batch_destroy(b)
        for h in hs:
            sw.sw_destroy(h)


@pytest.mark.parametrize("dim,L", [(2, 7), (2, 64), (3, 9), (3, 32)])
@pytest.mark.parametrize("offset", [0, 1])
def test_labels_into_any_buffer(sw, dim, L, offset):
    """Canonical labels by four sites a thread, into a buffer that is or is
    not 16-byte aligned; N a multiple of 4 or not."""
    import torch
    m = inputs.random_mask(dim, L, 0.4, seed=L)
    dm = torch.from_numpy(m.view(np.int32).copy()).cuda()
    out = torch.full((L ** dim + 8,), -1, dtype=torch.int32, device="cuda")
    sw.sw_label_from_bonds_noalloc(dim, L, dm.data_ptr(), out.data_ptr() + 4 * offset,
                                   torch.cuda.current_stream().cuda_stream)
    got = out.cpu().numpy()
    assert np.array_equal(got[offset:offset + L ** dim], oracle.labels(dim, L, m))
    assert (got[offset + L ** dim:] == -1).all() and (got[:offset] == -1).all()
