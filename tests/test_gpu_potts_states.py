"""Potts lattices of many states: the record's histogram is summed over fewer
slots the more states there are (needs a GB300)."""
from __future__ import annotations

import math
import time

import numpy as np
import pytest

import oracle
from oracle import POTTS

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sw():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1403_7560_gb300 import build, sw as swmod
    build.build()
    return swmod


def same_records(sw, h, o, first, recs):
    for r, ref in zip(sw.sw_get_series(h, first, len(recs)), recs):
        assert all(r[f] == ref[f] for f in ref if f in r), (r, ref)
    got, ref = sw.sw_measure(h), o.take_acc()
    assert all(got[f] == ref[f] for f in ref)
    assert np.array_equal(sw.sw_get_spins(h), o.spins)


# the numbers of states at which the slots halve, and one more
@pytest.mark.parametrize("q", [2, 8, 9, 16, 17, 32, 33, 64, 65, 128, 129, 256])
@pytest.mark.parametrize("dim,L", [(2, 130), (3, 26)])
def test_records_at_every_slot_count(sw, dim, L, q):
    T = 1 / math.log(1 + math.sqrt(q))
    h, o = sw.sw_create(POTTS, dim, L, q, T, 9 + q), oracle.Oracle(POTTS, dim, L, q, T, 9 + q)
    try:
        sw.sw_sweep(h, 3)
        recs = []
        for _ in range(3):
            o.sweep(1)
            recs.append(o.last_record())
        same_records(sw, h, o, 1, recs)
    finally:
        sw.sw_destroy(h)
        o.close()


@pytest.mark.parametrize("dim,L", [(2, 130), (3, 26)])
def test_batch_records_at_every_slot_count(sw, dim, L):
    """A call whose last records stay pending, then one that measures them."""
    b = sw.sw_batch_create(dim)
    spec = [(POTTS, dim, L, q, 1 / math.log(1 + math.sqrt(q)), 40 + q) for q in (3, 8, 9, 17, 33, 65, 129, 256)]
    hs, os_ = [sw.sw_create(*s) for s in spec], [oracle.Oracle(*s) for s in spec]
    try:
        for h in hs:
            sw.sw_batch_add(b, h)
        sw.sw_batch_sweep(b, 2)
        sw.sw_batch_sweep(b, 16)
        for h, o in zip(hs, os_):
            recs = []
            for _ in range(18):
                o.sweep(1)
                recs.append(o.last_record())
            same_records(sw, h, o, 1, recs)
    finally:
        sw.sw_batch_destroy(b)
        for h in hs:
            sw.sw_destroy(h)
        for o in os_:
            o.close()


def best_time(sw, run, sync, reps=6):
    best = math.inf
    for _ in range(reps):
        sync()
        t = time.perf_counter()
        run()
        sync()
        best = min(best, time.perf_counter() - t)
    return best


@pytest.mark.parametrize("batched", [False, True], ids=["alone", "batch"])
def test_many_states_cost_little_more_than_few(sw, batched):
    """The record of a sweep is written beside (alone) or before (batch) work of
    a few microseconds: summing 64 slots of 256 states there made a sweep 2.2
    (alone, 2D L = 2048) and 3.1 times (batch, L = 1024) as long as with 17
    states, whose lattice work is the same."""
    import torch
    L, n = (1024, 50) if batched else (2048, 50)
    times = []
    for q in (17, 256):
        h = sw.sw_create(POTTS, 2, L, q, 1 / math.log(1 + math.sqrt(q)), 3)
        b = sw.sw_batch_create(2)
        try:
            if batched:
                sw.sw_batch_add(b, h)
            run = (lambda: sw.sw_batch_sweep(b, n)) if batched else (lambda: sw.sw_sweep(h, n))
            run()
            times.append(best_time(sw, run, torch.cuda.synchronize))
        finally:
            sw.sw_batch_destroy(b)
            sw.sw_destroy(h)
    assert times[1] < 1.6 * times[0], times
