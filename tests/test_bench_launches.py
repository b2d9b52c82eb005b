"""The launch counts that bench.py reports for a batch call (CPU)."""
from __future__ import annotations

import os
import re
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
ISING, POTTS = 0, 1
TILED = [(ISING, 2, 113, 2, 2.0, 1), (POTTS, 2, 512, 3, 1.0, 2)]
SMALL = [(ISING, 2, 112, 2, 2.0, 3), (POTTS, 2, 64, 4, 0.9, 4)]


@pytest.mark.parametrize("sweeps", [1, 15, 16, 256, 257])
def test_launches_of_a_batch_call(sweeps):
    import bench
    last = 1 if sweeps >= 16 else 0
    chunks = 1 if sweeps <= 256 else 2
    # labels of two models, merge, compression, apply, step counter
    assert bench.batch_call_launches(TILED, 0, sweeps) == 6 * sweeps + last
    assert bench.batch_call_launches(TILED, 5, sweeps) == 6 * sweeps + last  # one label launch, a merge per axis
    assert bench.batch_call_launches(SMALL, 0, sweeps) == chunks
    assert bench.batch_call_launches(TILED + SMALL, 0, sweeps) == 6 * sweeps + last + chunks
    assert bench.batch_call_launches([(ISING, 3, 22, 2, 4.5, 5)], 0, sweeps) == chunks
    assert bench.batch_call_launches([(ISING, 3, 23, 2, 4.5, 5)], 0, sweeps) == 5 * sweeps + last


def test_the_rules_are_the_library_s():
    import bench
    csrc = os.path.join(ROOT, "paper_1403_7560_gb300", "csrc")
    text = "".join(open(os.path.join(csrc, f)).read() for f in ("sw_internal.h", "sw_batch.cu"))
    value = lambda name: int(re.search(rf"\b{name} = (\d+)", text).group(1))
    assert bench.SMALL_SITES == {2: value("kSmallSites2D"), 3: value("kSmallSites3D")}
    assert bench.SMALL_CHUNK == value("kSmallChunk")
    assert bench.MEASURE_AFTER == value("kMeasureAfter")
