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
