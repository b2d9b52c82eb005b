"""The bond kernels' fast estimate against 64 bits (CPU)."""
from __future__ import annotations

import numpy as np
import pytest


@pytest.mark.parametrize("twoK", [0.04, 0.9083304, 13.0, 40.0])
def test_xy_bond_estimate_within_its_margin(twoK):
    """The XY and clock bond kernels decide from (1 + u) + 2^(-2K log2(e) x) - 2
    with u cut to 23 bits: against 64 bits the estimate of u - p is off by the
    cut (2^-23), the hardware exp (2^-22 relative), its argument's rounding and
    two additions below 2 (2^-24 each), far inside the 2^-16 margin."""
    rng = np.random.default_rng(3)
    prod = np.concatenate([np.linspace(1e-7, 1.0, 200001), rng.random(200000)]).astype(np.float32)
    w = rng.integers(0, 2 ** 32, prod.size, dtype=np.uint64)
    kexp = -(np.float32(twoK) * np.float32(1.4426950))
    e = np.exp2((kexp * prod).astype(np.float32).astype(np.float64))
    one_u = (np.uint32(0x3F800000) | (w >> np.uint64(9)).astype(np.uint32)).view(np.float32)
    near = ((one_u + e.astype(np.float32)).astype(np.float32) - np.float32(2.0)).astype(np.float64)
    exact = (w >> np.uint64(8)).astype(np.float64) / 2 ** 24 + np.expm1(-np.float64(np.float32(twoK)) * prod)
    assert (np.abs(near - exact) + 2.0 ** -22 * e).max() < 2.0 ** -16 / 8
