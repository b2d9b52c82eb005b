"""The bond kernels' estimate of u - p against 64 bits (CPU): XY and clock.

Both kernels form near = (1 + u') + e - 2 in float, u' the uniform cut to 23
bits and e = ex2(kexp x) with kexp = -(2K log2 e) and x the product of two
projections, and let the exact form decide where |near| lies within a margin.
What near can be off by, with a = 2K x and one rounding r = 2^-24 relative:
  the cut                          2^-23
  log2 e as a float, its product with 2K, and that with x (three roundings of
  the exponent), and, for the clock, two rounded projections, their product
  and 2K (four more): n r a e <= n r / exp(1)               (a exp(-a) <= 1/e)
  the hardware ex2, 2^-22 e        <= 2^-22
  (1 + u') + e in [1, 3): at most 2^-23; the subtraction of 2 is exact
In all below 2^-23 + 2^-22 + 2^-23 + n 2^-24 / e < 5.5e-7 (XY, n = 3) and
< 6.4e-7 (clock, n = 7), 23 times inside the smallest margin, 2^-16."""
from __future__ import annotations

import math

import numpy as np
import pytest

ONE = np.uint32(0x3F800000)


def bound(n):
    return 2.0 ** -23 + 2.0 ** -22 + 2.0 ** -23 + n * 2.0 ** -24 / math.e


def estimate(twoK, prod, w):
    """near as the kernels form it (the ex2 rounded from 64 bits; its own error
    is added by the callers) and e in 64 bits."""
    kexp = -(np.float32(twoK) * np.float32(1.4426950))
    e = np.exp2((kexp * prod).astype(np.float32).astype(np.float64))
    one_u = (ONE | (w >> np.uint32(9))).view(np.float32)
    near = ((one_u + e.astype(np.float32)).astype(np.float32) - np.float32(2.0)).astype(np.float64)
    return near, e


@pytest.mark.parametrize("twoK", [0.04, 0.9083304, 13.0, 40.0, 1e4])
def test_xy_estimate(twoK):
    rng = np.random.default_rng(5)
    prod = np.concatenate([np.linspace(1e-7, 1.0, 200001), rng.random(100000) ** 8 + 1e-30]).astype(np.float32)
    twoK = np.float32(twoK)
    exact_p = -np.expm1(-(np.float64(twoK) * prod))
    for w in (rng.integers(0, 2 ** 32, prod.size, dtype=np.uint32), np.full(prod.size, 0xFFFFFFFF, np.uint32),
              np.zeros(prod.size, np.uint32)):
        near, e = estimate(twoK, prod, w)
        exact = (w >> np.uint32(8)).astype(np.float64) / 2 ** 24 - exact_p
        # ex2's error comes on top of the rounded e, which holds half an ulp of it already
        assert (np.abs(near - exact) + 2.0 ** -22 * e).max() <= bound(3) + 2.0 ** -25
    assert bound(3) + 2.0 ** -25 < 2.0 ** -16 / 23


@pytest.mark.parametrize("q", [2, 3, 6, 64, 512, 1024])
@pytest.mark.parametrize("T", [0.15, 0.5, 2.20184, 50.0])
def test_clock_estimate(q, T):
    """Every pair of states, each with a random uniform and one at the decision's
    edge; a float product that is not positive has a zero table entry."""
    x = np.sin((math.pi * np.arange(2 * q, dtype=np.float64)) / q)
    exact_prod = (x[:, None] * x[None, :]).reshape(-1)
    xf = x.astype(np.float32)
    prod = (xf[:, None] * xf[None, :]).reshape(-1)
    table = np.where(exact_prod > 0, np.floor(-np.expm1(-(2.0 / T) * exact_prod) * 2.0 ** 32), 0.0)
    table = np.minimum(table, 2.0 ** 32 - 1)
    assert np.all(table[prod <= 0] == 0)
    pos = prod > 0
    prod, t = prod[pos], table[pos]
    twoK = np.float32(2.0 / T)
    margin = np.float32(2.0 ** -16) + np.float32(twoK * np.float32(2.0 ** -20))
    rng = np.random.default_rng(q)
    for w in (rng.integers(0, 2 ** 32, prod.size, dtype=np.uint32), t.astype(np.uint32)):
        near, e = estimate(twoK, prod, w)
        exact = (w.astype(np.float64) - t) / 2.0 ** 32
        # the table's floor (2^-32) besides
        most = bound(7) + 2.0 ** -25 + 2.0 ** -32
        assert (np.abs(near - exact) + 2.0 ** -22 * e).max() <= most
        decided = np.abs(near) > float(margin)
        assert np.array_equal(near[decided] < 0, w[decided] < t[decided])
        assert most < 2.0 ** -16 / 23
