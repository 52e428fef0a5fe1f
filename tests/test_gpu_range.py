"""Networks of very small and very large entries (needs a GB300).

Eqs. 1-6 scale with the networks: all three times c give W', P' and C' times c.
With c a power of two every rounding scales too (FP32 and BF16 are binary, the
E4M3 scale is a power of two), so the results are the same to the bit as long
as nothing leaves the range of normal numbers."""
from __future__ import annotations

import numpy as np
import pytest

import gpu_helpers as gh

pytestmark = pytest.mark.gpu


def networks(T, G, seed=5):
    """Entries of about 1/4: squared norms of a few units at these sizes."""
    rng = np.random.default_rng(seed)
    nets = [rng.standard_normal((T, G)) / 4, gh.random_symmetric(rng, T) / 4, gh.random_symmetric(rng, G) / 4]
    return [x.astype(np.float32) for x in nets]


@pytest.mark.parametrize("prec", [1, 2, 3])
@pytest.mark.parametrize("T,G", [(40, 70), (300, 530)])  # edge blocks alone; whole blocks too
def test_small_networks_scale(T, G, prec):
    """Squared norms of about 1e-31 to 1e-30 and less, entries and products well
    inside the normal range (the smallest products are about 2^-120)."""
    nets = networks(T, G)
    one = gh.gpu_run(*nets, prec, 0.1, 0.0, 2, normalize=False)
    for k in (-20, -54):
        c = np.float32(2.0) ** k
        got = gh.gpu_run(*(x * c for x in nets), prec, 0.1, 0.0, 2, normalize=False)
        for n in ("W", "P", "C"):
            assert np.array_equal(got[n], one[n] * c), (n, k)


def close(got, one, c):
    """Each network within 1e-3 of its largest entry, P's and C's diagonals apart."""
    for n in ("W", "P", "C"):
        x, y = got[n].astype(np.float64) / float(c), one[n].astype(np.float64)
        if n != "W":
            d = np.diag(y)
            assert np.max(np.abs(np.diag(x) - d)) <= 1e-3 * np.max(np.abs(d)), n
            x, y = x - np.diag(np.diag(x)), y - np.diag(d)
        assert np.max(np.abs(x - y)) <= 1e-3 * np.max(np.abs(y)), n


def test_fp8mix_scales_whose_product_overflows():
    """Entries of about 2^-60: the E4M3 copies are scaled by 2^65 each, whose product
    is no float.  The scaled entries are the same bytes; what is lost is the BF16
    products' and squares' part below 2^-149, 2^-20 of them.  (With the product
    of the scales inverted, A and the new C were 0: 1e-1 of the largest entry.)"""
    nets = networks(40, 70)
    one = gh.gpu_run(*nets, 3, 0.1, 0.0, 2, normalize=False)
    c = np.float32(2.0) ** -58
    close(gh.gpu_run(*(x * c for x in nets), 3, 0.1, 0.0, 2, normalize=False), one, c)


@pytest.mark.parametrize("T,G", [(40, 70), (1024, 2048)])  # one CTA a tile; CTA pairs
def test_fp32_scales(T, G):
    """Where no part product leaves the normal range the bits are the same."""
    nets = networks(T, G)
    one = gh.gpu_run(*nets, 0, 0.1, 0.0, 2, normalize=False)
    for k in (-20, -48, 40):
        c = np.float32(2.0) ** k
        got = gh.gpu_run(*(x * c for x in nets), 0, 0.1, 0.0, 2, normalize=False)
        for n in ("W", "P", "C"):
            assert np.array_equal(got[n], one[n] * c), (n, k)


@pytest.mark.parametrize("k", [-64, -66])
def test_fp32_squared_norms_below_the_normal_range(k):
    """Entries of about 2^-66 and 2^-68 and less: their squares are subnormal, with a
    spacing of 2^-149, 2^-13 of a square; a sum of 40 to 70 of them and the square
    root of it are closer, about 2^-15.  Bound: 1e-3 of the largest entry of each
    network, against the run with entries of 1/4.  (Denominators held at the smallest
    normal float are 5 times too large at k = -65.)"""
    nets = networks(40, 70)
    one = gh.gpu_run(*nets, 0, 0.1, 0.0, 1, normalize=False)
    c = np.float32(2.0) ** k
    close(gh.gpu_run(*(x * c for x in nets), 0, 0.1, 0.0, 1, normalize=False), one, c)


def test_fp32_squared_norms_near_the_largest_float():
    """A denominator of 3.2e38, all its parts finite: R within FP32 rounding of Eq. 1
    (an FP64 evaluation), at alpha = 1, where W' is (R + A) / 2."""
    p, w1 = 1.30e19, 1.15e18
    w2 = np.sqrt(1.65e38 - w1 * w1)
    W = np.array([[w1], [w2]], np.float32)
    P, C = np.diag([p, p]).astype(np.float32), np.ones((1, 1), np.float32)
    got = gh.gpu_run(W, P, C, 0, 1.0, 0.0, 1, normalize=False)["W"].astype(np.float64)
    W, P, C = (x.astype(np.float64) for x in (W, P, C))

    def tan(x, y):
        return x @ y / np.sqrt(x @ x + y @ y - abs(x @ y))

    want = np.array([[(tan(P[i], W[:, 0]) + tan(W[i], C[0])) / 2] for i in range(2)])
    assert (P[0] @ P[0] + W[:, 0] @ W[:, 0] - P[0] @ W[:, 0]) > 3.1e38
    assert np.max(np.abs(got / want - 1.0)) <= 1e-6
