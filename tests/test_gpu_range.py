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
