"""The damped updates of Eqs. 2 and 5 in FP32 at large alpha (needs a GB300): at
alpha = 1 the new entries replace the old ones and nothing of the old ones'
size is left in them.

Tolerance: gpu_helpers.TOL[0] (W 1e-5; off-diagonals 2e-5 of the new network's
scale; diagonals 2e-5 relative).  The new entries are similarities of order 1
to 10 whatever the old ones were, since one of the two vectors is of that size
(Eq. 1 is at most the geometric mean of the norms, and the large networks
multiply the denominator as they do the numerator); an old entry of 1e4 rounds
at 5e-4, fifty times the bound."""
from __future__ import annotations

import os

import numpy as np
import pytest

import gpu_helpers as gh
from oracle.oracle import Oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,G", [(40, 70), (130, 300)])
@pytest.mark.parametrize("alpha,large", [(1.0, "W"), (1.0, "PC"), (1.0, ""), (0.9, ""), (0.5, "")])
def test_large_alpha(T, G, alpha, large):
    rng = np.random.default_rng(T + G)
    W = rng.standard_normal((T, G)).astype(np.float32)
    P, C = gh.random_symmetric(rng, T), gh.random_symmetric(rng, G)
    if large == "W":
        W *= np.float32(1e4)
    elif large == "PC":
        P, C = P * np.float32(1e4), C * np.float32(1e4)
    orc = Oracle()
    orc.set_threads(os.cpu_count() or 1)
    o = gh.oracle_run(orc, W, P, C, alpha, 0.0, 1, normalize=False)
    a = gh.gpu_run(W, P, C, 0, alpha, 0.0, 1, normalize=False)
    gh.assert_parity(a, o, 0, f"{T}x{G} alpha {alpha} {large}")
