"""The FP32 path's tiles (needs a GB300): networks whose tiles end inside,
at and just past a 128- or 256-edge, networks small enough that tiles are cut
along K and their parts' sums meet in memory, and the run-to-run bits.

Tolerance: gpu_helpers.TOL[0], the FP32 path's (W 1e-5; off-diagonals 2e-5 of
scale; diagonals 2e-5 relative), derived there for FP32 sums of K products
rounded one by one; the tile sums here round every 64 products."""
from __future__ import annotations

import os

import numpy as np
import pytest

import gpu_helpers as gh
from oracle.oracle import Oracle
from paper_1507_07039_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("diag", [0, 2])
@pytest.mark.parametrize("T,G", [(1, 130), (127, 129), (128, 256), (257, 255), (129, 1537), (520, 700)])
def test_tile_edges_and_cut_tiles(T, G, diag):
    from paper_1507_07039_gb300 import panda
    orc = Oracle()
    orc.set_threads(os.cpu_count() or 1)
    W0, P0, C0 = synth.make_inputs(synth.custom(T, G, 7000 + T + G, n_samples=30, n_factors=3))
    if T == 1:  # no spread to Z-score in a 1 x 1 network
        W0 = np.random.default_rng(T).standard_normal((T, G)).astype(np.float32)
    norm = T > 1
    o = gh.oracle_run(orc, W0, P0, C0, 0.1, 0.0, 3, normalize=norm, diag=diag)
    a = gh.gpu_run(W0, P0, C0, panda.PANDA_FP32, 0.1, 0.0, 3, normalize=norm, diag=diag)
    gh.assert_parity(a, o, 0, f"{T}x{G} D{diag}")
    b = gh.gpu_run(W0, P0, C0, panda.PANDA_FP32, 0.1, 0.0, 3, normalize=norm, diag=diag)
    for k in ("W", "P", "C"):  # which part of a cut tile comes last changes nothing
        assert np.array_equal(a[k], b[k]), k
