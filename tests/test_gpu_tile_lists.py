"""Phase 1 of the tensor-core modes where a CTA pair runs several tiles (needs
a GB300): the last K chunk of a tile that another one follows goes through the
running sum in memory, that of a pair's last tile straight from the tensor
memory.  Forty networks of four tiles each put more tiles on the 76 pairs than
there are pairs; alone, each network has one tile per pair.  Both must give the
same bits: the two ways add the same numbers in the same order."""
from __future__ import annotations

import numpy as np
import pytest

import gpu_helpers as gh
from paper_1507_07039_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [1, 2, 3])
@pytest.mark.parametrize("T,G", [(257, 300), (300, 2049), (260, 4200)])  # one chunk of genes, two, three
def test_tiles_that_follow_each_other(T, G, prec):
    from paper_1507_07039_gb300 import panda
    count = 40 if G < 2049 else 10  # (8 or more tiles each there)
    few = [synth.make_inputs(synth.custom(T, G, 8000 + G + k, n_samples=20, n_factors=3)) for k in range(2)]
    nets = [few[k % 2] for k in range(count)]
    with panda.PandaBatch(nets, prec=prec) as b:
        b.run(0.1, 0.0, 3)
        got = [b.get(k) for k in range(count)]
    for k in range(2):
        one = gh.gpu_run(*few[k], prec, 0.1, 0.0, 3)
        for n in range(k, count, 2):
            for x, y in zip((one["W"], one["P"], one["C"]), got[n]):
                assert np.array_equal(x, y), f"network {n}"
