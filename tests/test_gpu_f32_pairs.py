"""The FP32 path's 256 x 256 tiles on CTA pairs (needs a GB300), in every kernel
that has them: phase 1 and phase 2 with whole and cut tiles, under rule D2 too,
which keeps a third sum and stages fewer rows, and with both padded sizes an odd
multiple of 128, where the second CTA of the last tile lies past the array.  The
plan is asked which tiles a case runs.

Tolerance: gpu_helpers.TOL[0], the FP32 path's."""
from __future__ import annotations

import os

import numpy as np
import pytest

import gpu_helpers as gh
from oracle.oracle import Oracle
from paper_1507_07039_gb300 import synth

pytestmark = pytest.mark.gpu

# cut tiles on 152 SMs, phases 1 and 2: some in both (1024 x 2048, 1100 x 2100, 500 x 4000), none (2000 x 2000)
CASES = [(1024, 2048, True), (1100, 2100, True), (500, 4000, True), (2000, 2000, False)]


@pytest.mark.parametrize("diag", [0, 2])
@pytest.mark.parametrize("T,G,cut", CASES)
def test_pair_tiles(T, G, cut, diag):
    import torch
    from paper_1507_07039_gb300 import panda
    plan = panda.panda_fp32_plan(T, G, torch.cuda.get_device_properties(0).multi_processor_count)
    assert plan["pair"] and [c > 0 for c in plan["cuts"]] == [cut, cut], plan
    orc = Oracle()
    orc.set_threads(os.cpu_count() or 1)
    nets = synth.make_inputs(synth.custom(T, G, 6000 + T + G, n_samples=30, n_factors=3))
    o = gh.oracle_run(orc, *nets, 0.1, 0.0, 2, diag=diag)
    a = gh.gpu_run(*nets, 0, 0.1, 0.0, 2, diag=diag)
    gh.assert_parity(a, o, 0, f"{T}x{G} D{diag}")
    b = gh.gpu_run(*nets, 0, 0.1, 0.0, 2, diag=diag)
    for k in ("W", "P", "C"):
        assert np.array_equal(a[k], b[k]), k
