"""How FP32's row sums are added up (needs a GB300): rows of one large square in
32 small ones, at the places where one thread of a CTA pair adds them.

At alpha = 0 an iteration leaves W as it is and computes its norms again in the
tile epilogue; a checkpoint holds them.  In every block of 128 columns the
columns 0, 4, 8 and 12 hold 1, the others 2^-12.5, whose square 2^-25 is lost when
it is added to a sum of 1 alone.  A thread adds 32 of a row's columns, one 1 among
them.  Four columns first, then the next four to them: three squares of 2^-25 are
lost, the other 28 arrive as seven sums of 2^-23, one unit in the last place of
1; the sums over threads are exact, the last rounding is 2^-24 at most.  Bound:
3 * 2^-25 + 2^-24 = 1.5e-7 of the sum; one chain of 32 loses 31 * 2^-25 = 9.2e-7."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_row_norms_of_w():
    import torch
    from paper_1507_07039_gb300 import panda
    T, G = 1024, 2048
    assert panda.panda_fp32_plan(T, G, torch.cuda.get_device_properties(0).multi_processor_count)["pair"]
    row = np.full(G, 2.0 ** -12.5, np.float32)
    for j in (0, 4, 8, 12):
        row[j::128] = 1.0
    W = np.tile(row, (T, 1))
    with panda.PandaContext(W, np.eye(T, dtype=np.float32), np.eye(G, dtype=np.float32), normalize=False) as ctx:
        ctx.run(0.0, 0.0, 1)
        blob = panda.panda_save(ctx.h)
        assert np.array_equal(ctx.get()[0], W)
    # header, W, P, C, the FP64 diagonals, |P_i.|^2, |C_.j|^2, then |W_i.|^2
    at = 36 + 4 * (T * G + T * T + G * G) + 8 * (T + G) + 4 * (T + G)
    got = np.frombuffer(blob, np.float32, T, at).astype(np.float64)
    want = np.sum(row.astype(np.float64) ** 2)
    assert np.max(np.abs(got / want - 1.0)) <= 1.5e-7
