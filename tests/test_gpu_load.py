"""Networks read from and written to the caller's device arrays where they lie
(needs a GB300): any row length and base address, against the host path bit
for bit, Z-scored and as given; state in and out around an iteration."""
from __future__ import annotations

import numpy as np
import pytest

import gpu_helpers as gh
from paper_1507_07039_gb300 import synth

pytestmark = pytest.mark.gpu


def _unaligned(x):
    """The array on the GPU, its first element 4 bytes past a 16-byte boundary."""
    import torch
    buf = torch.empty(x.size + 1, device="cuda")
    v = buf[1:].view(x.shape)
    v.copy_(torch.from_numpy(x))
    assert v.data_ptr() % 16 == 4 and v.is_contiguous()
    return v


@pytest.mark.parametrize("prec", [0, 1, 2, 3])
@pytest.mark.parametrize("T,G", [(3, 31), (64, 65), (130, 259)])
def test_device_arrays_of_any_alignment(T, G, prec):
    import torch
    from paper_1507_07039_gb300 import panda
    nets = synth.make_inputs(synth.custom(T, G, 9000 + T + G, n_samples=30, n_factors=3))
    dev = [_unaligned(x) for x in nets]
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    for norm in (True, False):
        with panda.PandaContext(*nets, prec=prec, normalize=norm) as h, \
                panda.PandaContext(*dev, prec=prec, normalize=norm, device=True, stream=s.cuda_stream) as d:
            for ctx in (h, d):
                ctx.run(0.1, 0.0, 2)
            ref = h.get()
            out = [_unaligned(np.zeros_like(x)) for x in nets]
            torch.cuda.synchronize()
            panda.panda_get_device(d.h, *out)
            for a, b in zip(ref, out):
                assert np.array_equal(a, b.cpu().numpy())
            # back to the start from either kind of array: the same bits again
            panda.panda_set_state(h.h, *ref, 2)
            panda.panda_set_state_device(d.h, *out, 2)
            for ctx in (h, d):
                ctx.run(0.1, 0.0, 2)
            for a, b in zip(h.get(), d.get()):
                assert np.array_equal(a, b)
    bad = nets[2].copy()
    bad[G - 1, 0] += 0.5
    with pytest.raises(panda.PandaError) as e:
        panda.PandaContext(dev[0], dev[1], _unaligned(bad), prec=prec, device=True, stream=s.cuda_stream)
    assert e.value.code == -5
