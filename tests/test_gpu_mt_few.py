"""MT19937 fills of few streams (a block per stream) and of the first count
that takes a warp per stream: whole and part blocks of 624 words, continued.
Bit for bit against the oracle."""
import numpy as np
import pytest

import oracle as O
import paper_1307_5869_gb300 as P

pytestmark = pytest.mark.gpu

BITS = {"u32": np.uint32, "f32": np.uint32, "f64": np.uint64}


@pytest.mark.parametrize("more", [None, 0, 1])
def test_fills(more):
    import torch
    n = 3 if more is None else 6 * torch.cuda.get_device_properties(0).multi_processor_count + more
    g, sample = P.Generator("MT19937", 4, 7, n), [0, n // 2, n - 1]
    ref = [O.State.stream("MT19937", 4, 7 + j) for j in sample]
    for per, dt in ((1, "u32"), (623, "f32"), (624, "f64"), (625, "u32"), (1, "f32"), (1249, "u32"), (3000, "f64")):
        got = g.generate(per, dt).reshape(n, per)
        for j, s in zip(sample, ref):
            want = {"u32": s.u32, "f32": s.f32, "f64": s.f64}[dt](per)
            assert np.array_equal(got[j].cpu().numpy().view(BITS[dt]), want.view(BITS[dt])), (per, dt, j)
    g.close()
