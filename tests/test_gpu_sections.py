"""Streams split into sections, around the lines of the rules: LFSR113's
tabulated sections and those by bits, few and many streams, outputs off the
vectors; GQ58.3's splits between whole blocks per SM.  Against the oracle, with
continuation."""
import numpy as np
import pytest

import oracle as O
import paper_1307_5869_gb300 as P

pytestmark = pytest.mark.gpu

BITS = {"u32": np.uint32, "f32": np.uint32, "f64": np.uint64}


def _fill(gen, n, calls, offset):
    import torch
    g, ref = P.Generator(gen, 17, 2, n), O.Streams(gen, 17, 2, n)
    for per, dt in calls:
        tdt = {"u32": torch.int32, "f32": torch.float32, "f64": torch.float64}[dt]
        flat = torch.zeros(n * per + offset + 8, dtype=tdt, device="cuda")
        g.generate(per, dt, out=flat[offset:offset + n * per])
        got = flat.cpu().numpy().view(BITS[dt])
        assert np.array_equal(got[offset:offset + n * per].reshape(n, per), ref.generate(dt, per).view(BITS[dt])), (gen, n, per, dt)
        assert not got[:offset].any() and not got[offset + n * per:].any()
    g.close()


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("n", [1, 7, 8, 31, 32, 33, 300])
def test_lfsr113_sections(n, offset):
    _fill("LFSR113", n, [(64, "u32"), (320, "f64"), (777, "u32"), (1024, "f32"), (1025, "u32"), (1821, "f64"), (2560, "f64"),
                         (2561, "u32"), (5120, "u32"), (5121, "f32")], offset)


@pytest.mark.parametrize("n,per", [(1, 255), (1, 512), (1, 100001), (50, 30000), (2500, 513)])
def test_gq58_3_sections(n, per):
    _fill("GQ58_3", n, [(per, "u32"), (per, "f64")], 0)
    _fill("GQ58_3", n, [(per, "f32")], 1)
