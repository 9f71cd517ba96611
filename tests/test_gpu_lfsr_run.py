"""LFSR113 rows of whole chunks, whose second component comes sixteen outputs at
a time: rows around a chunk (64 words, 32 doubles), continued, from seeds whose
words' low bits are free.  Bit for bit against the oracle."""
import numpy as np
import pytest

import oracle as O
import paper_1307_5869_gb300 as P

pytestmark = pytest.mark.gpu

BITS = {"u32": np.uint32, "f32": np.uint32, "f64": np.uint64}


@pytest.mark.parametrize("seed", [1, 2, 3, 2**40 + 9])
@pytest.mark.parametrize("n", [32, 77])
def test_rows_around_the_chunks(seed, n):
    g, ref = P.Generator("LFSR113", seed, 0, n), O.Streams("LFSR113", seed, 0, n)
    for per, dt in ((64, "u32"), (128, "f32"), (32, "f64"), (60, "u32"), (68, "f32"), (196, "u32"), (96, "f64"), (5, "u32"), (64, "f64")):
        got = g.generate(per, dt).cpu().numpy().view(BITS[dt]).reshape(n, per)
        assert np.array_equal(got, ref.generate(dt, per).view(BITS[dt])), (per, dt)
    g.close()
