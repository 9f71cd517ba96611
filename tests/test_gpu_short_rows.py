"""Short rows of the thread-per-stream ensembles, whose states pass through
shared memory 32 streams at a time, and streams opened again on a handle's own
buffers.  Bit for bit against the oracle."""
import numpy as np
import pytest

import oracle as O
import paper_1307_5869_gb300 as P

pytestmark = pytest.mark.gpu

BITS = {"u32": np.uint32, "f32": np.uint32, "f64": np.uint64}


@pytest.mark.parametrize("gen", ["GM55", "GQ58_3", "GQ58_4"])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 257, 5000])
def test_rows(gen, n):
    g, ref = P.Generator(gen, 3, 4, n), O.Streams(gen, 3, 4, n)
    for per, dt in ((1, "u32"), (4, "f32"), (3, "f64"), (20, "u32"), (1, "f64")):
        got = g.generate(per, dt).cpu().numpy().view(BITS[dt]).reshape(n, per)
        assert np.array_equal(got, ref.generate(dt, per).view(BITS[dt])), (per, dt)
    g.close()


@pytest.mark.parametrize("gen", ["MT19937", "MRG32K3A", "GM61", "GQ58_3"])
def test_opened_again(gen):
    g = P.Generator(gen, 3, 0, 40)
    g.generate(700, "u32")
    for first, n in ((5, 40), (5, 40), (6, 39), (0, 40)):
        P.prand_init_streams(g.h, first, n)
        g.n_streams = n
        got = g.generate(30, "u32").cpu().numpy().view(np.uint32).reshape(n, 30)
        assert np.array_equal(got, O.Streams(gen, 3, first, n).generate("u32", 30)), (first, n)
    g.close()
