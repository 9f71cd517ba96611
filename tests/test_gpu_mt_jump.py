"""The MT19937 polynomial jump on the GPU: offsets whose polynomials are one
coefficient (2^b < 19937, near and at the ends of the kernel's blocks of 320 and
steps of 640) and dense ones, against the words generated one after another and
against the oracle.  Whole words, compared exactly."""
import numpy as np
import pytest

import oracle as O
import paper_1307_5869_gb300 as P

pytestmark = pytest.mark.gpu

N = 624


def _words(g, per):
    return g.generate(per, "u32").cpu().numpy().view(np.uint32)


@pytest.mark.parametrize("streams", [1, 5])
def test_skips_equal_generating(streams):
    offs = [1 << b for b in range(15)] + [319, 320, 639, 641, 19936, 19937, 1 << 15, (1 << 16) + 623, 150001]
    g = P.Generator("MT19937", 9, 3, streams)
    seq = _words(g, max(offs) + 2 * N + 40).reshape(streams, -1)
    for off in offs:
        h = P.Generator("MT19937", 9, 3, streams)
        _words(h, N)                   # a whole block: the skip is one jump per set bit
        h.skipahead(off)
        assert np.array_equal(_words(h, N + 40).reshape(streams, -1), seq[:, N + off:2 * N + 40 + off]), off
        h.close()
    g.close()


@pytest.mark.parametrize("first,n", [(0, 2), (6, 3), (2**33 + 5, 67), (1, 700)])
def test_streams_equal_the_oracle(first, n):
    g = P.Generator("MT19937", 21, first, n)
    got = _words(g, 700).reshape(n, 700)
    g.close()
    for j in {0, 1, n // 2, n - 1}:
        assert np.array_equal(got[j], O.Streams("MT19937", 21, first + j, 1).generate("u32", 700)[0]), j
