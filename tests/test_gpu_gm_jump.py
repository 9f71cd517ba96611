"""The GM/GQ jumps by bytes of the exponent, against the oracle, bit for bit:
single bytes at every position, runs of full bytes across the 64-bit words,
stream indices at both ends of the range, and the blocks of streams one handle
opens (128 to a block)."""
import numpy as np
import pytest

import oracle as O
import paper_1307_5869_gb300 as P

pytestmark = pytest.mark.gpu

GENS = ["GM19", "GM29", "GM31", "GM55", "GM61", "GQ58_1", "GQ58_3", "GQ58_4"]


def _words(g, per):
    return g.generate(per, "u32").cpu().numpy().view(np.uint32)


@pytest.mark.parametrize("gen", GENS)
def test_bytes_of_the_offset(gen):
    offs = [0xA5 << (8 * i) for i in range(32)] + [2**64 - 1, 2**128 - 1, 2**192 - 2**60, 2**256 - 1, 255, 256]
    g, s = P.Generator(gen, 5, 1, 1), O.State.stream(gen, 5, 1)
    for off in offs:
        g.skipahead(off)
        s.jump(off)
        assert np.array_equal(_words(g, 3).reshape(-1), s.u32(3)), hex(off)
    g.close()


@pytest.mark.parametrize("gen", GENS)
@pytest.mark.parametrize("n", [1, 127, 129])
def test_streams_of_a_handle(gen, n):
    for first in (0, 255, O.gm_param(gen, "nmax") - 200):
        g = P.Generator(gen, 8, first, n)
        got = _words(g, 5).reshape(n, 5)
        g.close()
        for j in {0, n // 2, n - 1}:
            assert np.array_equal(got[j], O.State.stream(gen, 8, first + j).u32(5)), (first, j)
