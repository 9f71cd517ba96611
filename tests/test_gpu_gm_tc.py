"""GPU parity of the GM/GQ tensor-core generation at the sizes where it can go
wrong: rows around the 32-word rows and 64-step blocks, streams around the
points of a product (4 or 16 streams), tiles that straddle two sections, split
streams and continuation, misaligned outputs.  Bit for bit against the oracle."""
import numpy as np
import pytest

import oracle as O
import paper_1307_5869_gb300 as P

pytestmark = pytest.mark.gpu

GENS = ["GM19", "GM29", "GM31", "GM55", "GM61", "GQ58_1", "GQ58_4"]
BITS = {"u32": np.uint32, "f32": np.uint32, "f64": np.uint64}


def _check(gen, n, calls, offset=0):
    import torch
    g, ref = P.Generator(gen, 77, 2, n), O.Streams(gen, 77, 2, n)
    for per, dt in calls:
        tdt = {"u32": torch.int32, "f32": torch.float32, "f64": torch.float64}[dt]
        flat = torch.zeros(n * per + offset + 8, dtype=tdt, device="cuda")
        out = flat[offset:offset + n * per]
        g.generate(per, dt, out=out)
        got = out.cpu().numpy().view(BITS[dt]).reshape(n, per)
        assert np.array_equal(got, ref.generate(dt, per).view(BITS[dt])), (gen, n, per, dt)
        assert not flat[:offset].any() and not flat[offset + n * per:].any()   # nothing outside the rows
    g.close()


@pytest.mark.parametrize("gen", GENS)
def test_rows_around_the_blocks(gen):
    # one stream, and one more or fewer than the streams of one product
    for n in (1, 3, 4, 5, 15, 17):
        _check(gen, n, [(128, "u32"), (191, "f32"), (192, "u32"), (193, "f64"), (224, "u32"), (225, "u32"), (255, "u32")])


@pytest.mark.parametrize("gen", GENS)
def test_split_streams(gen):
    # sections of 256 and more, several per stream and tile, the last one ragged
    _check(gen, 1, [(100003, "u32"), (256, "u32"), (65536, "f32")])
    _check(gen, 7, [(30001, "u32"), (513, "f64")], offset=1)


@pytest.mark.parametrize("gen", GENS)
def test_more_streams_than_one_wave(gen):
    # several tiles per block of threads (2432 or 9728 resident sections), the last one partial
    n = 9731 if gen in ("GM55", "GQ58_4") else 2437
    _check(gen, n, [(64, "u32"), (100, "f32"), (1030, "u32")])
