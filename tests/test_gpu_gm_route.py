"""GM/GQ fills on both sides of the lines at which they change kernels and
forms: rows around whole blocks of 64, stream counts around whole and partly
full waves, few and many streams, rows off the vectors, long splits.  Against the
oracle, and every stream against the same streams filled in other sizes."""
import numpy as np
import pytest

import oracle as O
import paper_1307_5869_gb300 as P

pytestmark = pytest.mark.gpu

BITS = {"u32": np.uint32, "f32": np.uint32, "f64": np.uint64}
WAVE = {"GM55": 9728, "GQ58_4": 9728}   # resident sections of the tensor-core kernel (32 points: 2432)


def _fill(gen, n, calls):
    import torch
    whole, parts = P.Generator(gen, 21, 3, n), [(a, P.Generator(gen, 21, 3 + a, min(700, n - a))) for a in range(0, n, 700)]
    refs = {j: O.State.stream(gen, 21, 3 + j) for j in {0, n // 2, n - 1}}
    for per, dt in calls:
        got = whole.generate(per, dt).reshape(n, per)
        for a, g in parts:
            assert torch.equal(g.generate(per, dt).reshape(-1, per), got[a:a + 700]), (gen, n, per, dt, a)
        for j, s in refs.items():
            want = {"u32": s.u32, "f32": s.f32, "f64": s.f64}[dt](per)
            assert np.array_equal(got[j].cpu().numpy().view(BITS[dt]), want.view(BITS[dt])), (gen, n, per, dt, j)


@pytest.mark.parametrize("gen", ["GM29", "GM31", "GM55", "GM61", "GQ58_1", "GQ58_4"])
def test_rows_and_waves_around_the_lines(gen):
    w = WAVE.get(gen, 2432)
    rows = [(23, "u32"), (24, "f64"), (32, "f32"), (56, "u32"), (87, "u32"), (88, "f32"), (96, "f64"), (112, "u32"), (119, "f32"),
            (121, "u32"), (128, "f64"), (191, "u32"), (256, "f32")]
    for n in (1, 8, 64, w * 7 // 8 + 1, w, w + 1, w * 5 // 4 + 1, 3 * w - 5):
        _fill(gen, n, rows if n < 3000 else rows[::3])


@pytest.mark.parametrize("gen", ["GM55", "GQ58_3", "GQ58_4"])
def test_states_by_threads_and_by_tiles(gen):
    for n in (1, 31, 63, 64, 65, 100, 4097):
        _fill(gen, n, [(1, "u32"), (7, "f64"), (17, "f32"), (22, "u32"), (33, "u32")])


def test_a_split_stream_fills_no_part_of_a_third_block():
    # two streams of rows off the vectors: 77824 sections on two blocks per SM
    _fill("GQ58_3", 2, [(10_000_002, "u32"), (5, "u32"), (3_000_000, "f64")])
