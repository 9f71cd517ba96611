"""Fills straight into page-locked memory, in the row forms of their own rules
(staged whatever the size when rows are on 16-byte boundaries): rows around a
128-byte segment, warps with idle lanes, split streams.  Against the oracle, with
nothing written outside the rows."""
import numpy as np
import pytest

import oracle as O
import paper_1307_5869_gb300 as P

pytestmark = pytest.mark.gpu

BITS = {"u32": np.uint32, "f32": np.uint32, "f64": np.uint64}


def check(gen, n, per, dt, offset=0):
    import torch
    tdt = {"u32": torch.int32, "f32": torch.float32, "f64": torch.float64}[dt]
    fill = {"u32": P.prand_generate_host_u32, "f32": P.prand_generate_host_f32, "f64": P.prand_generate_host_f64}[dt]
    flat = torch.zeros(n * per + offset + 8, dtype=tdt, pin_memory=True)
    g = P.Generator(gen, 3, 1, n)
    fill(g.h, flat[offset:].data_ptr(), per, 0)
    got = flat.numpy()[offset:offset + n * per].view(BITS[dt]).reshape(n, per)
    want = O.Streams(gen, 3, 1, n)
    assert np.array_equal(got, want.generate(dt, per).view(BITS[dt])), (gen, n, per, dt, offset)
    assert not flat[:offset].any() and not flat[offset + n * per:].any()
    assert np.array_equal(g.generate(5).cpu().numpy().view(np.uint32).reshape(n, 5), want.generate("u32", 5))
    g.close()


@pytest.mark.parametrize("dt", ["u32", "f32", "f64"])
@pytest.mark.parametrize("gen", ["MRG32K3A", "LFSR113", "GQ58_3"])
def test_rows_staged_into_host_memory(gen, dt):
    for n, per in ((1, 4), (1, 60000), (3, 9000), (33, 28), (100, 32), (257, 36), (1000, 64), (40, 1500)):
        check(gen, n, per, dt)
    check(gen, 65, 33, dt)
    check(gen, 33, 64, dt, offset=1)


@pytest.mark.parametrize("dt", ["f64", "u32"])
@pytest.mark.parametrize("gen", ["GM55", "GQ58_4"])
def test_rows_of_the_tensor_core_kernel_in_host_memory(gen, dt):
    # doubles leave four to a store where rows allow it, also in a block that ends early
    for n, per in ((5, 100), (17, 260), (33, 64), (700, 132)):
        check(gen, n, per, dt)
    check(gen, 17, 260, dt, offset=2)
    check(gen, 9, 131, dt)
    for per in (60, 130, 1026):   # many single elements: from 4 MiB on by the other kernel
        check(gen, 4 * 2**20 // per // (8 if dt == "f64" else 4) + 2, per, dt)
