"""Staged stores of rows that start anywhere (fills too large for L2, odd row
lengths, outputs off a 16-byte boundary): against the oracle on a few rows, and
all rows against the same streams filled in parts that are small enough for
each thread's own stores.  The MRG32K3A jumps by bytes of the exponent, against
the oracle.  Bit for bit."""
import numpy as np
import pytest

import oracle as O
import paper_1307_5869_gb300 as P

pytestmark = pytest.mark.gpu

BITS = {"u32": np.uint32, "f32": np.uint32, "f64": np.uint64}


@pytest.mark.parametrize("gen", ["MRG32K3A", "LFSR113", "GQ58_3"])
@pytest.mark.parametrize("n,per,dt,offset", [(2**21 + 5, 65, "u32", 1), (2**16, 1001, "f32", 3), (2**17 - 1, 333, "f64", 1)])
def test_rows_off_the_vectors(gen, n, per, dt, offset):
    import torch
    tdt = {"u32": torch.int32, "f32": torch.float32, "f64": torch.float64}[dt]
    flat = torch.zeros(n * per + offset + 8, dtype=tdt, device="cuda")
    g = P.Generator(gen, 6, 2, n)
    g.generate(per, dt, out=flat[offset:offset + n * per])
    got = flat[offset:offset + n * per].view(n, per)
    assert not flat[:offset].any() and not flat[offset + n * per:].any()   # nothing outside the rows
    for j in (0, 33, n - 1):
        s = O.State.stream(gen, 6, 2 + j)
        want = {"u32": s.u32, "f32": s.f32, "f64": s.f64}[dt](per)
        assert np.array_equal(got[j].cpu().numpy().view(BITS[dt]), want.view(BITS[dt])), j
    part = (n + 7) // 8
    for a in range(0, n, part):
        m = min(part, n - a)
        h = P.Generator(gen, 6, 2 + a, m)
        assert torch.equal(h.generate(per, dt).reshape(m, per), got[a:a + m]), a
        h.close()
    tail = g.generate(5, "u32").reshape(n, 5)[n - 1].cpu().numpy().view(np.uint32)   # the next state
    s = O.State.stream(gen, 6, 2 + n - 1)
    s.u32(per)
    assert np.array_equal(tail, s.u32(5))
    g.close()


def test_mrg_jumps_by_bytes():
    offs = [0xA5 << (8 * i) for i in range(32)] + [2**64 - 1, 2**128 - 1, 2**256 - 1, 255, 256]
    g, s = P.Generator("MRG32K3A", 5, 1, 1), O.State.stream("MRG32K3A", 5, 1)
    for off in offs:
        g.skipahead(off)
        s.jump(off)
        assert np.array_equal(g.generate(3, "u32").cpu().numpy().view(np.uint32).reshape(-1), s.u32(3)), hex(off)
    for per, dt in ((200000, "u32"), (100032, "f64"), (31, "f32")):   # sections of 32 outputs
        want = {"u32": s.u32, "f32": s.f32, "f64": s.f64}[dt](per)
        assert np.array_equal(g.generate(per, dt).cpu().numpy().reshape(-1).view(BITS[dt]), want.view(BITS[dt])), per
    g.close()
    for first in (0, 255, 2**40 + 77, 10**19 - 200):
        g = P.Generator("MRG32K3A", 8, first, 130)
        got = g.generate(5, "u32").cpu().numpy().view(np.uint32).reshape(130, 5)
        for j in (0, 64, 129):
            assert np.array_equal(got[j], O.State.stream("MRG32K3A", 8, first + j).u32(5)), (first, j)
        g.close()
