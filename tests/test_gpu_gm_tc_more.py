"""The tensor-core kernel for the generators that take it only beyond one wave
of streams (GM19, GM29), in all types and row forms, and two of its fills at once
on two streams, where their blocks share the SMs' tensor memory."""
import numpy as np
import pytest

import oracle as O
import paper_1307_5869_gb300 as P

pytestmark = pytest.mark.gpu

BITS = {"u32": np.uint32, "f32": np.uint32, "f64": np.uint64}


def _rows(gen, first, n, calls, offset):
    import torch
    g = P.Generator(gen, 77, first, n)
    refs = {j: O.State.stream(gen, 77, first + j) for j in (0, 1, 3, n // 2, n - 2, n - 1)}
    for per, dt in calls:
        tdt = {"u32": torch.int32, "f32": torch.float32, "f64": torch.float64}[dt]
        flat = torch.zeros(n * per + offset + 8, dtype=tdt, device="cuda")
        g.generate(per, dt, out=flat[offset:offset + n * per])
        got = flat[offset:offset + n * per].view(n, per)
        for j, s in refs.items():
            want = {"u32": s.u32, "f32": s.f32, "f64": s.f64}[dt](per)
            assert np.array_equal(got[j].cpu().numpy().view(BITS[dt]), want.view(BITS[dt])), (gen, n, per, dt, j)
        assert not flat[:offset].any() and not flat[offset + n * per:].any()
    g.close()


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("gen", ["GM19", "GM29"])
def test_beyond_one_wave(gen, offset):
    # 2432 sections are one wave: rows of whole blocks, one more and one fewer output
    _rows(gen, 0, 2441, [(1024, "u32"), (1025, "f32"), (1087, "f64"), (2050, "u32"), (896, "f64")], offset)
    _rows(gen, 0, 3000, [(2048, "f32"), (2111, "u32")], offset)


@pytest.mark.parametrize("gen", ["GM19", "GM29", "GM31", "GQ58_1"])
def test_batched_sections(gen):
    # batches take it from one request on: section ends around blocks, all types
    import torch
    reqs, outs = [], []
    for i, n in enumerate((192, 255, 256, 257, 1000, 4 * 4096, 4 * 4096 + 1, 50001)):
        for d, dt in enumerate(("u32", "f32", "f64")):
            t = torch.zeros(n + 1, dtype=[torch.int32, torch.float32, torch.float64][d], device="cuda")
            outs.append((n, dt, i, t[i % 2:][:n]))
            reqs.append((gen, d, i, n, t[i % 2:].data_ptr()))
    P.prand_batch_run(reqs, 78)
    torch.cuda.synchronize()
    for n, dt, k, t in outs:
        s = O.State.stream(gen, 78, k)
        want = {"u32": s.u32, "f32": s.f32, "f64": s.f64}[dt](n)
        assert np.array_equal(t.cpu().numpy().view(BITS[dt]), want.view(BITS[dt])), (n, dt)


def test_two_fills_at_once():
    import torch
    jobs = [("GM61", 9000, 700), ("GM55", 30000, 300), ("GM31", 5000, 1000), ("GQ58_4", 20000, 500)]
    gens, streams = [P.Generator(g, 5, 0, n) for g, n, _ in jobs], [torch.cuda.Stream() for _ in jobs]
    outs = [torch.zeros(n, per, dtype=torch.int32, device="cuda") for _, n, per in jobs]
    torch.cuda.synchronize()
    for _ in range(4):
        for g, st, out, (_, _, per) in zip(gens, streams, outs, jobs):
            g.generate(per, out=out, stream=st.cuda_stream)
    torch.cuda.synchronize()
    for (name, n, per), out in zip(jobs, outs):
        alone = P.Generator(name, 5, 0, n)
        for _ in range(4):
            want = alone.generate(per)
        assert torch.equal(out, want.view(n, per)), name
        s = O.State.stream(name, 5, n - 1)
        s.u32(3 * per)
        assert np.array_equal(out[n - 1].cpu().numpy().view(np.uint32), s.u32(per)), name
