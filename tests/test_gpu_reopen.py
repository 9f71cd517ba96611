"""Opening streams again, as many as before, while other work is about: another
thread's graph capture goes on, and work of the handle still on the device does
not reach the new states."""
import threading

import numpy as np
import pytest

import oracle as O
import paper_1307_5869_gb300 as P

pytestmark = pytest.mark.gpu


def _u32(t):
    return t.cpu().numpy().view(np.uint32)


@pytest.mark.parametrize("mode", ["thread_local", "relaxed"])
def test_another_threads_capture_goes_on(mode):
    import torch
    opened = P.Generator("GQ58_3", 9, 0, 300)
    buf = torch.zeros(500, dtype=torch.int32, device="cuda")
    plan = P.prand_batch_plan_create([("MRG32K3A", 0, 3, 500, buf.data_ptr())], 9)
    captured = P.Generator("LFSR113", 9, 0, 50)
    out = torch.zeros(50, 64, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    errors = []

    def other():
        try:
            P.prand_init_streams(opened.h, 70, 300)
            P.prand_batch_plan_launch(plan, 0)
            P.prand_batch_plan_destroy(plan)
        except Exception as e:
            errors.append(e)

    graph, st = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=st, capture_error_mode=mode):
        captured.generate(64, out=out, stream=st.cuda_stream)
        t = threading.Thread(target=other)
        t.start()
        t.join()
    assert not errors, errors
    graph.replay()
    torch.cuda.synchronize()
    assert np.array_equal(_u32(out), O.Streams("LFSR113", 9, 0, 50).generate("u32", 64))
    assert np.array_equal(_u32(opened.generate(40)).reshape(300, 40), O.Streams("GQ58_3", 9, 70, 300).generate("u32", 40))
    assert np.array_equal(_u32(buf), O.State.stream("MRG32K3A", 9, 3).u32(500))


def test_replayed_fills_do_not_reach_the_new_states():
    # fills captured on one stream and replayed on another, which the handle has not seen
    import torch
    n, per = 3000, 20000
    g = P.Generator("GM31", 9, 0, n)
    out = torch.zeros(n, per, dtype=torch.int32, device="cuda")
    graph, st = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=st):
        g.generate(per, out=out, stream=st.cuda_stream)
    with torch.cuda.stream(torch.cuda.Stream()):
        for _ in range(100):
            graph.replay()
    P.prand_init_streams(g.h, 40, n)
    torch.cuda.synchronize()
    got = _u32(g.generate(64)).reshape(n, 64)
    want = O.Streams("GM31", 9, 40, n).generate("u32", 64)
    assert np.array_equal(got, want)
