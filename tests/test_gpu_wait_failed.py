"""What calls do after a kernel's bounded wait has run out.  The wait itself
never does in these tests: the word it would set is set from the host."""
import ctypes
from contextlib import contextmanager

import numpy as np
import pytest

import oracle as O
import paper_1307_5869_gb300 as P

pytestmark = pytest.mark.gpu

TIMEOUT = 6


class DevTables(ctypes.Structure):  # the head of the library's per-device tables
    _fields_ = [("device", ctypes.c_int), ("mrg", ctypes.c_void_p), ("lfsr", ctypes.c_void_p),
                ("gm", ctypes.c_void_p * 8), ("gm_tc", ctypes.c_void_p * 8),
                ("wait_failed", ctypes.POINTER(ctypes.c_uint32))]


@contextmanager
def wait_word():
    get = P.load()._ZN5prand10get_tablesEiPPNS_9DevTablesE
    t = ctypes.POINTER(DevTables)()
    assert get(P.GEN_ID["GM31"], ctypes.byref(t)) == 0
    word = t.contents.wait_failed
    assert word[0] == 0
    try:
        yield word
    finally:
        word[0] = 0


@contextmanager
def failed_wait():
    with wait_word() as word:
        word[0] = 1
        yield


def _status(fn):
    with pytest.raises(P.PrandError) as e:
        fn()
    return e.value.status


def test_a_batch_that_fails_half_way_is_joined():
    # MRG32K3A, MT19937 and GQ58.3 tiles run beside the refused GM31 ones: the caller's
    # stream goes on only when they have ended (MT19937 takes some 7 ms)
    import torch
    n = 1 << 24
    buf = torch.zeros(n + 3 * 1000, dtype=torch.int32, device="cuda")
    at = lambda i: buf.data_ptr() + 4 * i
    reqs = [("MT19937", 0, 7, n, at(0)), ("GM31", 0, 7, 1000, at(n)), ("GQ58_3", 0, 7, 1000, at(n + 1000)),
            ("MRG32K3A", 0, 7, 1000, at(n + 2000))]
    P.prand_batch_run(reqs, 61)
    torch.cuda.synchronize()
    want = buf.clone()
    buf.zero_()
    torch.cuda.synchronize()
    st = torch.cuda.Stream()
    with failed_wait():
        assert _status(lambda: P.prand_batch_run(reqs, 61, st.cuda_stream)) == TIMEOUT
        with torch.cuda.stream(st):
            got = buf.clone()
        st.synchronize()
    assert torch.equal(got[:n], want[:n])
    assert np.array_equal(got[:2000].cpu().numpy().view(np.uint32), O.State.stream("MT19937", 61, 7).u32(2000))
    torch.cuda.synchronize()
    P.prand_batch_run(reqs, 61, st.cuda_stream)
    torch.cuda.synchronize()
    assert torch.equal(buf, want)


@pytest.mark.parametrize("pinned", [True, False])
def test_a_host_fill_reports_its_own_wait(pinned):
    # the word is set after the fill is launched: it waits behind some 0.15 s of MT19937
    import threading
    import time

    import torch
    st = torch.cuda.Stream()
    g, before = P.Generator("GM31", 5, 0, 3000), P.Generator("MT19937", 5)
    out = torch.zeros(3000, 500, dtype=torch.int32, pin_memory=pinned)
    fill = lambda: P.prand_generate_host_u32(g.h, out.data_ptr(), 500, st.cuda_stream)
    fill()
    assert np.array_equal(out.numpy().view(np.uint32), O.Streams("GM31", 5, 0, 3000).generate("u32", 500))
    buf = torch.empty(400_000_000, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    with wait_word() as word:
        t = threading.Thread(target=lambda: (time.sleep(0.04), word.__setitem__(0, 1)))
        P.prand_generate_u32(before.h, buf.data_ptr(), buf.numel(), st.cuda_stream)
        t.start()
        assert _status(fill) == TIMEOUT
        t.join()
    fill()


def test_calls_after_a_failed_wait():
    import torch
    buf = torch.zeros(4000, dtype=torch.int32, device="cuda")
    reqs = [("GM61", 0, 3, 1000, buf.data_ptr()), ("MRG32K3A", 0, 3, 1000, buf.data_ptr() + 4000)]
    other = reqs[1:] + [("GQ58_3", 0, 3, 1000, buf.data_ptr() + 8000)]
    g, mrg = P.Generator("GM61", 5, 0, 200), P.Generator("MRG32K3A", 5, 0, 200)
    blob = g.get_state()
    plan, plain = P.prand_batch_plan_create(reqs, 62), P.prand_batch_plan_create(other, 62)
    host = np.zeros((200, 300), dtype=np.uint32)
    with failed_wait():
        for call in (lambda: g.generate(300), lambda: P.prand_generate_host_u32(g.h, host.ctypes.data, 300, 0),
                     lambda: P.prand_batch_run(reqs, 62), lambda: P.prand_batch_plan_create(reqs, 62),
                     lambda: P.prand_batch_plan_launch(plan), lambda: P.prand_batch_run_per_request(reqs, 62),
                     g.get_state, lambda: g.set_state(blob), lambda: g.skipahead(5), lambda: P.prand_init_streams(g.h, 0, 200)):
            assert _status(call) == TIMEOUT
        # what does not use those kernels goes on
        mrg.generate(300)
        P.prand_batch_run(other, 62)
        P.prand_batch_plan_launch(plain)
        torch.cuda.synchronize()
    for _ in range(2):
        buf.zero_()
        P.prand_batch_plan_launch(plan)
        torch.cuda.synchronize()
        assert np.array_equal(buf[:1000].cpu().numpy().view(np.uint32), O.State.stream("GM61", 62, 3).u32(1000))
    g.set_state(blob)
    assert np.array_equal(g.generate(300).cpu().numpy().view(np.uint32).reshape(200, 300), O.Streams("GM61", 5, 0, 200).generate("u32", 300))
    P.prand_batch_plan_destroy(plan)
    P.prand_batch_plan_destroy(plain)
