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
def failed_wait():
    get = P.load()._ZN5prand10get_tablesEiPPNS_9DevTablesE
    t = ctypes.POINTER(DevTables)()
    assert get(P.GEN_ID["GM31"], ctypes.byref(t)) == 0
    word = t.contents.wait_failed
    assert word[0] == 0
    word[0] = 1
    try:
        yield
    finally:
        word[0] = 0


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
