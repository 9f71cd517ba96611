"""Batches one behind another on different streams and from different threads:
each call's outputs against the oracle and against the same requests alone."""
import threading

import numpy as np
import pytest

import oracle as O
import paper_1307_5869_gb300 as P

pytestmark = pytest.mark.gpu


def _spec(seed, count, maxlen):
    rng = np.random.default_rng(seed)
    return [(P.GENERATORS[i % 11], int(rng.integers(0, 10**18)), int(2 ** (np.log2(maxlen) * rng.random())) + 1) for i in range(count)]


def _batch(spec):
    import torch
    buf = torch.zeros(sum(n for *_, n in spec), dtype=torch.int32, device="cuda")
    at, reqs = 0, []
    for g, k, n in spec:
        reqs.append((g, 0, k, n, buf.data_ptr() + 4 * at))
        at += n
    return buf, reqs


def _check(buf, spec, seed, alone):
    import torch
    assert torch.equal(buf, alone)
    at = 0
    for i, (g, k, n) in enumerate(spec):
        if i % 9 == 0:
            want = O.State.stream(g, seed, k).u32(min(n, 2000))
            assert np.array_equal(buf[at:at + len(want)].cpu().numpy().view(np.uint32), want), (g, k, n)
        at += n


# the second batch larger (its list needs a larger buffer), smaller and of the same size
SPECS = [(21, 60, 1 << 17), (22, 400, 1 << 15), (23, 30, 1 << 10), (24, 400, 1 << 14)]


def _alone(seed):
    import torch
    out = []
    for s in SPECS:
        spec = _spec(*s)
        buf, reqs = _batch(spec)
        P.prand_batch_run(reqs, seed)
        torch.cuda.synchronize()
        out.append((spec, buf))
    return out


def test_two_streams_back_to_back():
    import torch
    alone = _alone(31)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for _ in range(3):
        bufs = [_batch(spec) for spec, _ in alone]
        torch.cuda.synchronize()
        for i, (_, reqs) in enumerate(bufs):
            P.prand_batch_run(reqs, 31, streams[i % 2].cuda_stream)
        torch.cuda.synchronize()
        for (spec, want), (buf, _) in zip(alone, bufs):
            _check(buf, spec, 31, want)


def test_threads_on_their_own_streams():
    import torch
    alone = _alone(32)
    bufs = [_batch(spec) for spec, _ in alone]
    streams = [torch.cuda.Stream() for _ in bufs]
    torch.cuda.synchronize()
    failed = []

    def run(i):
        try:
            for _ in range(3):
                P.prand_batch_run(bufs[i][1], 32, streams[i].cuda_stream)
        except Exception as e:  # a thread's assertion is reported by the test
            failed.append(e)

    threads = [threading.Thread(target=run, args=(i,)) for i in range(len(bufs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failed, failed
    for (spec, want), (buf, _) in zip(alone, bufs):
        _check(buf, spec, 32, want)
