"""Plans and servers keep their seed's base states however many other seeds
are used after them: bit for bit against the oracle."""
import numpy as np
import pytest

import oracle as O
import paper_1307_5869_gb300 as P

pytestmark = pytest.mark.gpu

STREAMS = [(g, 0, 3 + 5 * i, 700 + 64 * i) for i, g in enumerate(P.GENERATORS)]  # gen, u32, stream, length


def _requests(buf):
    at, reqs = 0, []
    for g, d, k, n in STREAMS:
        reqs.append((g, d, k, n, buf.data_ptr() + 4 * at))
        at += n
    return reqs


def _buffer():
    import torch
    return torch.zeros(sum(n for *_, n in STREAMS), dtype=torch.int32, device="cuda")


def _check(buf, seed):
    want = np.concatenate([O.State.stream(g, seed, k).u32(n) for g, _, k, n in STREAMS])
    assert np.array_equal(buf.cpu().numpy().view(np.uint32), want), seed


def _other_seeds(first):
    # more seeds than the library caches bases of, each with buffers of the same sizes
    import torch
    for seed in range(first, first + 6):
        buf = _buffer()
        P.prand_batch_run(_requests(buf), seed)
        torch.cuda.synchronize()
        _check(buf, seed)


def test_plan_after_other_seeds():
    import torch
    buf = _buffer()
    plan = P.prand_batch_plan_create(_requests(buf), 8001)
    _other_seeds(8100)
    for _ in range(2):
        buf.zero_()
        P.prand_batch_plan_launch(plan, torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        _check(buf, 8001)
    P.prand_batch_plan_destroy(plan)


def test_server_stream_first_seen_after_other_seeds():
    srv = P.prand_server_create(8002, 64 << 20, 16)
    try:
        _other_seeds(8200)
        ids = [P.prand_server_submit(srv, g, k, n, d) for g, d, k, n in STREAMS]
        for i, (g, _, k, n) in zip(ids, STREAMS):
            while not P.prand_server_query(srv, i)[0]:
                pass
            out = np.empty(n, dtype=np.uint32)
            P.prand_server_read(srv, i, out)
            assert np.array_equal(out, O.State.stream(g, 8002, k).u32(n)), (g, k)
    finally:
        P.prand_server_destroy(srv)
