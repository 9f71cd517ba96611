"""Batched and served requests whose tiles leave lanes idle or end rows apart:
lengths around whole chunks and sections, in both row sizes and block sizes, with
continuation through the server.  Bit for bit against the oracle."""
import numpy as np
import pytest

import oracle as O
import paper_1307_5869_gb300 as P

pytestmark = pytest.mark.gpu

BITS = {0: np.uint32, 1: np.uint32, 2: np.uint64}
DT = {0: "u32", 1: "f32", 2: "f64"}
GENS = ["MRG32K3A", "LFSR113", "GQ58_3"]
LENGTHS = [4, 32, 36, 64, 512, 1000, 2048, 2052, 2112, 3000, 4096 + 64, 10000, 33 * 2048 + 4]


@pytest.mark.parametrize("block,row_bytes", [(64, 128), (128, 256)])
def test_requests_of_few_sections(block, row_bytes):
    import torch
    reqs, outs = [], []
    for i, n in enumerate(LENGTHS):
        for g in GENS:
            for d in (0, 2):
                buf = torch.zeros(n + 2, dtype=[torch.int32, torch.float32, torch.float64][d], device="cuda")
                skew = i % 3 == 2   # off the vectors
                outs.append((g, d, 5 + i, n, buf, skew))
                reqs.append((g, d, 5 + i, n, buf[skew:].data_ptr()))
    P.prand_batch_set_params(2048, 4096, block, row_bytes)
    try:
        P.prand_batch_run(reqs, 91)
        torch.cuda.synchronize()
    finally:
        P.prand_batch_set_params(2048, 4096)
    for g, d, k, n, buf, skew in outs:
        got = buf.cpu().numpy().view(BITS[d])
        want = getattr(O.State.stream(g, 91, k), DT[d])(n).view(BITS[d])
        assert np.array_equal(got[skew:skew + n], want), (g, d, n)
        assert not got[:skew].any() and not got[skew + n:].any(), (g, d, n)


def test_served_requests_of_few_sections_continue():
    srv = P.prand_server_create(92, 64 << 20, 8)
    refs = {g: O.State.stream(g, 92, 3) for g in GENS}
    try:
        for n in LENGTHS + [7, 1001]:
            for d in (0, 2, 1):
                ids = [P.prand_server_submit(srv, g, 3, n, d) for g in GENS]
                for g, i in zip(GENS, ids):
                    while not P.prand_server_query(srv, i)[0]:
                        pass
                    out = np.empty(n, dtype=[np.uint32, np.float32, np.float64][d])
                    P.prand_server_read(srv, i, out)
                    P.prand_server_release(srv, i)
                    assert np.array_equal(out.view(BITS[d]), getattr(refs[g], DT[d])(n).view(BITS[d])), (g, n, d)
    finally:
        P.prand_server_destroy(srv)
