"""The slot-based tiles of the GM/GQ generators (a warp's sections, or a
thread's) in every kernel build the tuner can pick: through the request server,
which makes all GM/GQ requests that way, and through short batched requests."""
import numpy as np
import pytest

import oracle as O
import paper_1307_5869_gb300 as P

pytestmark = pytest.mark.gpu

GENS = [g for g in P.GENERATORS if g.startswith("G")]
BITS = {0: np.uint32, 1: np.uint32, 2: np.uint64}
DT = {0: "u32", 1: "f32", 2: "f64"}


@pytest.mark.parametrize("block,row_bytes", [(64, 128), (64, 256), (128, 128), (128, 256)])
def test_gm_tiles_of_every_build(block, row_bytes):
    import torch
    P.prand_batch_set_params(2048, 4096, block, row_bytes)
    try:
        srv = P.prand_server_create(51, 64 << 20, 16)
        bufs, reqs = [], []
        for i, g in enumerate(GENS):   # lane-per-point tiles of a batch: fewer than 96 outputs
            for n in (1, 31, 33, 95):
                t = torch.zeros(n + 1, dtype=torch.float64, device="cuda")
                bufs.append((g, 9 + i, n, t))
                reqs.append((g, 2, 9 + i, n, t[n % 2:].data_ptr()))
        P.prand_batch_run(reqs, 52)
        torch.cuda.synchronize()
    finally:
        P.prand_batch_set_params(2048, 4096)
    for g, k, n, t in bufs:
        got = t.cpu().numpy().view(np.uint64)[n % 2:][:n]
        assert np.array_equal(got, O.State.stream(g, 52, k).f64(n).view(np.uint64)), (g, n)
    refs = {}
    try:
        for n in (5, 127, 4096, 20001):   # 20001: several tiles, ragged section ends
            for d in (0, 2, 1):
                ids = [(g, P.prand_server_submit(srv, g, 4, n, d)) for g in GENS]
                for g, i in ids:
                    while not P.prand_server_query(srv, i)[0]:
                        pass
                    out = np.empty(n, dtype=[np.uint32, np.float32, np.float64][d])
                    P.prand_server_read(srv, i, out)
                    P.prand_server_release(srv, i)
                    ref = refs.setdefault(g, O.State.stream(g, 51, 4))
                    assert np.array_equal(out.view(BITS[d]), getattr(ref, DT[d])(n).view(BITS[d])), (g, n, d)
    finally:
        P.prand_server_destroy(srv)
