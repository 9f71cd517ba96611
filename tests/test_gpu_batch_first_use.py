"""The first batched calls of a process made by several threads at once."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = """
import threading
import numpy as np, torch
import oracle as O
import paper_1307_5869_gb300 as P
torch.cuda.init()
start, failed, plans, made = threading.Barrier(6), [], [], []
def run(i):
    try:
        spec = [(g, 11 * i + j, 900 + j) for j, g in enumerate(P.GENERATORS)]
        buf = torch.zeros(sum(n for *_, n in spec), dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        st = torch.cuda.Stream()
        at, reqs = 0, []
        for g, k, n in spec:
            reqs.append((g, 0, k, n, buf.data_ptr() + 4 * at))
            at += n
        start.wait()
        if i % 2:
            plan = P.prand_batch_plan_create(reqs, 40 + i)
            P.prand_batch_plan_launch(plan, st.cuda_stream)
            st.synchronize()
            plans.append(plan)
        else:
            P.prand_batch_run(reqs, 40 + i, st.cuda_stream)
            st.synchronize()
        made.append((i, spec, buf))
    except Exception as e:
        failed.append((i, repr(e)))
threads = [threading.Thread(target=run, args=(i,)) for i in range(6)]
for t in threads: t.start()
for t in threads: t.join()
for p in plans: P.prand_batch_plan_destroy(p)
assert not failed, failed
for i, spec, buf in made:  # (the oracle is one thread's)
    got = np.split(buf.cpu().numpy().view(np.uint32), np.cumsum([n for *_, n in spec])[:-1])
    for (g, k, n), words in zip(spec, got):
        assert np.array_equal(words, O.State.stream(g, 40 + i, k).u32(n)), (i, g, k, n)
print("ok")
"""


def test_threads_make_the_first_batches():
    r = subprocess.run([sys.executable, "-c", PROGRAM], capture_output=True, text=True, timeout=300, cwd=ROOT)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stderr[-2000:]
