"""Workloads the library is timed on, each through the public entry points.

Every case is a dict of plain values; ``prepare`` makes what a program has in
hand before the call (a handle with its streams, an output buffer, a batch
plan, a server), ``run`` makes one pass, ``work`` counts what the pass cannot
do without, and ``exact`` recomputes the floating outputs from the generators'
definitions in 64-bit integers (no MT19937: its streams start 2^432 outputs
apart, which takes polynomial jumps).
"""
from __future__ import annotations

import os
import time

os.environ.setdefault("CUDA_DEVICE_MAX_CONNECTIONS", "32")  # as the request server's users set it

import numpy as np
import torch

import paper_1307_5869_gb300 as P
from paper_1307_5869_gb300 import workloads as W

DTYPES = ("u32", "f32", "f64")
TORCH = {"u32": torch.int32, "f32": torch.float32, "f64": torch.float64}
NUMPY = {"u32": np.uint32, "f32": np.float32, "f64": np.float64}
M64 = (1 << 64) - 1

# points per word, bits per point, k, q, p, block length, sequences (the paper's Tables 2 and 4)
GM = {"GM19": (32, 1, 15, 28, (1 << 19) - 1, 6 * 10**6, 10**3),
      "GM29": (32, 1, 4, 2, (1 << 29) - 3, 8 * 10**7, 10**8),
      "GM31": (32, 1, 11, 14, (1 << 31) - 1, 8 * 10**7, 10**9),
      "GM55": (8, 4, 256, 176, (1 << 51) - 129, 10**10, 10**18),
      "GM61": (32, 1, 24, 74, (1 << 61) - 1, 10**10, 18 * 10**18),
      "GQ58_1": (32, 1, 8, 48, (1 << 29) - 3, 8 * 10**7, 10**8),
      "GQ58_3": (12, 3, 8, 48, (1 << 29) - 3, 8 * 10**7, 2 * 10**8),
      "GQ58_4": (8, 4, 8, 48, (1 << 29) - 3, 8 * 10**7, 3 * 10**8)}


def listed():
    n16, n20 = W.TABLE_STREAMS, W.BULK_STREAMS
    return [
        # a simulation on one host thread drawing an odd handful of numbers per stream: the
        # smallest calls, where the launch and the host path are all there is
        {"name": "few_streams_mt19937_f32", "kind": "fill", "gen": "MT19937", "dtype": "f32", "streams": 96, "per": 1001},
        # one long stream, split into sections by the library (the single-stream workload)
        {"name": "one_stream_mrg32k3a_f64", "kind": "fill", "gen": "MRG32K3A", "dtype": "f64", "streams": 1,
         "per": W.SINGLE_LENGTH},
        # a Monte Carlo step of an odd number of walkers with an odd number of draws each
        {"name": "ragged_gm31_u32", "kind": "fill", "gen": "GM31", "dtype": "u32", "streams": 12345, "per": 777},
        # the table of all generators at its shape (2^16 streams x 2^12): a torus-map ensemble
        # with four bits per point
        {"name": "table_gq58_4_f32", "kind": "fill", "gen": "GQ58_4", "dtype": "f32", "streams": n16,
         "per": W.TABLE_PER_STREAM},
        # the benchmark's bulk fill (2^20 streams x 2^10), its three generators
        {"name": "bulk_mt19937_u32", "kind": "fill", "gen": "MT19937", "dtype": "u32", "streams": n20, "per": W.BULK_PER_STREAM},
        {"name": "bulk_lfsr113_f32", "kind": "fill", "gen": "LFSR113", "dtype": "f32", "streams": n20, "per": W.BULK_PER_STREAM},
        {"name": "bulk_gm61_u32", "kind": "fill", "gen": "GM61", "dtype": "u32", "streams": n20, "per": W.BULK_PER_STREAM},
        # the same outputs wanted on the host, in page-locked memory (the end-to-end form)
        {"name": "host_gm61_f32", "kind": "host", "gen": "GM61", "dtype": "f32", "streams": n16, "per": W.BULK_PER_STREAM},
        # a job that opens its streams (jump-ahead to 2^16 streams) and draws a first block of each
        {"name": "open_mt19937_u32", "kind": "open", "gen": "MT19937", "dtype": "u32", "streams": n16, "per": 256},
        # ten thousand requests of mixed generators and uneven lengths, planned once, launched per step
        {"name": "batch_10000_u32", "kind": "batch", "requests": 10_000, "max_log2": 20, "dtype": "u32"},
        # a burst of requests on streams the server has not seen, read back to the host
        {"name": "serve_48_mixed", "kind": "serve", "requests": 48, "max_log2": 18},
        # the skip-ahead study: spaced streams, one word each, three tests' cell counts
        {"name": "study_gq58_3", "kind": "study", "gen": "GQ58_3", "skip": W.STUDY_SKIPS["GQ58_3"], "words": W.STUDY_WORDS},
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(lo * (hi / lo) ** rng.random())))


def draw(rng):
    kind = rng.choice(["fill"] * 7 + ["host", "open", "batch", "serve", "study"])
    gen = rng.choice(W.GENERATORS)
    dtype = rng.choice(DTYPES)
    if kind in ("fill", "host"):
        total = _log(rng, 1 << 8, 1 << (27 if kind == "fill" else 24))
        streams = _log(rng, 1, min(total, 1 << 20))
        per = max(1, total // streams)
        if rng.random() < 0.5:  # half of them on vector-friendly rows, half odd
            per, streams = (per + 3) // 4 * 4, max(1, streams)
        else:
            per |= 1
        return {"kind": kind, "gen": gen, "dtype": dtype, "streams": streams, "per": per}
    if kind == "open":
        return {"kind": kind, "gen": gen, "dtype": "u32", "streams": _log(rng, 1, 1 << 16), "per": _log(rng, 1, 1 << 9)}
    if kind == "batch":
        return {"kind": kind, "requests": _log(rng, 10, 10_000), "max_log2": rng.randint(8, 20), "dtype": "u32"}
    if kind == "serve":
        return {"kind": kind, "requests": _log(rng, 4, 60), "max_log2": rng.randint(8, 18)}
    words = _log(rng, 1 << 12, W.STUDY_WORDS_MT if gen == "MT19937" else W.STUDY_WORDS)
    return {"kind": kind, "gen": gen, "skip": W.STUDY_SKIPS[gen], "words": words}


def _seed(seed):
    return (W.BULK_SEED_BASE + 0x632BE59BD9B4E019 * (seed + 1)) & (M64 >> 1)


def _first(case, seed):
    """First stream of a job: below the generator's capacity, any 64-bit index for the large ones."""
    room = {"GM19": 500}.get(case["gen"], 1 << 20)
    return (seed * 7919 + 13) % room


def _batch_requests(case, seed):
    """The batched workload's generators and lengths; the streams of another seed are other streams."""
    streams = np.random.default_rng(7 + seed).integers(0, 10**19, size=case["requests"], dtype=np.uint64)
    return [(g, int(s), n) for (g, _, n, _), s in zip(W.batched_requests(case["requests"], 7, case["max_log2"]), streams)]


def _serve_requests(case, seed):
    """Generators in turn, lengths from 2^6 up, the three types in turn; the seed draws the streams."""
    n = case["requests"]
    lengths = np.floor(2.0 ** (6 + (case["max_log2"] - 6) * np.random.default_rng(11).random(n))).astype(np.int64)
    streams = np.random.default_rng(11 + seed).integers(0, 9 * 10**18, size=n, dtype=np.uint64)
    return [(W.GENERATORS[i % 11], int(streams[i]), int(lengths[i]), i % 3) for i in range(n)]


class _Server:
    def __init__(self, seed):
        self.h = P.prand_server_create(seed, 1 << 30, 1 << 15)

    def __del__(self):
        P.prand_server_destroy(self.h)


class _Plan:
    def __init__(self, requests, seed):
        self.h = P.prand_batch_plan_create(requests, seed)

    def __del__(self):
        P.prand_batch_plan_destroy(self.h)


def prepare(case, seed):
    kind, s = case["kind"], _seed(seed)
    st = {"case": case}
    if kind in ("fill", "host", "open"):
        shape = (case["streams"], case["per"])
        st["first"] = _first(case, seed)
        st["g"] = P.Generator(case["gen"], s, st["first"], 1 if kind == "open" else case["streams"])
        if kind == "host":
            st["out"] = torch.zeros(shape, dtype=TORCH[case["dtype"]], pin_memory=True)
        else:
            st["out"] = torch.zeros(shape, dtype=TORCH[case["dtype"]], device="cuda")
    elif kind == "batch":
        reqs = _batch_requests(case, seed)
        at, full = 0, []
        for g, k, n in reqs:
            full.append((g, k, n, at))
            at += (n + 63) // 64 * 64
        st["out"] = torch.zeros(at, dtype=torch.int32, device="cuda")
        base = st["out"].data_ptr()
        st["plan"] = _Plan([(g, P.DTYPE_U32, k, n, base + 4 * o) for g, k, n, o in full], s)
    elif kind == "serve":
        st["reqs"] = _serve_requests(case, seed)
        st["srv"] = _Server(s)
        st["passes"] = 0
        st["outs"] = [np.zeros(n, dtype=NUMPY[DTYPES[d]]) for _, _, n, d in st["reqs"]]
    else:
        st["h"] = P.Generator(case["gen"], s, 0, 1)
        st["out"] = torch.zeros(case["words"], dtype=torch.int32, device="cuda")
        kinds = {"frequency": P.TEST_FREQUENCY, "serial": P.TEST_SERIAL, "gap": P.TEST_GAP}
        st["tests"] = [P.make_test(kinds[nm], **kw) for nm, kw in W.STUDY_TESTS]
        st["counts"] = [torch.zeros(P.prand_test_cells(t), dtype=torch.int64, device="cuda") for t in st["tests"]]
    return st


def _serve(st):
    """Every pass asks for streams the server has not seen: the drawn ones, shifted by the pass."""
    srv, shift = st["srv"].h, st["passes"]
    st["passes"] += 1
    ids = [P.prand_server_submit(srv, g, k + shift, n, d) for g, k, n, d in st["reqs"]]
    left = len(ids)
    while left:
        got = len(P.prand_server_completed(srv, len(ids)))
        left -= got
        if not got:
            time.sleep(20e-6)
    for i, out in zip(ids, st["outs"]):
        P.prand_server_read(srv, i, out)
        P.prand_server_release(srv, i)
    return st["outs"]


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "fill":
        return st["g"].generate(case["per"], case["dtype"], out=st["out"])
    stream = torch.cuda.current_stream().cuda_stream
    if kind == "host":
        fn = {"u32": P.prand_generate_host_u32, "f32": P.prand_generate_host_f32, "f64": P.prand_generate_host_f64}
        fn[case["dtype"]](st["g"].h, st["out"].data_ptr(), case["per"], stream)
        return st["out"]
    if kind == "open":
        P.prand_init_streams(st["g"].h, st["first"], case["streams"])
        st["g"].n_streams = case["streams"]
        return st["g"].generate(case["per"], case["dtype"], out=st["out"])
    if kind == "batch":
        P.prand_batch_plan_launch(st["plan"].h, stream)
        return st["out"]
    if kind == "serve":
        return _serve(st)
    P.prand_init_streams_spaced(st["h"].h, case["skip"], 0, case["words"])
    P.prand_generate_u32(st["h"].h, st["out"].data_ptr(), 1, stream)
    for t, c in zip(st["tests"], st["counts"]):
        P.prand_test_counts(t, st["out"].data_ptr(), case["words"], c.data_ptr(), stream)
    return [st["out"]] + st["counts"]


def _ops(gen):
    """Operations per output: the recurrence's multiplies, adds and reductions, the output map."""
    if gen in GM:
        return 5 * GM[gen][0]
    return {"MT19937": 12, "MRG32K3A": 15, "LFSR113": 27}[gen]


def _state_bytes(gen):
    return 16 * GM[gen][0] if gen in GM else {"MT19937": 2496, "MRG32K3A": 24, "LFSR113": 16}[gen]


def work(case):
    kind = case["kind"]
    if kind in ("fill", "host", "open"):
        n, per = case["streams"], case["per"]
        state = n * _state_bytes(case["gen"]) * 2
        return {"bytes": n * per * (8 if case["dtype"] == "f64" else 4) + state, "flops": n * per * _ops(case["gen"])}
    if kind == "batch":
        reqs = _batch_requests(case, 0)
        return {"bytes": 4 * sum(n for _, _, n in reqs), "flops": sum(n * _ops(g) for g, _, n in reqs)}
    if kind == "serve":
        reqs = _serve_requests(case, 0)
        return {"bytes": sum(n * (8 if d == 2 else 4) for _, _, n, d in reqs), "flops": sum(n * _ops(g) for g, _, n, _ in reqs)}
    n = case["words"]
    return {"bytes": n * (2 * _state_bytes(case["gen"]) + 4 + 3 * 4), "flops": n * _ops(case["gen"])}


# ------------------------------------------------------------------ the generators, from their definitions
def _splitmix(s):
    while True:
        s = (s + 0x9E3779B97F4A7C15) & M64
        z = s
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & M64
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & M64
        yield z ^ (z >> 31)


def _mulmod(a, b, p):
    """a * b mod p of int64 tensors below p."""
    if p == (1 << 61) - 1:
        lo, m = (1 << 31) - 1, (1 << 30) - 1
        a0, a1, b0, b1 = a & lo, a >> 31, b & lo, b >> 31
        mid = (a0 * b1) % p + (a1 * b0) % p
        r = (a0 * b0) % p + (2 * ((a1 * b1) % p)) % p
        return (r % p + ((mid >> 30) + ((mid & m) << 31)) % p) % p
    w = 61 - p.bit_length()  # pieces of b
    r = torch.zeros_like(a * b)
    for s in reversed(range(0, p.bit_length(), w)):
        r = ((r << w) + a * ((b >> s) & ((1 << w) - 1))) % p
    return r


def _matmul(X, Y, m):
    n = len(X)
    return [[sum(X[i][k] * Y[k][j] for k in range(n)) % m for j in range(n)] for i in range(n)]


def _matpow(M, e, m):
    R = [[int(i == j) for j in range(len(M))] for i in range(len(M))]
    while e:
        if e & 1:
            R = _matmul(R, M, m)
        M, e = _matmul(M, M, m), e >> 1
    return R


def _apply(mats, v, p):
    """mats: one matrix (Python integers) per row of v's first axis; v: [rows, dim, ...] -> the products."""
    d = len(mats[0])
    m = torch.tensor([[c for r in M for c in r] for M in mats], dtype=torch.int64, device=v.device)
    m = m.reshape(len(mats), d, d, *([1] * (v.dim() - 2)))
    return torch.stack([sum(_mulmod(m[:, i, k], v[:, k], p) for k in range(d)) % p for i in range(d)], 1)


def _spread(M, v, p, first, step, count, then):
    """Linear recurrence states at M^((first + j step)) v, j < count, then each at `then` = (length,
    sections) further section starts: [count * sections, dim, ...]."""
    v = _apply([_matpow(M, first, p)], v[None], p)
    J = _matpow(M, step, p)
    while v.shape[0] < count:  # doubling
        v = torch.cat([v, _apply([J], v, p)])[:max(count, 1)]
        J = _matmul(J, J, p)
    length, sections = then
    S, J = v, _matpow(M, length, p)
    parts = []
    for _ in range(sections):
        parts.append(S)
        S = _apply([J], S, p)
    return torch.stack(parts, 1).flatten(0, 1)


def _words(gen, seed, first, n, per, start=0):
    """u32 outputs start .. start + per - 1 of streams first .. first + n - 1 as an int64 tensor [n, per],
    or None where that takes too long here."""
    sec = 1
    while per > 2048 * sec and sec < 4096:
        sec *= 2
    length = -(-per // sec)
    if gen == "MT19937" or length > 8192 or n * sec * length > 1 << 31:
        return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    out = torch.empty((n * sec, length), dtype=torch.int64, device=dev)
    rng = _splitmix(seed)
    then = (length, sec)
    if gen == "MRG32K3A":
        m1, m2 = 2**32 - 209, 2**32 - 22853
        parts = []
        for m, M in ((m1, [[0, 1403580, m1 - 810728], [1, 0, 0], [0, 1, 0]]), (m2, [[527612, 0, m2 - 1370589], [1, 0, 0], [0, 1, 0]])):
            v = [next(rng) % m for _ in range(3)]
            v = torch.tensor(v, dtype=torch.int64, device=dev)
            parts.append(_spread(M, v, m, (first << 127) + start, 1 << 127, n, then))
        (x0, x1, x2), (y0, y1, y2) = (list(v.unbind(1)) for v in parts)
        for i in range(length):
            x0, x1, x2 = (1403580 * x1 - 810728 * x2) % m1, x0, x1
            y0, y1, y2 = (527612 * y0 - 1370589 * y2) % m2, y0, y1
            z = (x0 - y0) % m1
            out[:, i] = torch.where(z == 0, m1, z)
    elif gen == "LFSR113":
        out.zero_()
        for p, q, s in ((31, 6, 18), (29, 2, 2), (28, 13, 7), (25, 3, 13)):
            z = next(rng) >> 32
            while not z >> (32 - p):
                z = next(rng) >> 32
            mask = (0xFFFFFFFF << (32 - p)) & 0xFFFFFFFF

            def step(v):
                return (((v & mask) << s) & 0xFFFFFFFF) ^ ((((v << q) & 0xFFFFFFFF) ^ v) >> (p - s))

            def image(cols, v):  # GF(2) matrix by its columns, on an int or a tensor
                r = v & 0
                for b in range(32):
                    r = r ^ (((v >> b) & 1) * cols[b])
                return r

            def power(e):
                cols, res = [step(1 << b) for b in range(32)], [1 << b for b in range(32)]
                while e:
                    if e & 1:
                        res = [image(cols, c) for c in res]
                    cols, e = [image(cols, c) for c in cols], e >> 1
                return res

            v = torch.tensor([image(power((first << 34) + start), z)], dtype=torch.int64, device=dev)
            J = power(1 << 34)
            while v.shape[0] < n:
                v = torch.cat([v, image(J, v)])[:n]
                J = [image(J, c) for c in J]
            J, parts = power(length), []
            for _ in range(sec):
                parts.append(v)
                v = image(J, v)
            v = torch.stack(parts, 1).flatten()
            for i in range(length):
                v = step(v)
                out[:, i] ^= v
    else:
        s, v, k, q, p, L, nmax = GM[gen]
        a, b = next(rng) % p, next(rng) % p
        while not (a | b):
            a, b = next(rng) % p, next(rng) % p
        M = [[k, p - q], [1, 0]]
        pts = [_matpow(M, i * nmax * L, p) for i in range(s)]
        pts = [((m[0][0] * b + m[0][1] * a) % p, (m[1][0] * b + m[1][1] * a) % p) for m in pts]
        st = torch.tensor(pts, dtype=torch.int64, device=dev).T  # [2, points]
        st = _spread(M, st, p, first * L + start, L, n, then)
        zc, zp = st[:, 0], st[:, 1]
        at = torch.arange(s, device=dev) * v
        big = p > 1 << 60
        kt, qt = (torch.tensor(c, dtype=torch.int64, device=dev) for c in (k, q))
        for i in range(length):
            zn = (_mulmod(zc, kt, p) - _mulmod(zp, qt, p)) % p if big else (k * zc - q * zp) % p
            zp, zc = zc, zn
            if v == 1:
                strip = (zc >= (p + 1) // 2).long()
            else:
                strip = sum((zc >= -(-j * p // (1 << v))).long() for j in range(1, 1 << v))
            out[:, i] = torch.where(at < 32, strip << at.clamp(max=31), 0).sum(1) & 0xFFFFFFFF
    return out.reshape(n, sec * length)[:, :per]


def _float(gen, words, dtype):
    if dtype == "f32":
        return (words >> 8).double() * 2.0**-24
    return words.double() * (1.0 / (2**32 - 208)) if gen == "MRG32K3A" else words.double() * 2.0**-32


def exact(case, seed):
    s = _seed(seed)
    if case["kind"] in ("fill", "host"):
        if case["dtype"] == "u32":
            return None
        w = _words(case["gen"], s, _first(case, seed), case["streams"], case["per"])
        return None if w is None else _float(case["gen"], w, case["dtype"])
    if case["kind"] == "serve":
        outs = []
        for g, k, n, d in _serve_requests(case, seed):
            w = _words(g, s, k, 1, n) if d else None
            outs.append(None if w is None else _float(g, w, DTYPES[d])[0].cpu().numpy())
        return outs
    return None
