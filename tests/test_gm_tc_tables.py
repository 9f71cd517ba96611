"""The constants of the GM/GQ tensor-core generation, on the CPU: the products
the kernel asks the tensor cores for, evaluated in exact integers from the
table the library builds, against the recurrence in Python integers.

For every step of a block: each partial sum of the product fits the exact
range of the accumulator, the fraction t built from the two digit columns gives
floor(2^v x / p) whenever it is not within the margin of a strip boundary (the
kernel computes those points again), and values on strip boundaries are always
inside that margin."""
import ctypes

import numpy as np
import pytest

import kernel_model as KM
import paper_1307_5869_gb300 as P

M = 64            # steps per block: two products of 32
M32 = (1 << 32) - 1
GENS = ["GM19", "GM29", "GM31", "GM55", "GM61", "GQ58_1", "GQ58_4"]
MARGIN = {"GM19": 212, "GM29": 314, "GM31": 314, "GM55": 62, "GM61": 82, "GQ58_1": 314, "GQ58_4": 37}
NIBBLES = ("GM55", "GM61", "GQ58_4")
# bit position and width of the limb in each slot of a value; the last slot is the bias's
SLOTS = {False: [(0, 8), (8, 8), (16, 8), (24, 8), None, None, None],
         True: [(0, 4), (8, 4), (16, 4), (24, 4), (4, 4), (12, 4), (20, 4), (28, 4),
                (32, 4), (40, 4), (48, 4), (56, 8), (36, 4), (44, 4), (52, 4)]}


class Table(ctypes.Structure):
    _fields_ = [("image", ctypes.c_uint8 * 4096 * 2), ("v", ctypes.c_uint64), ("q", ctypes.c_uint64),
                ("a", ctypes.c_uint64), ("b", ctypes.c_uint64), ("al", ctypes.c_uint64 * (M + 2)),
                ("be", ctypes.c_uint64 * (M + 2))]


def _table(gen):
    build = P.load(build_if_missing=True)._ZN5prand11gm_tc_buildEiPNS_9GmTcTableE
    build.restype = ctypes.c_bool
    t = Table()
    assert build(P.GEN_ID[gen], ctypes.byref(t))
    return t


def _columns(t, slots):
    """B of both products as integers [128 columns][slots], in units of 2^-20 per unit limb or per 1.0."""
    out = []
    for h in range(2):
        raw = np.frombuffer(bytes(t.image[h])[:64 * slots * 2], dtype=np.float16)
        b = raw.reshape(8, slots // 8, 8, 8).transpose(0, 2, 1, 3).reshape(64, slots).astype(np.float64)
        unit = np.full(slots, 2.0**-24)   # a limb f is the f16 subnormal f 2^-24
        unit[[slots // 2 - 1, slots - 1]] = 1.0   # the bias slots hold 1.0
        units = b * unit * 2.0**20
        assert np.array_equal(units, np.rint(units))
        out.append(units.astype(np.int64))
    return np.concatenate(out)


def _row(x, nibbles):
    f = [0 if s is None else (x >> s[0]) & ((1 << s[1]) - 1) for s in SLOTS[nibbles]]
    assert sum(v << s[0] for v, s in zip(f, SLOTS[nibbles]) if s) == x
    return f + [1]


def _values(gen, x_prev, x, count):
    k, q, p = KM.PARAMS[gen][:3]
    out = [x_prev, x]
    for _ in range(count):
        out.append((k * out[-1] - q * out[-2]) % p)
    return out   # x^(n-1), x^(n), x^(n+1), ...


def _step_of(v, c):
    h, g = divmod(c, 32)
    return 1 + (2 * (31 - g) + h if v == 1 else 32 * h + 4 * (7 - g % 8) + g // 8)


@pytest.mark.parametrize("gen", GENS)
def test_products_give_the_strips(gen):
    t = _table(gen)
    k, q, p, _, v, _, _ = KM.PARAMS[gen]
    nib, margin = gen in NIBBLES, MARGIN[gen]
    cols = _columns(t, 32 if nib else 16)
    rng = np.random.default_rng(61)
    pairs = [(int(rng.integers(0, p)), int(rng.integers(0, p))) for _ in range(60)]
    pairs += [(y, z) for z, y in KM.boundary_states(gen, rng)] + [(0, 1), (p - 1, p - 1), (1, 0)]
    flagged = 0
    for n, (xp, x) in enumerate(pairs):
        val = _values(gen, xp, x, 2 * M)
        x0, x1, x2 = val[1], val[1 + M], val[1 + 2 * M]
        assert (t.a * x0 + t.b * xp) % p == x1 and (t.v * x1 + t.q * x0) % p == x2
        for j in range(-1, M + 1):
            assert (t.al[j + 1] * x1 + t.be[j + 1] * x2) % p == val[1 + j]
        if x0 < 8:
            x0 += p   # a lazy residue stands for the same value
        prod = cols * np.array(_row(x0, nib) + _row(x1, nib), dtype=np.int64)
        big = prod == 3 << 22   # the bias of 1.5 2^23 units is one of the products
        assert np.array_equal(big.sum(1), np.ones(2 * M))
        # any subset of the others stays within 2^22 of it
        rest = np.where(big, 0, prod)
        assert rest.clip(min=0).sum(1).max() < 1 << 22 and rest.clip(max=0).sum(1).min() >= -(1 << 22)
        bits = 0x41400000 + rest.sum(1)   # the accumulator as a 32-bit word
        for c in range(M):
            tt = ((int(bits[2 * c]) << 20) + (int(bits[2 * c + 1]) << 8)) & M32
            want = val[1 + _step_of(v, c)] * (1 << v) // p
            near = ((tt << v) & M32) < 2 * margin << 8 + v
            flagged += near and n < 60
            if not near:
                assert tt >> (32 - v) == want, (n, c)
            frac = val[1 + _step_of(v, c)] * (1 << 32) / p  # distance to the nearest boundary, in 2^-32
            dist = min(frac % (1 << (32 - v)), -frac % (1 << (32 - v)))
            if dist < 0.5:
                assert near, (n, c)
    # the 60 random pairs' values, flagged with probability 2 margin / (2^24 / 2^v)
    expect = 60 * M * 2 * margin / 2**(24 - v)
    assert flagged <= expect + 6 * expect**0.5 + 1
