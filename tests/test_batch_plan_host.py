"""The tiles a batch is cut into, on the CPU: every output in one tile, sections
within the lengths the launch parameters ask for, and both parameters used."""
import os
import shutil
import subprocess

import pytest

import paper_1307_5869_gb300 as P
from paper_1307_5869_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
TC = 8   # kTileTc
SECTIONS = {"GM19": 4, "GM29": 4, "GM31": 4, "GM61": 4, "GQ58_1": 4, "GM55": 16, "GQ58_4": 16}


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("g++ not found")
    lib = B.build()
    exe = tmp_path_factory.mktemp("plan") / "plan"
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B.nvcc()))), "include")
    subprocess.run(["g++", "-std=c++17", "-w", os.path.join(HERE, "batch_plan.cpp"), "-I", B.CSRC, "-I", os.path.join(ROOT, "include"),
                    "-I", cuda, lib, f"-Wl,-rpath,{os.path.dirname(lib)}", "-o", str(exe)], check=True)

    def tiles(gen, length, mrg_lfsr=0, gm=0):
        r = subprocess.run([str(exe), str(P.GEN_ID[gen]), str(length), str(mrg_lfsr), str(gm)], capture_output=True, text=True, check=True)
        out = [tuple(map(int, line.split())) for line in r.stdout.splitlines()]
        at = 0
        for start, n, sec, _, to in out:
            assert start == at and n > 0 and to == 0x1000 + 4 * at, (gen, length)
            at += n
        assert at == length, (gen, length)
        return out

    return tiles


@pytest.mark.parametrize("gen", sorted(SECTIONS))
def test_tensor_core_sections_follow_the_parameter(plan, gen):
    n = SECTIONS[gen]
    for seclen in (0, 4, 64, 100, 2048, 8192, 32768, 2**32 - 4):
        most = -(-(seclen or 4096) // 64) * 64
        for length in (192, 193, 1000, n * 4096, n * 4096 + 1, 1 << 20, 3_000_001):
            for start, size, sec, flags, _ in plan(gen, length, 0, seclen):
                assert flags & TC and sec % 64 == 0 and 64 <= sec <= most and size <= n * sec
    assert len(plan(gen, 1 << 20, 0, 2048)) > len(plan(gen, 1 << 20, 0, 8192)) > len(plan(gen, 1 << 20, 0, 32768))


def test_short_requests_of_the_lane_per_point_generators(plan):
    for gen, line in (("GM19", 160), ("GM29", 192), ("GM31", 96), ("GM61", 120), ("GQ58_1", 96)):
        assert not plan(gen, line - 1)[0][3] & TC and plan(gen, line)[0][3] & TC
    for gen in ("GM55", "GQ58_4"):
        assert plan(gen, 1)[0][3] & TC
    assert not plan("GQ58_3", 100000)[0][3] & TC


def test_thread_sections_follow_the_other(plan):
    for gen in ("MRG32K3A", "LFSR113"):
        assert [len(plan(gen, 1 << 20, s)) for s in (2048, 8192, 32768)] == [16, 4, 1]
    assert plan("GQ58_3", 1 << 20, 8192)[0][2] == 512
