"""The staged row stores on a warp of 32 host threads: every row complete, no
write outside the rows, no output made that a row does not have, and every warp
operation met by all lanes together."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
HEADER = os.path.join(os.path.dirname(HERE), "paper_1307_5869_gb300", "csrc", "devcommon.cuh")


def test_rows_by_a_warp_of_host_threads(tmp_path):
    if not shutil.which("g++"):
        pytest.skip("g++ not found")
    text = open(HEADER).read()
    first = text.index("template <typename OutT, int ROWB = 128>\nstruct RowFill")
    last = text.index("// Whether a fill of n rows of nper outputs")
    (tmp_path / "fill_rows.inc").write_text(text[first:last])
    exe = tmp_path / "warp"
    subprocess.run(["g++", "-std=c++20", "-O1", "-w", "-pthread", "-I", str(tmp_path), os.path.join(HERE, "fill_rows_warp.cpp"),
                    "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout == "ok\n", r.stderr
