"""CPU test of the quadratic ACE tables (body order 4, float32) and of the host check that
apip_create runs on them: the forms give the record-wise tables' phi (double, 1e-12 of the
sum of magnitudes), valid tables pass and one bad entry of each kind fails.  The harness
(quad_table_check.cu) is compiled with the library's table builder."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2512_07693_gb300", "csrc")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")


@pytest.mark.skipif(not os.path.exists(NVCC), reason="nvcc not found")
def test_quad_table_check(tmp_path):
    exe = str(tmp_path / "quad_table_check")
    cmd = [NVCC, "-std=c++17", "-O1", "-I" + os.path.join(ROOT, "include"), "-I" + CSRC, "-x", "cu",
           os.path.join(ROOT, "tests", "quad_table_check.cu"), os.path.join(CSRC, "ace_tables.cpp"), "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr
    lines = dict(line.split() for line in out.stdout.splitlines())
    assert len(lines) == 2 * 6 + 14
    assert [k for k, v in lines.items() if v != "ok"] == []
