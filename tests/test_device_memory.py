"""CPU test of a float64 context's device memory against a fake CUDA runtime: the kept
pair terms are optional, so a device with just the memory that everything else needs,
and any with more, accepts the context and its box; a large device gets them, and the
learned switch, whose pass 1 keeps none, never does.  (The harness device_memory.cpp
compiles the library's context management; no device code runs.)"""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2512_07693_gb300", "csrc")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")


@pytest.mark.skipif(not os.path.exists(NVCC), reason="nvcc not found")
def test_optional_memory_never_refuses(tmp_path):
    exe = str(tmp_path / "device_memory")
    inc = ["-I" + os.path.join(ROOT, "include"), "-I" + CSRC]
    objs = [str(tmp_path / n) for n in ("harness.o", "apip.o", "tables.o")]
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(NVCC))), "include")
    for cmd in (["g++", "-std=c++17", "-O1", "-I" + cuda, *inc, "-c", os.path.join(ROOT, "tests", "device_memory.cpp"), "-o", objs[0]],
                [NVCC, "-std=c++17", "-O1", *inc, "-c", os.path.join(CSRC, "apip.cu"), "-o", objs[1]],
                [NVCC, "-std=c++17", "-O1", *inc, "-x", "cu", "-c", os.path.join(CSRC, "ace_tables.cpp"), "-o", objs[2]],
                [NVCC, "-cudart", "none", "-Xlinker", "--unresolved-symbols=ignore-all", *objs, "-o", exe, "-ldl"]):
        r = subprocess.run(cmd, capture_output=True, text=True)
        assert r.returncode == 0, r.stderr[-2000:]
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr
    paper, learned = ([int(v) for v in line.split()] for line in out.stdout.splitlines())
    assert paper[3] == 0 and learned[3] == 0, out.stdout
    assert paper[2] == 1 and learned[2] == 0
    assert learned[1] - paper[1] < 20000 * 16   # (the learned switch has one more list)
