"""The float64 path's own functions against the host's long double on a million arguments
of their whole range: the exponential by table within 0.62 units in the last place (its
error analysis: 0.5 of the last addition, 0.1 of what enters it), r within 1 and 1/r
within 2; and zero, subnormal, infinite and NaN arguments as CUDA's functions."""
import os
import subprocess

import pytest

from gpu_helpers import torch_cuda

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")


def test_against_long_double(tmp_path):
    torch_cuda()
    exe = str(tmp_path / "fp64_math")
    csrc = os.path.join(ROOT, "paper_2512_07693_gb300", "csrc")
    r = subprocess.run([NVCC, "-std=c++17", "-O3", "-gencode", "arch=compute_103a,code=sm_103a", "-I" + csrc,
                        "-I" + os.path.join(ROOT, "include"), os.path.join(ROOT, "tests", "fp64_math.cu"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    out = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0
    lines = out.stdout.splitlines()
    e, r1, ir = (float(v) for v in lines[0].split())
    assert e <= 0.62 and r1 <= 1.0 and ir <= 2.0, lines[0]
    assert not lines[1:], lines[1:]
