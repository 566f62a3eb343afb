"""CPU test of the rounding of the quadratic ACE kernel's sums (body order 4, float32):
on the densities of a crack's faces and of a hot vacancy crystal, phi_1 and phi_2 as the
kernel adds them (its tables' column order included) are no further from 64 bits than
the record-wise kernel's compensated sums, and nearer than with the columns by their
index.  Everything is seeded; the harness
(quad_sums.cu) is compiled with the library's table builder and runs no device code."""
import os
import subprocess

import numpy as np
import pytest

from oracle import ace, neighbors
from paper_2512_07693_gb300 import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2512_07693_gb300", "csrc")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")


def _densities(kind, n_max, l_max):
    rng = np.random.default_rng(0)
    if kind == "crack":
        s = W.crack_slab(nx=24, ny=12, nz=7)
        pos, box = s["pos"], s["box"]
        sel = np.nonzero((np.abs(pos[:, 1] - box[1] / 2) < 4) & (pos[:, 0] < box[0] / 2))[0]
    else:
        s = W.vacancy_crystal(cells=8, sigma=0.1, seed=5)
        pos, box = s["pos"], s["box"]
        sel = np.arange(len(pos))
    i, _, rvec, r = neighbors.pairs(pos, box, 5.0)
    model = ace.AceModel.__new__(ace.AceModel)
    model.p = dict(n_max=n_max, l_max=l_max, rc=5.0, rc_width=1.0, a_scale=0.25)
    return model.densities(len(pos), i, rvec, r)[0][rng.permutation(sel)[:150]].astype(np.float32)


@pytest.mark.skipif(not os.path.exists(NVCC), reason="nvcc not found")
def test_no_further_from_64_bits_than_the_records(tmp_path):
    exe = str(tmp_path / "quad_sums")
    cmd = [NVCC, "-std=c++17", "-O1", "-Xcompiler", "-ffp-contract=off", "-I" + os.path.join(ROOT, "include"),
           "-I" + CSRC, "-x", "cu", os.path.join(ROOT, "tests", "quad_sums.cu"), os.path.join(CSRC, "ace_tables.cpp"),
           "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    for kind in ("crack", "vacancy"):
        for n_max, l_max in ((8, 4), (5, 3)):
            path = str(tmp_path / "A.bin")
            _densities(kind, n_max, l_max).tofile(path)
            out = subprocess.run([exe, str(n_max), str(l_max), path], capture_output=True, text=True, timeout=300)
            assert out.returncode == 0
            a = np.array([[float(x) for x in line.split()] for line in out.stdout.splitlines()])
            assert len(a) == 150
            records, quad, by_index = np.sqrt((a ** 2).mean(axis=0)).reshape(3, 2)
            assert (quad <= records).all() and (quad < by_index).all(), (kind, n_max, l_max, records, quad, by_index)
