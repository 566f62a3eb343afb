"""The streamed ACE kernel picks its atoms per block (2, 4, 8, 32) by the number of
compacted atoms: both sides of every line of that rule (which depends on the SM count,
2 SMs, 4 and 16 resident blocks), and one atom, against a fixed group of 8.

Bars: the float64 path's 1e-9 eV/A and eV, the float32 path's 2e-4 eV/A and 1e-5 eV."""
import numpy as np
import pytest

from gpu_helpers import run_gpu, torch_cuda
from paper_2512_07693_gb300 import apip, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol_f,tol_e", [("fp32", 2e-4, 1e-5), ("fp64", 1e-9, 1e-9)])
def test_group_rule_edges(prec, tol_f, tol_e):
    torch = torch_cuda()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    s = W.config("void250k", apip.apip_ace_basis_size, scale=16)
    n = len(s["pos"])
    order = np.random.default_rng(3).permutation(n)
    for edge in (1, 2 * sms, 8 * sms, 32 * sms):
        for count in (edge, edge + 1):
            lam = np.zeros(n)
            lam[order[:min(count, n)]] = 0.75
            kw = dict(precision=prec, lam_mode="const0", lam_fixed=lam, fields=False, max_nb=80)
            a, b = run_gpu(s, **kw), run_gpu(s, ace_group=8, **kw)
            assert np.abs(a["F"] - b["F"]).max() <= tol_f, count
            assert np.abs(a["e_atom"] - b["e_atom"]).max() <= tol_e, count
            for r in (a, b):
                r["model"].close()
