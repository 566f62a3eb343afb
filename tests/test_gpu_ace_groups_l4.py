"""The streamed ACE kernel with l_max = 4 and a large basis (8/4, 1274 couplings), where
each number of atoms per block has a kernel of its own and the count picks one: both
sides of every line of the rule and one atom against a fixed group of 8 (bars: the
float64 path's 1e-9 eV/A and eV, the float32 path's 2e-4 eV/A and 1e-5 eV; totals at the
sum of the atoms' bars: a kernel that is not picked must add nothing), and the time
of the automatic choice against the fixed groups: no more than 1.2 times the best."""
import numpy as np
import pytest

from gpu_helpers import run_gpu, to_dev, torch_cuda
from paper_2512_07693_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _system(cells):
    from paper_2512_07693_gb300 import apip
    s = W.config("void250k", apip.apip_ace_basis_size, scale=cells)
    s["prm"]["ace"] = W.ace_params(8, 4, 3, 2, apip.apip_ace_basis_size(8, 4, 3))
    return s, np.random.default_rng(3).permutation(len(s["pos"]))


@pytest.mark.parametrize("prec,tol_f,tol_e", [("fp32", 2e-4, 1e-5), ("fp64", 1e-9, 1e-9)])
def test_rule_edges(prec, tol_f, tol_e):
    torch = torch_cuda()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    s, order = _system(14)
    n = len(s["pos"])
    edges = (0, 4 * sms, 8 * sms, 16 * sms) if prec == "fp32" else (0, sms * 2 // 3 * 2, sms * 2 // 3 * 8, 16 * sms)
    for count in sorted({e + d for e in edges for d in (0, 1)} - {0}):
        lam = np.zeros(n)
        lam[order[:min(count, n)]] = 0.75
        kw = dict(precision=prec, lam_mode="const0", lam_fixed=lam, fields=False, max_nb=80)
        a, b = run_gpu(s, **kw), run_gpu(s, ace_group=8, **kw)
        assert np.abs(a["F"] - b["F"]).max() <= tol_f, count
        assert np.abs(a["e_atom"] - b["e_atom"]).max() <= tol_e, count
        assert abs(a["E"] - b["E"]) <= n * tol_e, count
        for r in (a, b):
            r["model"].close()


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_choice_is_near_the_best(prec):
    from paper_2512_07693_gb300 import apip
    torch = torch_cuda()
    s, order = _system(16)
    t, n, box = to_dev(torch, s), len(s["pos"]), [float(b) for b in s["box"]]
    lam = np.zeros(n)
    lam[order[:2 * torch.cuda.get_device_properties(0).multi_processor_count]] = 0.75
    F = torch.empty((n, 3), dtype=torch.float64, device="cuda")
    took = {}
    for group in (0, 4, 8, 32):
        m = apip.Apip(s["prm"], n, precision=prec, lam_mode="paper", max_nb=80, ace_group=group)
        m.set_lam_fixed(torch.tensor(lam, device="cuda"))
        m.init_csp_pairs(t["pos"], box, t["ids"])
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(22)]
        for k in range(25):
            m.energy_forces(t["pos"], box, t["types"], t["ids"], F)
            if k >= 3:
                ev[k - 3].record()
        m.sync()
        took[group] = float(np.median([a.elapsed_time(b) for a, b in zip(ev, ev[1:])]))
        m.close()
    assert took[0] <= 1.2 * min(took[g] for g in (4, 8, 32)), took
