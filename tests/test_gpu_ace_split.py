"""Body order 4 in float32 without a group size asked for: the record-wise pool kernel
for small bases, the quadratic kernel for large ones, and on the bases between the two
(pools of 1 or 2 atoms, up to 32 768 functions) either by the number of compacted atoms.

- The atoms per block that the library reports say which evaluation a basis gets.
- On both sides of the line by atom count, and at one atom, forces and energies of the
  automatic evaluation agree with the pool kernel's (a group size asked for) at the
  float32 path's bars, 2e-4 eV/A and 1e-5 eV, and so does the total at the sum of the
  atoms' bars (the kernel that has no part in a call must add nothing to it)."""
import numpy as np
import pytest

from gpu_helpers import run_gpu, torch_cuda
from paper_2512_07693_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _system(basis, cells):
    from paper_2512_07693_gb300 import apip
    s = W.config("void250k", apip.apip_ace_basis_size, scale=cells)
    s["prm"]["ace"] = W.ace_params(*basis, 4, 2, apip.apip_ace_basis_size(*basis, 4))
    return s


@pytest.mark.parametrize("basis,quad", [((1, 4), False), ((4, 2), False), ((6, 3), False), ((4, 4), False),
                                        ((5, 4), True), ((7, 3), True), ((8, 4), True)])
def test_evaluation_by_basis(basis, quad):
    from paper_2512_07693_gb300 import apip
    torch_cuda()
    pool = {}
    for prec, g in (("fp32", 0), ("fp32", 8), ("fp32", 4), ("fp32", 2), ("fp32", 1)):
        try:
            m = apip.Apip(_system(basis, 7)["prm"], 100, precision=prec, lam_mode="const0", ace_group=g)
        except apip.ApipError:
            continue
        pool[g] = apip.apip_ace_info(m.ctx)
        m.close()
    auto = pool.pop(0)
    if quad:
        assert auto["group"] == 8 and 8 not in pool
    else:   # the very evaluation that the group size gives
        assert auto == pool[auto["group"]]


@pytest.mark.parametrize("basis,group", [((5, 4), 2), ((6, 4), 1)])
def test_both_sides_of_the_line(basis, group):
    torch = torch_cuda()
    line = torch.cuda.get_device_properties(0).multi_processor_count * group * 2 // 3
    s = _system(basis, 8)
    n = len(s["pos"])
    order = np.random.default_rng(3).permutation(n)
    for count in (1, line, line + 1):
        lam = np.zeros(n)
        lam[order[:count]] = 0.75
        kw = dict(precision="fp32", lam_mode="const0", lam_fixed=lam, fields=False)
        a, b = run_gpu(s, **kw), run_gpu(s, ace_group=group, **kw)
        assert np.abs(a["F"] - b["F"]).max() <= 2e-4, count
        assert np.abs(a["e_atom"] - b["e_atom"]).max() <= 1e-5, count
        assert abs(a["E"] - b["E"]) <= 1e-5 * n, count
        for r in (a, b):
            r["model"].close()
