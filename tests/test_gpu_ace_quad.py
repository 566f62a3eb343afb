"""The quadratic ACE kernel (body order 4, float32) over the shapes of its tables:
one radial function or one degree only, tiles with a remainder, the largest basis;
atom counts that leave the last group of 8 with one to seven atoms, and fewer than 8
atoms in all.  Against the float64 path (the record-wise pool kernel, pinned to the
oracle at 1e-9 in test_gpu_parity.py) at the float32 path's bars, 2e-4 eV/A and 1e-5 eV
per atom; the record-wise kernel in float32 (a group size asked for) at the same bars."""
import numpy as np
import pytest

from gpu_helpers import run_gpu
from paper_2512_07693_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _system(n_max, l_max, drop):
    from paper_2512_07693_gb300 import apip
    pos, box = W.bcc(6, 6, 6)
    rng = np.random.default_rng(17)
    pos = np.delete(pos, rng.choice(len(pos), drop, replace=False), axis=0)
    pos = W.displace(pos, 0.06, 5)
    s = W._finish(pos, np.zeros_like(pos), box)
    nb = apip.apip_ace_basis_size(n_max, l_max, 4)
    s["prm"] = dict(precise_adds_eam=True, eam=dict(W.EAM), csp=dict(W.CSP),
                    switch=dict(W.SWITCH, d_lo=0.25, d_hi=0.9), ace=W.ace_params(n_max, l_max, 4, 2, nb))
    return s


@pytest.mark.parametrize("n_max,l_max,drop,lam_mode", [
    (1, 0, 1, "const1"), (1, 4, 2, "const1"), (8, 0, 3, "paper"), (2, 1, 4, "const1"), (3, 2, 5, "paper"),
    (5, 3, 6, "const1"), (7, 4, 7, "paper"), (8, 4, 1, "const1")])
def test_shapes_against_float64(n_max, l_max, drop, lam_mode):
    s = _system(n_max, l_max, drop)
    a, b, c = (run_gpu(s, precision=p, lam_mode=lam_mode, ace_group=k, fields=False)
               for p, k in (("fp32", 0), ("fp64", 0), ("fp32", 1)))
    for x in (a, c):
        assert np.abs(x["F"] - b["F"]).max() <= 2e-4
        assert np.abs(x["e_atom"] - b["e_atom"]).max() <= 1e-5


def test_few_atoms():
    """Three compacted atoms in one group of eight."""
    s = _system(4, 4, 1)
    lam = np.zeros(len(s["pos"]))
    lam[[5, 77, 301]] = 0.5
    a, b = (run_gpu(s, precision=p, lam_mode="const0", lam_fixed=lam, fields=False) for p in ("fp32", "fp64"))
    assert np.abs(a["F"] - b["F"]).max() <= 2e-4 and np.abs(a["e_atom"] - b["e_atom"]).max() <= 1e-5
