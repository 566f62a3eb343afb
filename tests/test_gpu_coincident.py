"""Two atoms at exactly one place, where r = 0 and 1/r is infinite.

Float64: the EAM terms are finite (the taper is 1 there), so every per-atom energy and
the total are the oracle's, at the float64 path's 1e-9 relative to the pair's own
energy (Phi(0) is about 4e3 eV); the two atoms' forces have no direction and are NaN.
Float32: r = r^2 / r is NaN, and what depends on the pair says so: the two atoms'
energies, weights and lam are NaN and no other atom's."""
import numpy as np
import pytest

from gpu_helpers import to_dev, torch_cuda
from oracle import eam, neighbors
from paper_2512_07693_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _system():
    from paper_2512_07693_gb300 import apip
    s = W.config("void250k", apip.apip_ace_basis_size, scale=8)
    pos = s["pos"].copy()
    d = np.linalg.norm(neighbors.min_image(pos - pos[10], s["box"]), axis=1)
    d[10] = np.inf
    pair = [10, int(d.argmin())]
    pos[pair[0]] = pos[pair[1]]
    return dict(s, pos=pos), s, pair


def _run(s, perfect, precision, lam_mode):
    from paper_2512_07693_gb300 import apip
    torch = torch_cuda()
    t, n = to_dev(torch, s), len(s["pos"])
    box = [float(b) for b in s["box"]]
    m = apip.Apip(s["prm"], n, precision=precision, lam_mode=lam_mode)
    if lam_mode == "paper":
        m.init_csp_pairs(to_dev(torch, perfect)["pos"], box, t["ids"])
    F, e, E = (torch.empty(k, dtype=torch.float64, device="cuda") for k in ((n, 3), n, 1))
    m.energy_forces(t["pos"], box, t["types"], t["ids"], F, e, E)
    m.sync()
    out = {k: m.field(k, n).cpu().numpy() for k in ("wbar", "lam")}
    out.update(F=F.cpu().numpy(), e=e.cpu().numpy(), E=float(E))
    m.close()
    return out


def test_float64_energies_are_finite():
    s, perfect, pair = _system()
    g = _run(s, perfect, "fp64", "const0")
    p, n = W.EAM, len(s["pos"])
    i, _, _, r = neighbors.pairs_bruteforce(s["pos"], s["box"], p["rc"])
    zeta = np.bincount(i, weights=eam.rho(r, p), minlength=n)
    e = eam.xi(zeta) + 0.5 * np.bincount(i, weights=eam.phi(r, p), minlength=n)
    bar = 1e-9 * float(eam.phi(np.zeros(1), p)[0])
    assert np.abs(g["e"] - e).max() <= bar and abs(g["E"] - e.sum()) <= bar
    assert sorted(np.nonzero(np.isnan(g["F"]).any(axis=1))[0]) == sorted(pair)


def test_float32_says_nan():
    s, perfect, pair = _system()
    g = _run(s, perfect, "fp32", "paper")
    for k in ("e", "wbar", "lam"):
        assert sorted(np.nonzero(np.isnan(g[k]))[0]) == sorted(pair), k
