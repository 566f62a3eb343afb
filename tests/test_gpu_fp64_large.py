"""The float64 path with one thread per atom (from 4 x 64 atoms per SM on), which takes the
exponential by table, its own blocks and the one-thread list fill: a small crystal, where
eight threads share an atom, tiled until it is large gives every copy the small one's
energies, forces and lam at float64's 1e-9; also with more pairs within the EAM cutoff
than are kept from pass 1 for pass 2, and against the oracle.  And the list of an atom
with exactly max_nb neighbours and one more atom just beyond r_list (within the fill's
first, wider test)."""
import numpy as np
import pytest

from gpu_helpers import run_oracle, to_dev, torch_cuda
from paper_2512_07693_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _large(torch, per):   # copies along each axis for one thread per atom
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    k = 1
    while k ** 3 * per <= 256 * sms:
        k += 1
    return k


def _run(torch, s, **kw):
    from paper_2512_07693_gb300 import apip
    t, n, box = to_dev(torch, s), len(s["pos"]), [float(b) for b in s["box"]]
    m = apip.Apip(s["prm"], n, precision="fp64", lam_mode="paper", **kw)
    m.init_csp_pairs(t["pos"], box, t["ids"])
    F, e = torch.empty_like(t["pos"]), torch.empty(n, dtype=torch.float64, device="cuda")
    m.energy_forces(t["pos"], box, t["types"], t["ids"], F, e)
    m.sync()
    out = dict(F=F.cpu().numpy(), e_atom=e.cpu().numpy(), lam=m.field("lam", n).cpu().numpy())
    m.close()
    return out


def _tile(s, k):
    shift = np.array([(x, y, z) for x in range(k) for y in range(k) for z in range(k)]) * s["box"]
    pos = (shift[:, None, :] + s["pos"][None]).reshape(-1, 3)
    return dict(s, **{q: v for q, v in W._finish(pos, np.zeros_like(pos), k * s["box"]).items()})


@pytest.mark.parametrize("eam_rc,kw", [(4.4, dict(max_nb=80)), (5.0, dict(skin=0.1, max_nb=72))])
def test_every_copy_as_the_small_crystal(eam_rc, kw):
    from paper_2512_07693_gb300 import apip
    torch = torch_cuda()
    s = W.vacancy_crystal(cells=7, sigma=0.06, seed=9)
    s["prm"] = dict(precise_adds_eam=True, eam=dict(W.EAM, rc=eam_rc), csp=dict(W.CSP), switch=dict(W.SWITCH, d_lo=0.25, d_hi=0.9),
                    ace=W.ace_params(4, 2, 3, 2, apip.apip_ace_basis_size(4, 2, 3)))
    k, n = _large(torch, len(s["pos"])), len(s["pos"])
    small, large = _run(torch, s, **kw), _run(torch, _tile(s, k), **kw)
    ref = run_oracle(s)
    for q, o in (("F", ref["F"]), ("e_atom", ref["e_atom"]), ("lam", ref["lam"])):
        assert np.abs(small[q] - o).max() <= 1e-9, q
        assert np.abs(large[q].reshape((k ** 3,) + small[q].shape) - small[q]).max() <= 1e-9, q


@pytest.mark.parametrize("large", [False, True])
def test_list_at_its_capacity(large):
    from paper_2512_07693_gb300 import apip
    torch = torch_cuda()
    r_list = 5.5
    # a centre with five neighbours that see only it, and one atom just beyond r_list
    cluster = np.array([[0, 0, 0], [3.0, 0, 0], [0, 5.2, 0], [-4.6, 0, 0], [0, -5.3, 0], [0, 0, 5.4], [0, 0, -r_list * (1 + 1e-5)]])
    k = _large(torch, 7) if large else 2
    grid = np.array([(x, y, z) for x in range(k) for y in range(k) for z in range(k)]) * 20.0 + 10.0
    pos = (grid[:, None, :] + cluster[None]).reshape(-1, 3)
    s = W._finish(pos, np.zeros_like(pos), np.array([20.0 * k] * 3))
    prm = dict(precise_adds_eam=True, eam=dict(W.EAM), csp=dict(W.CSP), switch=dict(W.SWITCH),
               ace=W.ace_params(1, 0, 1, 2, apip.apip_ace_basis_size(1, 0, 1)))
    t, n, box = to_dev(torch, s), len(pos), [float(b) for b in s["box"]]
    m = apip.Apip(prm, n, precision="fp64", lam_mode="const0", max_nb=5)
    m.build_neighbors(t["pos"], box, t["ids"])
    m.sync()
    nnb, nbl = m.field("nnb", n).cpu().numpy(), m.field("nblist", n).cpu().numpy()
    m.close()
    want = np.array([5, 1, 1, 1, 1, 1, 0])
    assert np.array_equal(nnb.reshape(-1, 7), np.tile(want, (k ** 3, 1)))
    c = 7 * np.arange(k ** 3)
    centre = nbl.reshape(-1, 7, 5)[:, 0] - c[:, None]
    assert np.array_equal(centre[:, :2], np.tile([1, 3], (k ** 3, 1)))   # within the EAM cutoff, within its skin
    assert np.array_equal(np.sort(centre[:, 2:], axis=1), np.tile([2, 4, 5], (k ** 3, 1)))
    assert np.array_equal(nbl.reshape(-1, 7, 5)[:, 1:6, 0], np.tile(c[:, None], (1, 5)))
