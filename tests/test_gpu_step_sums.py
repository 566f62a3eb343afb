"""The step's float64 sums (total energy, kinetic energy, momentum), which many
small blocks and a last one add up, at atom counts around the edges of their
partials: one partial, one per warp, one block, several blocks.

Tolerance: each value is a compensated float64 sum of exact per-atom terms, so it
agrees with another float64 order of summation to a few rounding errors of the
largest partial sum: 1e-12 of the sum of magnitudes."""
import numpy as np
import pytest

from gpu_helpers import to_dev, torch_cuda


@pytest.mark.gpu
@pytest.mark.parametrize("cells,drop", [(6, 0), (16, 1), (21, 300), (26, 7)])
def test_sums_against_torch(cells, drop):
    torch = torch_cuda()
    from paper_2512_07693_gb300 import apip, workloads as W
    s = W.vacancy_crystal(cells=cells, sigma=0.04, seed=3, temp=300.0)
    prm = W.config("vacancy2k", apip.apip_ace_basis_size, scale=6)["prm"]
    t = {k: v[drop:].contiguous() for k, v in to_dev(torch, s).items()}
    n = t["pos"].shape[0]
    ids = torch.arange(n, dtype=torch.int32, device="cuda")
    box = [float(b) for b in s["box"]]
    m = apip.Apip(prm, n, precision="fp64", lam_mode="const0")
    F = torch.empty((n, 3), dtype=torch.float64, device="cuda")
    e = torch.empty(n, dtype=torch.float64, device="cuda")
    E = torch.zeros(1, dtype=torch.float64, device="cuda")
    for _ in range(2):   # the second call finds the first one's scratch
        m.energy_forces(t["pos"], box, t["types"], ids, F, e, E)
        m.sync()
        assert abs(float(E) - float(e.sum())) <= 1e-12 * float(e.abs().sum())
    steps = 3
    thermo = torch.zeros((steps, 5), dtype=torch.float64, device="cuda")
    rows = []
    pos, vel, force = t["pos"].clone(), t["vel"].clone(), F.clone()
    for k in range(steps):   # one step per call: the state after each step is at hand
        m.verlet_step(pos, vel, force, t["inv_mass"], box, t["types"], ids, 0.001, 1, thermo[k:k + 1])
        m.sync()
        p = vel / t["inv_mass"][:, None]
        rows.append([float(0.5 * (vel * p).sum()), *[float(x) for x in p.sum(0)]])
        scale = float(0.5 * (vel * p).abs().sum()), *[float(x) for x in p.abs().sum(0)]
        got = thermo[k].cpu().numpy()
        for q in range(4):
            assert abs(got[1 + q] - rows[k][q]) <= 1e-12 * scale[q]
        m.energy_forces(pos, box, t["types"], ids, F, e, E)
        m.sync()
        assert abs(got[0] - float(E)) <= 1e-11 * abs(float(E))
    many = torch.zeros_like(thermo)
    m.verlet_step(t["pos"], t["vel"], _forces(m, t, box, ids, torch), t["inv_mass"], box,
                  t["types"], ids, 0.001, steps, many)
    m.sync()
    assert np.allclose(many.cpu().numpy()[:, :2], thermo.cpu().numpy()[:, :2], rtol=1e-11, atol=0.0)
    m.close()


def _forces(m, t, box, ids, torch):
    F = torch.empty_like(t["pos"])
    m.energy_forces(t["pos"], box, t["types"], ids, F)
    return F
