"""Workloads by which the library's speed is measured, through its public entry points.

Every case is a plain dict; ``prepare`` makes what a program holds before the
call (seeded inputs on the GPU, a context with its pair list and network), ``run``
is one pass of that program, ``work`` what the pass cannot do without, and
``exact`` the same results in float64 from plain torch operations.

The kinds of case, after the programs of this package:
  md      ``steps`` velocity-Verlet steps with their thermo rows: positions, velocities,
          forces and the thermo rows come back, and the next pass goes on from there
  ef      energy, per-atom energies and forces of two snapshots of one system (single
          points along a path: the positions differ, so each needs a new list)
  labels  training labels and bfloat16 descriptors of a few defect crystals through
          one context, every atom with the precise model
  train   one optimiser step of the indicator network on the next of four batches
and the systems: ``vacancy``, ``void``, ``crack`` and ``slab`` (under an indenter), sized by ``cells``.
"""
import functools
import math

import numpy as np
import torch

from paper_2512_07693_gb300 import apip
from paper_2512_07693_gb300 import workloads as W

DT = 0.001                       # ps
N6L3 = dict(n_max=6, l_max=3, nu_max=3)
N8L4 = dict(n_max=8, l_max=4, nu_max=4)
LABEL_REF = 0.718                # eV/atom, the models' difference in the perfect lattice


def listed():
    return [
        # the accuracy reference: a small crystal in float64, latency above all
        dict(name="md_vacancy2k_fp64", kind="md", system="vacancy", cells=10, precision="fp64", lam="paper", steps=10),
        # training labels: small crystals one after the other, each with a new list
        dict(name="labels_2k", kind="labels", cells=10, configs=4),
        # a mid-sized adaptive run
        dict(name="md_void27k", kind="md", system="void", cells=24, precision="fp32", lam="paper", steps=10),
        # the benchmark's crystal: adaptive float32 run
        dict(name="md_void250k", kind="md", system="void", cells=50, precision="fp32", lam="paper", steps=10),
        # ... single points of it, where every call builds a list
        dict(name="ef_void250k", kind="ef", system="void", cells=50, precision="fp32", lam="paper", adds_eam=True),
        # ... in float64
        dict(name="md_void250k_fp64", kind="md", system="void", cells=50, precision="fp64", lam="paper", steps=4),
        # ... with the precise model on every atom
        dict(name="md_void250k_all_ace", kind="md", system="void", cells=50, precision="fp32", lam="const1", steps=2),
        # the cracked slab: two million atoms, body order 4 on the crack's faces
        dict(name="md_crack2m", kind="md", system="crack", cells=100, precision="fp32", lam="paper", steps=1),
        # the indentation run: four million atoms under the indenter
        dict(name="md_slab4m", kind="md", system="slab", cells=160, precision="fp32", lam="paper", steps=4),
        # the same slab at a quarter of the size with the learned switch
        dict(name="md_slab900k_learned", kind="md", system="slab", cells=96, precision="fp32", lam="learned", steps=4),
        # one optimiser step at the training run's batch size
        dict(name="train_64k", kind="train", batch=65536),
        # ... and at the end of an epoch of a small set, a ragged batch
        dict(name="train_3k", kind="train", batch=3001),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.randrange(8)
    if what == 0:
        return dict(kind="train", batch=_log_int(rng, 300, 65536))
    if what == 1:
        return dict(kind="labels", cells=rng.randint(7, 16), configs=rng.randint(1, 5))
    if what == 2:
        return dict(kind="md", system="crack", cells=_log_int(rng, 20, 90), precision="fp32", lam="paper", steps=1)
    if what == 3:
        return dict(kind="md", system="slab", cells=_log_int(rng, 24, 150), precision="fp32", lam="paper",
                    steps=rng.randint(2, 5))
    if what == 4:
        return dict(kind="md", system="slab", cells=_log_int(rng, 24, 90), precision="fp32", lam="learned",
                    steps=rng.randint(1, 4))
    if what == 5:
        return dict(kind="ef", system="void", cells=_log_int(rng, 8, 60), precision=rng.choice(["fp32", "fp64"]),
                    lam=rng.choice(["paper", "const1"]), adds_eam=rng.random() < 0.5)
    if what == 6:
        return dict(kind="md", system=rng.choice(["void", "vacancy"]), cells=_log_int(rng, 8, 50), precision="fp64",
                    lam="paper", steps=rng.randint(2, 6))
    return dict(kind="md", system="void", cells=_log_int(rng, 10, 110), precision="fp32",
                lam=rng.choice(["paper", "paper", "const0"]), steps=rng.randint(4, 12))


# ------------------------------------------------------------------- inputs
def _bcc(nx, ny, nz, dev):
    a = W.LATTICE_A
    ax = [torch.arange(k, dtype=torch.float64, device=dev) for k in (nx, ny, nz)]
    g = torch.stack(torch.meshgrid(*ax, indexing="ij"), dim=-1).reshape(-1, 1, 3)
    off = torch.tensor([[0.0, 0.0, 0.0], [0.5, 0.5, 0.5]], dtype=torch.float64, device=dev)
    return ((g + off) * a).reshape(-1, 3), [nx * a, ny * a, nz * a]


def _normal(shape, sigma, gen):
    return torch.randn(shape, generator=gen, dtype=torch.float64, device=gen.device) * sigma


def _maxwell(n, temp, gen):
    v = _normal((n, 3), math.sqrt(W.KB_EV * temp / (W.MASS_AMU * W.MVV2E)), gen)
    return v - v.mean(dim=0)


def _wrap(pos, box):
    b = torch.tensor(box, dtype=torch.float64, device=pos.device)
    return pos - b * torch.floor(pos / b)


def _system(case, seed, dev="cuda"):
    """Sites (snapshot 0's positions), velocities, box, constant lam and indenter of a system."""
    gen = torch.Generator(device=dev).manual_seed(int(seed))
    s, c = case["system"], case["cells"]
    lam_fixed, indenter, vac, sigma = None, None, 0.0, 0.03
    if s == "vacancy":
        pos, box = _bcc(c, c, c, dev)
        keep = torch.ones(len(pos), dtype=torch.bool, device=dev)
        keep[torch.randint(len(pos), (1,), generator=gen, device=dev)] = False
        pos, sigma = pos[keep], 0.05
    elif s == "void":
        pos, box = _bcc(c, c, c, dev)
        mid = torch.tensor(box, dtype=torch.float64, device=dev) / 2
        pos = pos[((pos - mid) ** 2).sum(1) >= (15.0 * c / 50.0) ** 2]
    elif s == "crack":
        pos, box = _bcc(2 * c, c, c // 2, dev)
        h = torch.clamp(2.0 * (1.0 - pos[:, 0] / (0.5 * box[0])), min=0.0)
        pos = pos[(pos[:, 1] - 0.5 * box[1]).abs() >= 0.5 * h]
        vac = 15.0
        z = pos[:, 2]
        lam_fixed = (z < 3.0) | (z > z.max() - 3.0)
    else:
        pos, box = _bcc(c, c, max(78 * c // 160, 8), dev)
        radius = 40.0 * c / 160.0
        vac = 2.0 * radius + 15.0
        z = pos[:, 2]
        axis = [0.5 * box[0], 0.5 * box[1]]
        lateral = torch.sqrt((pos[:, 0] - axis[0]) ** 2 + (pos[:, 1] - axis[1]) ** 2)
        lam_fixed = (z < 3.0) | ((z > z.max() - 3.0) & (lateral > radius + 10.0))
        indenter = dict(center=[axis[0], axis[1], float(z.max()) + 0.5 * vac + radius],
                        velocity=[0.0, 0.0, -0.1], radius=radius, k=10.0)
    box[2] += vac
    shift = torch.tensor([0.0, 0.0, 0.5 * vac], dtype=torch.float64, device=dev)
    n = len(pos)
    snaps = [_wrap(pos + shift + _normal((n, 3), sigma, gen), box)]
    if case["kind"] == "ef":    # ... and sheared by a long wave
        wave = torch.zeros_like(pos)
        wave[:, 0] = 0.35 * torch.sin(2 * math.pi * pos[:, 1] / box[1])
        snaps.append(_wrap(pos + wave + _normal((n, 3), sigma, gen), box))
    if lam_fixed is not None:
        lam_fixed = torch.where(lam_fixed, 0.0, math.nan).to(torch.float64)
    return dict(snaps=snaps, vel=_maxwell(n, 300.0, gen), box=[float(b) for b in box], n=n, lam_fixed=lam_fixed,
                indenter=indenter)


@functools.lru_cache(maxsize=4)
def _ace(n_max, l_max, nu_max):
    return W.ace_params(n_max, l_max, nu_max, 2, apip.apip_ace_basis_size(n_max, l_max, nu_max))


def _params(case):
    sw = dict(W.SWITCH)
    if case.get("system") == "vacancy":
        sw.update(d_lo=1.2, d_hi=2.2)
    if case.get("lam") == "learned":
        sw.update(d_lo=0.25, d_hi=0.6)
    form = N8L4 if case.get("system") == "crack" else N6L3
    return dict(precise_adds_eam=case.get("adds_eam", True), eam=dict(W.EAM), switch=sw, csp=dict(W.CSP),
                ace=dict(_ace(**form)))


@functools.lru_cache(maxsize=1)
def _network():
    """A network that tells surface atoms (output near 1) from bulk atoms (near 0): seeded
    hidden layers, the output layer fitted to a small slab's descriptors."""
    w = W.mlp_params(7)
    gen = torch.Generator().manual_seed(11)
    pos, box = _bcc(6, 6, 12, "cpu")
    z = pos[:, 2]
    top = ((z < 2.0) | (z > z.max() - 2.0)).to(torch.float64)
    box[2] += 15.0
    pos = pos + _normal(pos.shape, 0.05, gen)
    d = pos[None] - pos[:, None]
    b = torch.tensor(box, dtype=torch.float64)
    d = d - b * torch.round(d / b)
    r = torch.sqrt((d * d).sum(-1)) + 1e3 * torch.eye(len(pos), dtype=torch.float64)
    h = _hidden(_features(r).sum(1), {k: torch.tensor(np.asarray(v)) for k, v in w.items()})[-1]
    h1 = torch.cat([h, torch.ones(len(h), 1, dtype=torch.float64)], dim=1)
    sol = torch.linalg.solve(h1.T @ h1 + 1e-5 * torch.eye(65, dtype=torch.float64), h1.T @ top)
    w.update(w4=sol[:64].numpy(), b4=float(sol[64]))
    return torch.tensor(apip.mlp_flat(w))


def _batches(case, seed):
    """Descriptors (bfloat16) and labels of four batches of thermal defect crystals."""
    n = case["batch"]
    cells = max(8, math.ceil((4 * n / 2) ** (1 / 3)) + 1)
    sysd = _system(dict(kind="md", system="void", cells=cells), seed)
    pos = sysd["snaps"][0]
    pos = pos + _normal(pos.shape, 0.05, torch.Generator(device="cuda").manual_seed(int(seed) + 5))
    nb = _neighbours(pos, sysd["box"], 5.0)
    G = torch.cat([_features(_dist(pos, nb, sysd["box"], q)[1]).sum(1) for q in _chunks(len(pos), 50000)])
    perm = torch.randperm(len(G), generator=torch.Generator(device="cuda").manual_seed(int(seed)), device="cuda")[:4 * n]
    G = G[perm]
    y = 0.05 + 0.02 * (G[:, 9] - 8.0 * G[:, 3] - 3.0).abs() / (1.0 + G[:, 20])
    return G.to(torch.bfloat16).contiguous(), y.to(torch.float32).contiguous()


def _crystals(case, seed, dev="cuda"):
    """Positions and box of thermal crystals with one to three point defects, vacancies and
    octahedral interstitials in turn."""
    gen = torch.Generator(device=dev).manual_seed(int(seed))
    c, out = case["cells"], []
    for k in range(case["configs"]):
        pos, box = _bcc(c, c, c, dev)
        for q in range(1 + k % 3):
            if (k + q) % 2 == 0:
                drop = int(torch.randint(len(pos), (1,), generator=gen, device=dev))
                pos = torch.cat([pos[:drop], pos[drop + 1:]])
            else:
                cell = torch.randint(c, (1, 3), generator=gen, device=dev).to(torch.float64)
                face = torch.tensor([[0.5, 0.5, 0.0]], dtype=torch.float64, device=dev)
                pos = torch.cat([pos, (cell + face) * W.LATTICE_A])
        temp = 300.0 + 900.0 * float(torch.rand((), generator=gen, dtype=torch.float64, device=dev))
        out.append(_wrap(pos + _normal(pos.shape, 0.05 * math.sqrt(temp / 300.0), gen), box))
    return out, [float(b) for b in box]


def prepare(case, seed):
    dev = torch.device("cuda")
    kind = case["kind"]
    if kind == "train":
        G, y = _batches(case, seed)
        model = apip.Apip(_params(case), 8, precision="fp32", lam_mode="const0")
        p = torch.tensor(apip.mlp_flat(W.mlp_params(7)), device=dev)
        return dict(kind=kind, model=model, G=G, y=y, n=case["batch"], t=0, p=p, m=torch.zeros_like(p),
                    v=torch.zeros_like(p), grad=torch.empty_like(p), loss=torch.zeros(1, device=dev))
    if kind == "labels":
        conf, box = _crystals(case, seed)
        nmax = 2 * case["cells"] ** 3 + 8
        model = apip.Apip(_params(case), nmax, precision="fp32", lam_mode="const1")
        return dict(kind=kind, model=model, box=box, pos=conf,
                    ids=torch.arange(nmax, dtype=torch.int32, device=dev),
                    types=torch.zeros(nmax, dtype=torch.int32, device=dev),
                    F=torch.empty((nmax, 3), dtype=torch.float64, device=dev))
    s = _system(case, seed)
    n, box = s["n"], s["box"]
    model = apip.Apip(_params(case), n, precision=case["precision"], lam_mode=case["lam"], max_nb=80, cell_cap=48)
    st = dict(kind=kind, model=model, box=box, n=n, snaps=s["snaps"], vel=s["vel"], lam_fixed=s["lam_fixed"],
              steps=case.get("steps", 0), ids=torch.arange(n, dtype=torch.int32, device=dev),
              types=torch.zeros(n, dtype=torch.int32, device=dev),
              F=torch.empty((n, 3), dtype=torch.float64, device=dev))
    pos = st["snaps"][0]
    if s["lam_fixed"] is not None:
        model.set_lam_fixed(s["lam_fixed"])
    if s["indenter"] is not None:
        model.set_indenter(**s["indenter"])
    if case["lam"] == "paper":
        model.init_csp_pairs(pos, box, st["ids"])
    if case["lam"] == "learned":
        model.set_mlp(_network().to(dev))
    if kind == "md":
        st["inv_mass"] = torch.full((n,), 1.0 / (W.MASS_AMU * apip.MVV2E), dtype=torch.float64, device=dev)
        st["thermo"] = torch.zeros((st["steps"], 5), dtype=torch.float64, device=dev)
        model.energy_forces(pos, box, st["types"], st["ids"], st["F"])
    else:
        st["out"] = [dict(F=torch.empty_like(st["F"]), e=torch.empty(n, dtype=torch.float64, device=dev),
                          E=torch.zeros(1, dtype=torch.float64, device=dev)) for _ in range(2)]
    model.sync()
    return st


# --------------------------------------------------------------------- run
def run(state):
    m = state["model"]
    if state["kind"] == "train":
        k, n = state["t"] % 4, state["n"]
        state["t"] += 1
        apip.apip_mlp_loss_grad(m.ctx, state["G"][k * n:(k + 1) * n], state["y"][k * n:(k + 1) * n], n, state["p"],
                                state["grad"], state["loss"])
        apip.apip_mlp_adam(m.ctx, state["p"], state["grad"], state["m"], state["v"], state["t"], 1e-3)
        return {k: state[k] for k in ("loss", "grad", "p", "m", "v")}
    if state["kind"] == "labels":
        out = []
        for pos in state["pos"]:
            n = pos.shape[0]
            ids, types = state["ids"][:n], state["types"][:n]
            e = torch.empty(n, dtype=torch.float64, device=pos.device)
            G = torch.empty((n, 32), dtype=torch.bfloat16, device=pos.device)
            m.energy_forces(pos, state["box"], types, ids, state["F"], e_atom_out=e)
            d = e - m.field("e_eam", n)
            m.descriptors(pos, state["box"], ids, G)
            out.append({"label": (d - LABEL_REF).abs().to(torch.float32), "G": G})
        return out
    if state["kind"] == "ef":
        for pos, o in zip(state["snaps"], state["out"]):
            m.energy_forces(pos, state["box"], state["types"], state["ids"], o["F"], o["e"], o["E"])
        return state["out"]
    pos = state["snaps"][0]
    m.verlet_step(pos, state["vel"], state["F"], state["inv_mass"], state["box"], state["types"], state["ids"], DT,
                  state["steps"], state["thermo"])
    return {"pos": pos, "vel": state["vel"], "F": state["F"], "thermo": state["thermo"]}


# -------------------------------------------------------------------- work
def _sizes(case):
    """(atoms, atoms with the precise model) of a system, to a few per cent."""
    s, c = case["system"], case["cells"]
    if s == "crack":
        n = 2 * (2 * c) * c * (c // 2)
        ace = 7.3 * c * c
    elif s == "slab":
        n = 2 * c * c * max(78 * c // 160, 8)
        ace = 0.6 * c * c
    else:
        n = 2 * c ** 3
        ace = 0.05 * n if s == "vacancy" else 0.8 * c * c
    return n, n if case["lam"] == "const1" else 0 if case["lam"] == "const0" else ace


def work(case):
    if case["kind"] == "train":
        # per sample: 32 bfloat16 descriptors, a label; three matrix products each way.
        # Parameters, gradient and both moments are read and written.
        n = case["batch"]
        return {"bytes": 68 * n + 10497 * 4 * 8, "flops": 57600 * n}
    if case["kind"] == "labels":
        n = 2 * case["cells"] ** 3 * case["configs"]
        return {"bytes": n * (24 + 4 + 4 + 64), "flops": n * (58 * 60 + 26 * 60 + 140e3)}
    n, ace = _sizes(case)
    per_ace = 140e3 if case["system"] != "crack" else 2.0e6
    per_atom = 58 * 30 + 26 * 60
    if case["lam"] == "learned":
        per_atom += 20.5e3 + 58 * 60
    flops = n * per_atom + ace * per_ace
    if case["kind"] == "ef":   # positions and ids in; forces, energies out
        return {"bytes": 2 * n * (24 + 4 + 24 + 8), "flops": 2 * flops}
    # positions, velocities, forces read and written, inverse masses and ids read
    return {"bytes": case["steps"] * n * (6 * 24 + 8 + 4), "flops": case["steps"] * flops}


# ------------------------------------------- the same in float64, from plain torch
def _chunks(n, size):
    return [slice(k, min(k + size, n)) for k in range(0, n, size)]


def _neighbours(pos, box, rc):
    """[n, K] indices of the neighbours within rc, -1 where there are fewer."""
    n, dev = len(pos), pos.device
    b = torch.tensor(box, dtype=torch.float64, device=dev)
    nc = torch.tensor([int(x // rc) for x in box], device=dev)
    p = _wrap(pos, box)
    c = torch.minimum((p / b * nc).long(), nc - 1)
    cell = (c[:, 0] * nc[1] + c[:, 1]) * nc[2] + c[:, 2]
    order = torch.argsort(cell, stable=True)
    count = torch.bincount(cell, minlength=int(nc.prod()))
    first = torch.cumsum(count, 0) - count
    cap = int(count.max())
    off = torch.tensor([(x, y, z) for x in (-1, 0, 1) for y in (-1, 0, 1) for z in (-1, 0, 1)], device=dev)
    slot = torch.arange(cap, device=dev)
    rows = []
    for q in _chunks(n, 100000):
        cc = (c[q, None, :] + off) % nc
        ci = (cc[..., 0] * nc[1] + cc[..., 1]) * nc[2] + cc[..., 2]
        at = first[ci][..., None] + slot
        ok = (slot < count[ci][..., None]).reshape(len(ci), -1)
        j = order[at.clamp(max=n - 1)].reshape(len(ci), -1)
        d = p[j] - p[q, None]
        d = d - b * torch.round(d / b)
        ok &= (d * d).sum(-1) < rc * rc
        ok &= j != torch.arange(q.start, q.stop, device=dev)[:, None]
        k = torch.cumsum(ok, 1) - 1
        r = torch.full((len(ci), int(ok.sum(1).max()) if len(ci) else 0), -1, dtype=torch.long, device=dev)
        i = torch.arange(len(ci), device=dev)[:, None].expand_as(j)
        r[i[ok], k[ok]] = j[ok]
        rows.append(r)
    K = max(r.shape[1] for r in rows)
    return torch.cat([torch.nn.functional.pad(r, (0, K - r.shape[1]), value=-1) for r in rows])


def _dist(pos, nb, box, rows):
    """Separations and distances of some rows' neighbours (1000 A where there is none)."""
    b = torch.tensor(box, dtype=torch.float64, device=pos.device)
    j = nb[rows]
    d = pos[j.clamp(min=0)] - pos[rows][:, None]
    d = d - b * torch.round(d / b)
    d = torch.where((j >= 0)[..., None], d, torch.tensor([1e3, 0.0, 0.0], dtype=torch.float64, device=pos.device))
    return d, torch.sqrt((d * d).sum(-1))


def _taper(x, lo, hi):
    t = torch.clamp((hi + lo - 2.0 * x) / (hi - lo), -1.0, 1.0)
    return 0.5 + t * (15.0 / 16.0 + t * t * (-5.0 / 8.0 + t * t * 3.0 / 16.0))


def _features(r, rc=5.0, width=1.0):
    mu = torch.linspace(1.5, 5.0, 32, dtype=torch.float64, device=r.device)
    return torch.exp(-(r[..., None] - mu) ** 2 / (2 * 0.15 ** 2)) * _taper(r, rc - width, rc)[..., None]


def _hidden(G, w):
    h = [0.25 * G]
    for k in ("1", "2", "3"):
        h.append(torch.nn.functional.silu(h[-1] @ w["W" + k].T + w["b" + k]))
    return h


def _ylm(u, lmax):
    """Real orthonormal harmonics of unit vectors, index l^2 + l + m."""
    x, y, z = u.unbind(-1)
    C, S = [torch.ones_like(x)], [torch.zeros_like(x)]
    for m in range(1, lmax + 1):
        C, S = C + [x * C[-1] - y * S[-1]], S + [x * S[-1] + y * C[-1]]
    out = [None] * (lmax + 1) ** 2
    for m in range(lmax + 1):
        P = {m: torch.full_like(z, float(np.prod(np.arange(2 * m - 1, 0, -2.0))))}
        for l in range(m + 1, lmax + 1):
            P[l] = ((2 * l - 1) * z * P[l - 1] - ((l + m - 1) * P[l - 2] if l > m + 1 else 0.0)) / (l - m)
        for l in range(m, lmax + 1):
            k = math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - m) / math.factorial(l + m) * (2 if m else 1))
            out[l * l + l + m] = k * P[l] * C[m]
            if m:
                out[l * l + l - m] = k * P[l] * S[m]
    return torch.stack(out, -1)


@functools.lru_cache(maxsize=2)
def _tables(n_max, l_max, nu_max):
    """Gaunt integrals and the coefficients of every product function, as dense matrices
    over (n, n') per pair of degrees (l <= l') and coupled degree L, for both channels."""
    t = torch.tensor
    zg, wz = np.polynomial.legendre.leggauss(2 * l_max + 4)
    ph = 2 * math.pi * np.arange(8 * l_max + 4) / (8 * l_max + 4)
    Z, PH = np.meshgrid(zg, ph, indexing="ij")
    st = np.sqrt(1 - Z ** 2)
    Y = _ylm(t(np.stack([st * np.cos(PH), st * np.sin(PH), Z], -1).reshape(-1, 3)), 2 * l_max)
    wt = t(np.repeat(wz, len(ph)) * 2 * math.pi / len(ph))
    ysl = lambda l: Y[:, l * l:(l + 1) ** 2]  # noqa: E731
    slots, gaunt = {}, {}       # L -> {(l, l'): first index}, (l, l', L) -> integrals
    for L in range(2 * l_max + 1):
        slots[L] = {}
        for l in range(l_max + 1):
            for k in range(l, l_max + 1):
                if k - l <= L <= k + l and (l + k + L) % 2 == 0:
                    slots[L][(l, k)] = len(slots[L]) * n_max ** 2
                    gaunt[(l, k, L)] = torch.einsum("q,qa,qb,qc->abc", wt, ysl(l), ysl(k), ysl(L))

    def at(p, q, L):
        (n, l), (m, k) = (p, q) if p[1] <= q[1] else (q, p)
        return slots[L][(l, k)] + (n - 1) * n_max + m - 1

    P = [(n, l) for n in range(1, n_max + 1) for l in range(l_max + 1)]
    ace = _ace(n_max, l_max, nu_max)
    coef = np.stack([ace["c1"], ace["c2"]])
    k1 = np.zeros((2, n_max))
    k2 = np.zeros((2, l_max + 1, n_max, n_max))
    k3 = {L: np.zeros((2, len(slots[L]) * n_max ** 2, n_max)) for L in range(l_max + 1)}
    k4 = {L: np.zeros((2, len(slots[L]) * n_max ** 2, len(slots[L]) * n_max ** 2)) for L in slots} if nu_max > 3 else {}
    f = 0
    for n in range(n_max):
        k1[:, n] = coef[:, f]
        f += 1
    for a, p in enumerate(P):
        for q in P[a:]:
            if p[1] == q[1]:
                k2[:, p[1], p[0] - 1, q[0] - 1] = coef[:, f]
                f += 1
    for a, p in enumerate(P):
        for b, q in enumerate(P[a:], a):
            for s in P[b:]:
                if (p[1] + q[1] + s[1]) % 2 == 0 and abs(p[1] - q[1]) <= s[1] <= p[1] + q[1]:
                    k3[s[1]][:, at(p, q, s[1]), s[0] - 1] += coef[:, f]
                    f += 1
    if nu_max > 3:
        for a, p in enumerate(P):
            for b, q in enumerate(P[a:], a):
                for c, s in enumerate(P[b:], b):
                    for u in P[c:]:
                        lo = max(abs(p[1] - q[1]), abs(s[1] - u[1]))
                        for L in range(lo, min(p[1] + q[1], s[1] + u[1]) + 1):
                            if (p[1] + q[1] + L) % 2 == 0 and (s[1] + u[1] + L) % 2 == 0:
                                k4[L][:, at(p, q, L), at(s, u, L)] += coef[:, f]
                                f += 1
    assert f == coef.shape[1]
    return slots, gaunt, t(k1), t(k2), {L: t(v) for L, v in k3.items()}, {L: t(v) for L, v in k4.items()}


def _ace_energy(d, r, p):
    """E^ACE of atoms from their neighbours' separations."""
    n_max, l_max, dev = p["n_max"], p["l_max"], r.device
    slots, gaunt, k1, k2, k3, k4 = _tables(n_max, l_max, p["nu_max"])
    x = 1.0 - 2.0 * r / p["rc"]
    T = [torch.ones_like(x), x]
    for _ in range(2, n_max):
        T.append(2.0 * x * T[-1] - T[-2])
    inside = (r < p["rc"])[..., None]
    R = torch.where(inside, torch.stack(T[:n_max], -1) * _taper(r, p["rc"] - p["rc_width"], p["rc"])[..., None], 0.0)
    A = p["a_scale"] * R.transpose(1, 2) @ _ylm(d / r[..., None], l_max)
    Al = [A[:, :, l * l:(l + 1) ** 2] for l in range(l_max + 1)]
    phi = [A[:, :, 0] @ k1[c].to(dev) for c in range(2)]
    for l in range(l_max + 1):
        for c in range(2):
            phi[c] = phi[c] + torch.einsum("xam,ab,xbm->x", Al[l], k2[c, l].to(dev), Al[l])
    for L in slots:
        if L > l_max and L not in k4:
            continue
        C = torch.cat([torch.einsum("xai,xbj,ijm->xabm", Al[l], Al[k], gaunt[(l, k, L)].to(dev)).flatten(1, 2)
                       for l, k in slots[L]], 1)
        for c in range(2):
            if L <= l_max:
                phi[c] = phi[c] + torch.einsum("xum,un,xnm->x", C, k3[L][c].to(dev), Al[L])
            if L in k4:
                phi[c] = phi[c] + (C * torch.einsum("uv,xvm->xum", k4[L][c].to(dev), C)).sum((1, 2))
    return phi[0] + (phi[1] ** 2 + p["eps"] ** 2) ** 0.25 - math.sqrt(p["eps"])


def _csp_pairs(pos, nb, box, rcut, nnb):
    """Opposite neighbours: the nearest ones paired greedily by |r_a + r_b|^2."""
    out = []
    for q in _chunks(len(pos), 200000):
        d, r = _dist(pos, nb, box, q)
        r, k = torch.sort(torch.where(r < rcut, r, math.inf), dim=1, stable=True)
        k, r = k[:, :nnb], r[:, :nnb]
        dd = torch.gather(d, 1, k[..., None].expand(-1, -1, 3))
        j = torch.where(r < math.inf, torch.gather(nb[q], 1, k), -1)
        s = ((dd[:, :, None] + dd[:, None]) ** 2).sum(-1)
        dead = torch.tril(torch.ones(nnb, nnb, dtype=torch.bool, device=pos.device)) | (j < 0)[:, :, None] | (j < 0)[:, None]
        rows = []
        for _ in range(nnb // 2):
            best, at = torch.where(dead, math.inf, s).flatten(1).min(1)
            a, b = at // nnb, at % nnb
            good = best < math.inf
            rows += [torch.where(good, j.gather(1, x[:, None])[:, 0], -1) for x in (a, b)]
            used = torch.zeros(len(j), nnb, dtype=torch.bool, device=pos.device)
            used.scatter_(1, a[:, None], True)
            used.scatter_(1, b[:, None], True)
            dead = dead | used[:, :, None] | used[:, None]
        out.append(torch.stack(rows, 1))
    return torch.cat(out)


def _energy_forces(pos, nb, box, prm, lam_mode, pairs=None, lam_fixed=None, ind=None, net=None):
    """E, per-atom energies and F = -grad E."""
    n, dev = len(pos), pos.device
    b = torch.tensor(box, dtype=torch.float64, device=dev)
    e, sw, rows = prm["eam"], prm["switch"], slice(0, n)
    adds = 1.0 if prm["precise_adds_eam"] else 0.0
    pos = pos.detach().requires_grad_(True)
    d, r = _dist(pos, nb, box, rows)
    fc = _taper(r, e["rc"] - e["rc_width"], e["rc"])
    near = r < e["rc"]
    zeta = torch.where(near, e["A"] * torch.exp(-e["beta"] * (r - e["r_e"])) * fc, 0.0).sum(1)
    x = torch.exp(-e["alpha"] * (r - e["r_0"]))
    e_eam = 0.5 * torch.where(near, e["D"] * (x * x - 2 * x) * fc, 0.0).sum(1) - torch.sqrt(zeta)
    if lam_mode in ("paper", "learned"):
        if lam_mode == "paper":
            u = pos[pairs.clamp(min=0)] - pos[:, None]
            u = u - b * torch.round(u / b)
            g = torch.where(pairs[:, 0::2] >= 0, ((u[:, 0::2] + u[:, 1::2]) ** 2).sum(-1), 0.0).sum(1)
        else:
            g = torch.cat([_hidden(_features(r[q]).sum(1), net)[-1] @ net["w4"] + net["b4"]
                           for q in _chunks(n, 100000)])
        w = torch.where(nb >= 0, _taper(r, sw["r_w"] - sw["r_w_width"], sw["r_w"]), 0.0)
        dd = (g + (w * g[nb.clamp(min=0)]).sum(1)) / (1.0 + w.sum(1)) - sw["d0"]
        lam = 1.0 - _taper(dd, sw["d_lo"], sw["d_hi"])
    else:
        lam = torch.full((n,), 1.0 if lam_mode == "const1" else 0.0, dtype=torch.float64, device=dev)
    if lam_fixed is not None:
        lam = torch.where(torch.isnan(lam_fixed), lam, lam_fixed)
    lam0 = lam.detach()
    ace, grad = torch.zeros(n, dtype=torch.float64, device=dev), torch.zeros(n, 3, dtype=torch.float64, device=dev)
    P = torch.nonzero(lam0 > 0)[:, 0]
    for q in _chunks(len(P), 4000):
        p2 = pos.detach().requires_grad_(True)
        ea = _ace_energy(*_dist(p2, nb, box, P[q]), prm["ace"])
        grad += torch.autograd.grad((lam0[P[q]] * ea).sum(), p2)[0]
        ace[P[q]] = ea.detach()
    e_prec = ace + adds * e_eam.detach()
    delta = e_prec - e_eam.detach()
    total = ((1.0 - lam0 + adds * lam0) * e_eam).sum() + (lam * delta).sum()
    e_atom = lam0 * e_prec + (1.0 - lam0) * e_eam.detach()
    if ind is not None:
        v = pos - torch.tensor(ind["center"], dtype=torch.float64, device=dev)
        v = v - b * torch.round(v / b)
        ei = ind["k"] / 3.0 * torch.clamp(ind["radius"] - torch.sqrt((v * v).sum(1)), min=0.0) ** 3
        total = total + ei.sum()
        e_atom = e_atom + ei.detach()
    grad += torch.autograd.grad(total, pos)[0]
    return e_atom.sum(), e_atom, -grad


def _bf16(x):
    return x.to(torch.float32).to(torch.bfloat16).to(torch.float64)


def _exact_train(case, seed):
    G, y = _batches(case, seed)
    n = case["batch"]
    G, y = G[:n].double(), y[:n].double()
    w = {k: torch.tensor(v, device="cuda") for k, v in apip.mlp_unflat(apip.mlp_flat(W.mlp_params(7))).items()}
    sig = torch.sigmoid
    z, h = [], [0.25 * G]
    for k in "123":     # operands of every product rounded to bfloat16, as the training does by definition
        z.append(h[-1] @ _bf16(w["W" + k]).T + w["b" + k])
        s = z[-1] * sig(z[-1])
        h.append(_bf16(s))
    res = s @ w["w4"] + w["b4"] - y
    dg = 2.0 * res / n
    grad = {"w4": h[3].T @ _bf16(dg), "b4": _bf16(dg).sum()}
    back = dg[:, None] * w["w4"]
    for k in (3, 2, 1):
        s = sig(z[k - 1])
        dz = _bf16(back * s * (1.0 + z[k - 1] * (1.0 - s)))
        grad["W%d" % k], grad["b%d" % k] = dz.T @ h[k - 1], dz.sum(0)
        back = dz @ _bf16(w["W%d" % k])
    names = ("W1", "b1", "W2", "b2", "W3", "b3", "w4", "b4")
    g, p = (torch.cat([d[k].reshape(-1) for k in names]) for d in (grad, w))
    return {"loss": (res * res).mean().reshape(1), "grad": g, "p": p - 1e-3 * g / (g.abs() + 1e-8), "m": 0.1 * g,
            "v": 1e-3 * g * g}


def exact(case, seed):
    if case["kind"] == "train":
        return _exact_train(case, seed)
    prm = _params(case)
    if case["kind"] == "labels":
        out = []
        conf, box = _crystals(case, seed)
        for pos in conf:
            nb = _neighbours(pos, box, 5.0)
            d, r = _dist(pos, nb, box, slice(0, len(pos)))
            ace = torch.cat([_ace_energy(d[q], r[q], prm["ace"]) for q in _chunks(len(pos), 4000)])
            out.append({"label": (ace - LABEL_REF).abs(), "G": _features(r).sum(1)})
        return out
    s = _system(case, seed)
    box, pos = s["box"], s["snaps"][0]
    if s["n"] > 2.5e6 or (case["lam"] == "const1" and s["n"] > 6e4):
        return None      # over some twenty seconds
    nb = _neighbours(pos, box, 5.3)
    pairs = _csp_pairs(pos, nb, box, prm["csp"]["rcut"], prm["csp"]["nnb"])
    net = None
    if case["lam"] == "learned":
        net = {k: torch.tensor(v, device="cuda") for k, v in apip.mlp_unflat(_network().numpy()).items()}
    ind = s["indenter"]
    args = dict(prm=prm, lam_mode=case["lam"], pairs=pairs, lam_fixed=s["lam_fixed"], net=net)
    if case["kind"] == "ef":
        out = []
        for p in s["snaps"]:
            E, e, F = _energy_forces(p, _neighbours(p, box, 5.0), box, **args)
            out.append({"F": F, "e": e, "E": E.reshape(1)})
        return out
    v, im = s["vel"], 1.0 / (W.MASS_AMU * apip.MVV2E)
    F = _energy_forces(pos, nb, box, ind=ind, **args)[2]
    rows = []
    for _ in range(case["steps"]):
        v = v + 0.5 * DT * im * F
        pos = pos + DT * v
        if ind is not None:
            ind = dict(ind, center=[c + DT * u for c, u in zip(ind["center"], ind["velocity"])])
        E, _, F = _energy_forces(pos, nb, box, ind=ind, **args)
        v = v + 0.5 * DT * im * F
        rows.append(torch.cat([E.reshape(1), (v * v).sum().reshape(1) / (2 * im), v.sum(0) / im]))
    return {"pos": _wrap(pos, box), "vel": v, "F": F, "thermo": torch.stack(rows)}
