"""Two host threads, each with a context of its own whose ACE kernel is the same function
with another amount of dynamic shared memory (basis 8/3: 150 KB, basis 1/3: 20 KB): no
launch of either is refused, and both end where a lone run of theirs ends.  Bar: a force
difference of the float32 path's 2e-4 eV/A moves an atom by 1.6e-7 A in 3e-3 ps; 1e-6."""
import threading

import pytest

from gpu_helpers import to_dev, torch_cuda
from paper_2512_07693_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _run(torch, n_max, out, key, start=None):
    from paper_2512_07693_gb300 import apip
    s = W.config("void250k", apip.apip_ace_basis_size, scale=8)
    s["prm"]["ace"] = W.ace_params(n_max, 3, 3, 2, apip.apip_ace_basis_size(n_max, 3, 3))
    t, n, box = to_dev(torch, s), len(s["pos"]), [float(b) for b in s["box"]]
    stream = torch.cuda.Stream()
    try:
        with torch.cuda.stream(stream):
            m = apip.Apip(s["prm"], n, precision="fp32", lam_mode="paper")
            h = stream.cuda_stream
            m.init_csp_pairs(t["pos"], box, t["ids"], stream=h)
            F = torch.empty_like(t["pos"])
            m.energy_forces(t["pos"], box, t["types"], t["ids"], F, stream=h)
            m.sync(h)
            if start:
                start.wait()
            for _ in range(60):
                m.verlet_step(t["pos"], t["vel"], F, t["inv_mass"], box, t["types"], t["ids"], 1e-6, 50, stream=h)
            m.sync(h)
            out[key] = t["pos"].clone()
            stream.synchronize()
            m.close()
    except Exception as e:   # reported by the test's thread
        out[key] = e


def test_contexts_of_other_sizes():
    torch = torch_cuda()
    alone, both = {}, {}
    for n_max in (8, 1):
        _run(torch, n_max, alone, n_max)
    start = threading.Barrier(2)
    threads = [threading.Thread(target=_run, args=(torch, n_max, both, n_max, start)) for n_max in (8, 1)]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    for n_max in (8, 1):
        assert not isinstance(both[n_max], Exception), both[n_max]
        assert (both[n_max] - alone[n_max]).abs().max() <= 1e-6
