"""What apip_ace_info says of each evaluation: its kind, the atoms per block that a large
system takes, and counts that follow from the basis alone (float32 and float64, a group
size asked for or not)."""
import pytest

from gpu_helpers import torch_cuda
from paper_2512_07693_gb300 import workloads as W

pytestmark = pytest.mark.gpu

POOL, STREAMED, QUAD = 0, 1, 2


def _info(basis, precision, group=0, lam_mode="const1"):
    from paper_2512_07693_gb300 import apip
    torch_cuda()
    s = W.config("void250k", apip.apip_ace_basis_size, scale=7)
    s["prm"]["ace"] = W.ace_params(*basis, 2, apip.apip_ace_basis_size(*basis))
    m = apip.Apip(s["prm"], 100, precision=precision, lam_mode=lam_mode, ace_group=group)
    out = apip.apip_ace_info(m.ctx)
    m.close()
    return out


@pytest.mark.parametrize("basis,precision,group,kind,atoms", [
    ((6, 3, 3), "fp32", 0, STREAMED, 32), ((6, 3, 3), "fp64", 0, STREAMED, 32), ((6, 3, 3), "fp32", 8, STREAMED, 8),
    ((8, 4, 3), "fp64", 0, STREAMED, 32), ((4, 2, 4), "fp32", 0, POOL, 8), ((4, 2, 4), "fp64", 0, POOL, 8),
    ((8, 4, 4), "fp32", 1, POOL, 1), ((8, 4, 4), "fp32", 0, QUAD, 8), ((5, 4, 4), "fp32", 0, QUAD, 8)])
def test_kind_and_group(basis, precision, group, kind, atoms):
    i = _info(basis, precision, group)
    assert i["kind"] == kind and i["group"] == atoms


@pytest.mark.parametrize("lam_mode", ["const1", "paper"])
def test_automatic_group_is_what_a_large_system_takes(lam_mode):
    """basis 6/3 in float32: 32 atoms per block leave two resident blocks as 8 do."""
    assert _info((6, 3, 3), "fp32", 0, lam_mode)["group"] == 32


def test_quadratic_counts():
    q, p = _info((8, 4, 4), "fp32"), _info((8, 4, 4), "fp32", 1)
    for k in ("couplings", "gaunt_products", "c_to_a_entries"):
        assert q[k] == p[k], k
    # every function is one entry of K2 and two of each S, times 2 L + 1 (squares one): at
    # least the records' elements, and no more than 1.5 times that with the tiles' padding
    el = p["record_len_sum"]
    assert el <= q["record_len_sum"] <= 1.5 * el
    assert 3.9 * el <= q["row_len_sum"] <= 1.5 * 4 * el
    assert q["table_flops"] > 2 * (q["record_len_sum"] + q["row_len_sum"])
