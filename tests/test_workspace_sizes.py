"""Workspace sizes: the float-pair copies of the lower orders, which only refined
cumulant tables read, are part of the refined size alone; and a workspace of the FP64
size serves every call, as it did before there were such copies."""
from math import comb

import pytest
import torch

import synthetic
import paper_2511_14923_gb300 as gbs

FNS = ("vacuum_probs", "click_moments", "cumulants", "spin_correlators", "spin_cumulants")


@pytest.fixture(scope="module", autouse=True)
def built():
    gbs.build()


@pytest.mark.parametrize("M,kmax", [(3, 3), (12, 4), (40, 5), (300, 4), (600, 5), (1024, 4)])
def test_fp64_size_has_no_float_pairs(M, kmax):
    low = gbs.order_offset(M, kmax)  # entries of the orders below kmax
    sizes = {p: gbs.workspace_bytes(M, kmax, p) for p in ("fp64", "fp32r")}
    ranged = {p: int(gbs.lib().gbs_range_workspace_bytes(M, kmax, gbs.PRECISIONS[p])) for p in ("fp64", "fp32r")}
    for s in (sizes, ranged):
        extra = s["fp32r"] - s["fp64"]
        assert 16 * low <= extra < 16 * low + 1024 if kmax >= 4 else extra == 0
    assert 8 * low <= ranged["fp64"] - sizes["fp64"] < 8 * low + 256


@pytest.mark.gpu
@pytest.mark.parametrize("kmax", [3, 4, 5])
def test_fp64_sized_workspace_serves_refined_calls(kmax):
    M = 20
    V = torch.from_numpy(synthetic.random_instance(M, kmax, seed=9900).V).cuda()
    ws = gbs.Workspace(M, kmax, "fp64")
    raw = torch.empty(int(gbs.lib().gbs_range_workspace_bytes(M, kmax, 0)), dtype=torch.uint8, device="cuda")
    lo = 7
    first = gbs.order_offset(M, kmax) + comb(lo, kmax)
    for name in FNS:
        f = getattr(gbs, name)
        got = f(V, kmax, "fp32r", workspace=ws)
        table = {"vacuum_probs": "p0", "click_moments": "mu", "cumulants": "kappa", "spin_correlators": "spin_c",
                 "spin_cumulants": "spin_kappa"}[name]
        part = gbs.table_range(V, kmax, lo, M, table, "fp32r", workspace=raw)
        # refined arithmetic where it needs no pairs, FP64 where it would
        prec = "fp64" if kmax >= 4 and "cumulants" in name else "fp32r"
        want = f(V, kmax, prec)
        assert torch.equal(got, want)
        assert torch.equal(part, want[first:])
    assert gbs.autotune(V, kmax, "fp32r", workspace=ws) > 0
    assert torch.equal(gbs.cumulants(V, kmax, "fp32r", workspace=ws), gbs.cumulants(V, kmax, "fp64" if kmax >= 4 else "fp32r"))
    with pytest.raises(gbs.GbsError):
        small = gbs.Workspace(M - 1, kmax, "fp32r")
        small.nbytes = ws.nbytes - 1
        gbs.cumulants(V, kmax, "fp32r", workspace=small)
