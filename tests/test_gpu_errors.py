"""A runtime call that fails is reported by the call it failed in and by no later one."""
import pytest
import torch

import synthetic
import paper_2511_14923_gb300 as gbs

pytestmark = pytest.mark.gpu


def test_failed_launch_is_reported_once(monkeypatch):
    gbs.build()
    V = torch.from_numpy(synthetic.random_instance(9, 3, seed=9700).V).cuda()
    want = gbs.cumulants(V, 3)
    monkeypatch.setenv("GBS_FAULT_INJECT", "forward_launch")
    with pytest.raises(gbs.GbsError):
        gbs.cumulants(V, 3)
    monkeypatch.delenv("GBS_FAULT_INJECT")
    assert torch.equal(gbs.cumulants(V, 3), want)  # the library's own check
    monkeypatch.setenv("GBS_FAULT_INJECT", "forward_launch")
    with pytest.raises(gbs.GbsError):
        gbs.cumulants(V, 3)
    monkeypatch.delenv("GBS_FAULT_INJECT")
    assert torch.equal(want + 0, want)  # the caller's
