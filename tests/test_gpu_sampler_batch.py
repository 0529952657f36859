"""Sampling at the largest batch the library accepts: the same samples, bit for bit, as
in two batches of half of it (a sample's values do not depend on the batch)."""
import pytest
import torch

import synthetic
import paper_2511_14923_gb300 as gbs

pytestmark = pytest.mark.gpu
LARGEST = 1 << 21  # GBS_MAX_SAMPLE_BATCH


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("K", [3, 4, 5])
def test_largest_batch(K, precision):
    gbs.build()
    M = 5
    V = torch.from_numpy(synthetic.random_instance(M, K, seed=9600 + K).V).cuda()
    kappa = gbs.spin_cumulants(V, K, "fp64")
    u = torch.rand((LARGEST, M), dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(7))
    got = gbs.sample(kappa, M, K, u=u, batch=LARGEST, precision=precision)
    want = gbs.sample(kappa, M, K, u=u, batch=LARGEST // 2, precision=precision)
    assert torch.equal(got[0], want[0])
    assert torch.equal(got[1].nan_to_num(nan=1.0), want[1].nan_to_num(nan=1.0))
