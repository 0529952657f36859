"""The adjoint's dL/dP0 gather with several teams of threads to a block: kmax and M at
which a team of order 1 (kmax = 4) or 2 (kmax = 5) has 32, 64, 128, 256 and 512 lanes,
the last block in part empty, against the oracle's gradient."""
import numpy as np
import pytest
import torch

import oracle
import synthetic
import paper_2511_14923_gb300 as gbs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,kmax", [(16, 4), (17, 4), (25, 4), (34, 4), (47, 4), (18, 5), (24, 5)])
def test_gradient_across_team_sizes(M, kmax):
    """Tolerance: the adjoint's, 1e-10 of the gradient's largest element."""
    gbs.build()
    inst = synthetic.random_instance(M, kmax, seed=9800 + M)
    g = np.random.default_rng(M).standard_normal(gbs.table_size(M, kmax))
    got = gbs.cumulants_backward(torch.from_numpy(inst.V).cuda(), kmax, torch.from_numpy(g).cuda()).cpu().numpy()
    want = oracle.grad(inst.V, kmax, g)
    assert np.abs(got - want).max() <= 1e-10 * np.abs(want).max()
