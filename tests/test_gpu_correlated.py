"""Tables of two-mode squeezed pairs, the strongest correlations a state can have
between two of its modes: where both are in a subset, the elimination cancels down to
about e^{-2r} of its operands. Pairs of modes at random places with squeezing r up to
3, random phases and losses, in both precisions, against the oracle.

Tolerances, as the library states them: P0 relative 1e-12 (FP64) / 1e-11 (refined),
moments and cumulants absolute 1e-12."""
import numpy as np
import pytest
import torch

import oracle
import synthetic
import paper_2511_14923_gb300 as gbs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    gbs.build()


def squeezed_pairs(M, r, seed):
    """M modes in two-mode squeezed pairs: two single-mode squeezed inputs on a 50:50
    beam splitter each, then a random phase and loss per mode (an odd M leaves one
    mode in vacuum)."""
    rng = np.random.default_rng(seed)
    order = rng.permutation(M)
    U, rr = np.eye(M, dtype=complex), np.zeros(M)
    for a, b in zip(order[: M // 2 * 2 : 2], order[1::2]):
        rr[a] = rr[b] = r
        U[a, a] = U[b, b] = np.sqrt(0.5)
        U[a, b] = U[b, a] = 1j * np.sqrt(0.5)
    U = np.exp(2j * np.pi * rng.random(M))[:, None] * U
    return synthetic.covariance(rr, rng.uniform(0.8, 1.0, M), U)


# order 3 and 4 by chunks and order 5 by the tree; order 4 by the tree as well
@pytest.mark.parametrize("precision", ["fp64", "fp32r"])
@pytest.mark.parametrize("M,kmax,seeds", [(8, 5, 6), (9, 5, 3), (65, 4, 1)])
@pytest.mark.parametrize("r", [1.0, 2.25, 3.0])
def test_two_mode_squeezed_pairs(M, kmax, seeds, r, precision):
    rel = 1e-12 if precision == "fp64" else 1e-11
    for seed in range(seeds):
        V = squeezed_pairs(M, r, 9000 + 10 * M + seed)
        p0, mu, kt = oracle.tables(V, kmax)
        t = torch.from_numpy(V).cuda()
        assert np.abs(gbs.vacuum_probs(t, kmax, precision).cpu().numpy() / p0 - 1).max() <= rel
        assert np.abs(gbs.click_moments(t, kmax, precision).cpu().numpy() - mu).max() <= 1e-12
        assert np.abs(gbs.cumulants(t, kmax, precision).cpu().numpy() - kt).max() <= 1e-12
