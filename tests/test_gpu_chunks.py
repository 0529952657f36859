"""Forms that calls take by their size: orders 3 and 4 by chunks of pairs, the
cumulant recursion on float pairs, and the sampler's blocked p2 update and product
tiles, at the sizes where they begin, end or leave a remainder, against the oracle
or against the form used at another size.

Tolerances: P0 relative 1e-12 (FP64) / 1e-11 (refined), tables absolute 1e-12, as
the library states them; spin tables 2^d times that. Sampler, FP64: bits equal,
log-probabilities within 1e-11."""
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


@pytest.mark.parametrize("precision", ["fp64", "fp32r"])
@pytest.mark.parametrize("M,kmax", [(3, 3), (4, 4), (5, 4), (6, 5), (17, 4), (24, 3), (33, 4), (63, 4), (64, 4)])
def test_chunked_orders_match_oracle(M, kmax, precision):
    inst = synthetic.random_instance(M, kmax, seed=7000 + M, r_range=(0.4, 1.4))
    V = torch.from_numpy(inst.V).cuda()
    p0, mu, kt = oracle.tables(inst.V, kmax)
    rel = 1e-12 if precision == "fp64" else 1e-11
    assert np.abs(gbs.vacuum_probs(V, kmax, precision).cpu().numpy() / p0 - 1).max() <= rel
    assert np.abs(gbs.click_moments(V, kmax, precision).cpu().numpy() - mu).max() <= 1e-12
    k = gbs.cumulants(V, kmax, precision).cpu().numpy()
    assert np.abs(k - kt).max() <= 1e-12
    spin = gbs.spin_cumulants(V, kmax, precision).cpu().numpy()
    for d in range(2, kmax + 1):  # exact powers of two apart
        s = slice(gbs.order_offset(M, d), gbs.order_offset(M, d + 1) if d < kmax else None)
        assert np.array_equal(spin[s], (-2.0) ** d * k[s])


@pytest.mark.parametrize("M", [4, 9, 40])
def test_chunked_orders_of_displaced_states_match_oracle(M):
    inst = synthetic.random_instance(M, 4, seed=7100 + M)
    mean = synthetic.displaced_mean(inst, 5)
    p0 = gbs.displaced_tables(torch.from_numpy(inst.V).cuda(), torch.from_numpy(mean).cuda(), 4, "p0").cpu().numpy()
    sets = synthetic.random_subsets(M, 4, 300, 3)
    off = gbs.order_offset(M, 4)
    for s in sets:
        ref = oracle.p0_displaced(inst.V, mean, [int(x) for x in s])
        assert abs(p0[off + gbs.rank(s)] / ref - 1) <= 1e-12


@pytest.mark.parametrize("precision", ["fp64", "fp32r"])
def test_not_positive_definite_prefix_is_reported(precision):
    """A pivot that fails in the prefix, in the chunk's rows or in a leaf leaves NaN
    in every subset that holds the bad pair, and nowhere else."""
    M = 12
    V = np.eye(2 * M) * 3.0
    V[2, 9] = V[9, 2] = 5.0  # modes 2 and 9: not positive definite together
    t = torch.from_numpy(V).cuda()
    k = gbs.cumulants(t, 4, precision, check=False).cpu().numpy()
    with pytest.raises(gbs.GbsError):
        gbs.cumulants(t, 4, precision)
    for d in (3, 4):
        off = gbs.order_offset(M, d)
        for r in range(gbs.table_size(M, d) - off):
            s = gbs.unrank(r, d)
            assert np.isnan(k[off + r]) == (2 in s and 9 in s), s


def draws(M, K, n, batch, precision, seed=11):
    inst = synthetic.random_instance(M, K, seed=7200 + M, r_range=(0.5, 1.3))
    kap = gbs.spin_cumulants(torch.from_numpy(inst.V).cuda(), K, "fp64")
    u = np.random.default_rng(seed).random((n, M))
    out = gbs.sample(kap, M, K, u=torch.from_numpy(u).cuda(), batch=batch, precision=precision, want_q0=True)
    return kap, u, [x.cpu().numpy() for x in out]


@pytest.mark.parametrize("M", [8, 9, 10, 16, 17, 18])
def test_blocked_p2_update_matches_oracle(M):
    """Blocks of eight steps: M at, before and after a block's end."""
    kap, u, (bits, logp, q0) = draws(M, 5, 130, 256, "fp64")
    rb, rp, rq = oracle.sample(kap.cpu().numpy(), M, 5, u=u)
    assert np.array_equal(bits, rb)
    np.testing.assert_allclose(logp, np.log(rp), rtol=0, atol=1e-11)
    assert np.abs(q0 - rq).max() <= 1e-12


@pytest.mark.parametrize("K,M", [(3, 40), (4, 33), (5, 26)])
@pytest.mark.parametrize("precision,small,large", [("fp32", 256, 16384), ("fp64", 128, 2048), ("fp32", 128, 2176)])
def test_samples_do_not_depend_on_the_batch(K, M, precision, small, large):
    """Tiles, rings and schedules follow the batch; a sample's values don't. (FP32
    batches that are no multiple of 256 run the CUDA-core product in both calls.)"""
    a = draws(M, K, small, small, precision)[2]
    inst_u = np.random.default_rng(11).random((small, M))
    kap, _, _ = draws(M, K, 1, small, precision)
    u = np.concatenate([inst_u, np.random.default_rng(5).random((large - small, M))])
    b = gbs.sample(kap, M, K, u=torch.from_numpy(u).cuda(), batch=large, precision=precision, want_q0=True)
    for x, y in zip(a, b):
        assert np.array_equal(x, y.cpu().numpy()[:small])
