"""Parameter draws of many genes: rows shared by clusters of two, four and eight
blocks (edges of the split, a last block without genes, rows beyond the
blocks' caches), one chain, a batch and a local iteration, against the
oracle; the noise split between blocks with and without rows."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1812_10048_gb300 import build
    build.build()
    import paper_1812_10048_gb300 as P
    return P


def counts(N, D, rng):
    from scipy.sparse import random as sprandom
    X = sprandom(N, D, min(1.0, 60.0 / D), format="csr", random_state=rng,
                 data_rvs=lambda n: rng.integers(1, 9, size=n).astype(np.float64))
    X.sort_indices()
    return (X.indptr.astype(np.int32), X.indices.astype(np.int32), X.data.astype(np.int32))


def check(logpi, logtheta, nsub, Ssub, seed, chain, t):
    from oracle.sampler import draw_pi, draw_theta
    np.testing.assert_allclose(logpi, draw_pi(nsub.sum(axis=1), 1.0, seed, chain, t), rtol=1e-5,
                               atol=1e-4)
    ref = draw_theta(Ssub, 0.5, seed, chain, t)
    # an FP32 accept decision on its tie changes one variate
    off = ~np.isclose(logtheta, ref, rtol=1e-5, atol=1e-4)
    assert off.sum() <= max(2, 1e-4 * ref.size), off.sum()
    lse = np.logaddexp.reduce(logtheta.astype(np.float64), axis=1)
    # an FP32 log-sum-exp of D terms, its sum taken by warps, blocks and the cluster
    np.testing.assert_allclose(lse, 0.0, atol=2e-5)


@pytest.mark.parametrize("D", [2048, 2049, 4095, 8193, 32738, 66001])
@pytest.mark.parametrize("K", [1, 7])
def test_wide_rows(P, D, K):
    rng = np.random.default_rng([D, K])
    N = 300
    csr = counts(N, D, rng)
    lab, sub = np.arange(N) % K, rng.integers(0, 2, N).astype(np.uint8)
    s = P.Sampler(*csr, N, D, 1.0, 0.5, kmax=16, seed=9, chain_id=2)
    s.set_state(lab, sub, K, t=4)
    nsub, Ssub, _ = s.stats()
    P.dpmm_draw_params(s.ctx)
    logpi, logtheta = P.dpmm_get_params(s.ctx, K, D)
    s.close()
    check(logpi, logtheta, nsub.astype(np.int64), Ssub.astype(np.int64), 9, 2, 4)


def test_wide_batch_equals_single_chains(P):
    """Chains of 9,000 genes (clusters of eight blocks) evolve in a batch as alone."""
    rng = np.random.default_rng(5)
    D, Ns = 9000, [257, 40, 900]
    data = [counts(N, D, rng) + (N,) for N in Ns]
    b = P.BatchSampler(data, D, 1.0, 0.5, kmax=16, seed=3, local_iters=2)
    b.step(4)
    for i, d in enumerate(data):
        s = P.Sampler(*d[:3], d[3], D, 1.0, 0.5, kmax=16, seed=3, chain_id=i, local_iters=2)
        s.step(4)
        for x, y in zip(s.get_state(), b.chain(i).get_state()):
            np.testing.assert_array_equal(x, y)
        np.testing.assert_array_equal(s.stats()[1], b.chain(i).stats()[1])
        s.close()
    b.close()


@pytest.mark.parametrize("N,K", [(129, 3), (70001, 40), (200003, 3)])
def test_noise_shares_cover_every_cell(P, N, K):
    """A sweep reads noise that was drawn for it: labels of every cell equal
    those of the label call alone (whose noise another kernel deals out)."""
    rng = np.random.default_rng(N)
    csr = counts(N, 70, rng)
    lab, sub = np.arange(N) % K, rng.integers(0, 2, N).astype(np.uint8)
    got = []
    for whole in (True, False):
        s = P.Sampler(*csr, N, 70, 1.0, 0.5, kmax=64, seed=9, engine=P.ENGINE_TILE_BF16)
        s.set_state(lab, sub, K, t=1)
        if whole:
            s.sweep(1)
        else:
            P.dpmm_draw_params(s.ctx)
            P.dpmm_assign(s.ctx)
        got.append(s.get_state())
        s.close()
    for x, y in zip(*got):
        np.testing.assert_array_equal(x, y)
