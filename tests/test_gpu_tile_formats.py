"""Dense-tile engine: operand formats (FP16, BF16 where log theta passes FP16's
range), second planes of large counts, and the item order's edges (tiles in
pairs or alone, one, two or an odd number of chunks), scores against FP64."""

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


def sparse(N, D, density, rng, big=0, top=60000):
    """CSR with counts below 6 and `big` counts up to `top` in random places."""
    from scipy.sparse import random as sprandom
    X = sprandom(N, D, density, format="csr", random_state=rng,
                 data_rvs=lambda n: rng.integers(1, 6, size=n).astype(np.float64))
    X.sort_indices()
    if big and X.nnz:
        at = rng.choice(X.nnz, size=min(big, X.nnz), replace=False)
        X.data[at] = rng.integers(1500, top + 1, size=at.size)
    return X


def check_scores(P, X, K, logtheta, eps):
    """debug_tile_scores of every cell within the representation bound eps per
    |x d| and the accumulation's: at most 8 (chunks + 1) FP32 additions per sum,
    each within 2^-22 of the running total, plus the FP32 mean m_u."""
    N, D = X.shape
    g = P.Sampler(X.indptr.astype(np.int32), X.indices.astype(np.int32),
                  X.data.astype(np.int32), N, D, 1.0, 0.5, kmax=64, seed=3,
                  engine=P.ENGINE_TILE_BF16)
    lab = np.arange(N) % K
    g.set_state(lab, np.zeros(N, np.uint8), K)
    logpi = np.full(K + 1, -np.log(K + 1.0))
    P.dpmm_set_params(g.ctx, logpi, logtheta)
    got = P.dpmm_debug_tile_scores(g.ctx, N, K).astype(np.float64)
    g.close()
    L = logtheta.astype(np.float32).astype(np.float64)
    d = L - L.mean(axis=0)
    order = np.concatenate([np.arange(0, 3 * K, 3),
                            np.stack([np.arange(1, 3 * K, 3), np.arange(2, 3 * K, 3)], 1).ravel()])
    ref = np.asarray(X @ d[order].T)
    size = np.asarray(X @ np.abs(d[order]).T)
    rows = np.asarray(X @ np.abs(L).max(axis=0))[:, None]
    chunks = (D + 63) // 64
    bound = (eps + 8 * (chunks + 1) * 2.0 ** -22) * size + 2.0 ** -20 * rows + 1e-6
    err = np.abs(got - ref)
    assert np.all(err <= bound), (err.max(), (err / bound).max())


@pytest.mark.parametrize("N,D,K", [
    (1, 1, 1), (129, 63, 2), (127, 65, 3), (300, 129, 10), (260, 321, 23), (140, 200, 40),
    (38989, 40, 5),     # tiles in pairs and alone, one chunk
    (38989, 130, 2),    # three chunks: a lone last chunk for unpaired tiles
    (60001, 70, 40),    # pairs that wait for both accumulators
])
def test_fp16_scores(P, N, D, K):
    rng = np.random.default_rng([N, D, K])
    X = sparse(N, D, min(1.0, 40.0 / D), rng)
    logtheta = np.log(rng.dirichlet(np.full(D, 0.3), size=3 * K) + 1e-30)
    check_scores(P, X, K, logtheta, 2.0 ** -21)


@pytest.mark.parametrize("N,D,K,deep", [(38989, 330, 10, 0), (38989, 330, 40, 0),
                                        (38989, 330, 10, 300), (20001, 650, 40, 200)])
def test_scores_repeat_bit_for_bit(P, N, D, K, deep):
    """Every hand-over between the label kernel's roles is ordered (entries -> A stage
    -> MMA -> epilogue, and each buffer back): a stage read before it is complete or
    refilled while it is read shows as another score.  The same call ten times, with
    segments in fixed slots and, where some cells are many times as deep as the
    others, end to end in the ring."""
    rng = np.random.default_rng([N, K, deep])
    X = sparse(N, D, 40.0 / D, rng)
    if deep:
        from scipy.sparse import csr_matrix, vstack
        full = csr_matrix(rng.integers(1, 200, size=(deep, D)).astype(np.float64))
        X = vstack([X[:N - deep], full], format="csr")[rng.permutation(N)]
    g = P.Sampler(X.indptr.astype(np.int32), X.indices.astype(np.int32), X.data.astype(np.int32),
                  N, D, 1.0, 0.5, kmax=64, seed=3, engine=P.ENGINE_TILE_BF16)
    g.set_state(np.arange(N) % K, np.zeros(N, np.uint8), K)
    logtheta = np.log(rng.dirichlet(np.full(D, 0.3), size=3 * K) + 1e-30)
    P.dpmm_set_params(g.ctx, np.full(K + 1, -np.log(K + 1.0)), logtheta)
    first = P.dpmm_debug_tile_scores(g.ctx, N, K)
    for _ in range(9):
        np.testing.assert_array_equal(P.dpmm_debug_tile_scores(g.ctx, N, K), first)
    g.close()


@pytest.mark.parametrize("N,D,K,big", [(300, 200, 5, 40), (38989, 130, 10, 3000),
                                       (2000, 500, 40, 20000)])
def test_second_planes(P, N, D, K, big):
    """Counts above 2,047: few, in many items of a CTA (more than the second
    planes' stages), in nearly every item."""
    rng = np.random.default_rng([N, big])
    X = sparse(N, D, min(1.0, 40.0 / D), rng, big=big)
    logtheta = np.log(rng.dirichlet(np.full(D, 0.3), size=3 * K) + 1e-30)
    check_scores(P, X, K, logtheta, 2.0 ** -21)


@pytest.mark.parametrize("N,D,K", [(300, 200, 5), (20001, 130, 40)])
def test_bf16_where_log_theta_passes_fp16(P, N, D, K):
    """A log theta of -1e6 (a hopeless gene of one row) takes BF16 operands for
    every row; counts above 255 take a second plane there."""
    rng = np.random.default_rng([N, 9])
    X = sparse(N, D, min(1.0, 40.0 / D), rng, big=60, top=3000)
    logtheta = np.log(rng.dirichlet(np.full(D, 0.3), size=3 * K) + 1e-30)
    logtheta[1, 3] = -1e6
    check_scores(P, X, K, logtheta, 2.0 ** -15)


def test_small_beta_draws_take_bf16(P):
    """beta = 1e-4: drawn log theta values lie beyond FP16's range; the chain
    keeps finding the planted clusters."""
    from paper_1812_10048_gb300 import synth
    ds = synth.make_dataset(1500, 200, 4, gamma=0.1, lib_mu=np.log(800.0), lib_sigma=0.5, seed=3)
    s = P.Sampler(ds.indptr, ds.indices, ds.data, ds.N, ds.D, 1.0, 1e-4, kmax=32, seed=5,
                  engine=P.ENGINE_TILE_BF16)
    s.set_state(ds.labels, np.random.default_rng(1).integers(0, 2, ds.N).astype(np.uint8), 4)
    s.step(20)
    labels, K = s.labels()
    s.close()
    from oracle.ari import adjusted_rand_index
    assert adjusted_rand_index(labels, ds.labels) > 0.98


def test_batch_whose_first_chain_has_no_blocked_copy(P):
    """Unpackable counts in the first dataset: the others still go to the
    tensor cores, each evolving as alone."""
    rng = np.random.default_rng(8)
    data = []
    for i, N in enumerate([300, 700, 150]):
        X = sparse(N, 200, 0.2, rng)
        if i == 0:
            X.data[5] = 70000
        data.append((X.indptr.astype(np.int32), X.indices.astype(np.int32),
                     X.data.astype(np.int32), N))
    b = P.BatchSampler(data, 200, 1.0, 0.5, kmax=16, seed=3, engine=P.ENGINE_TILE_BF16)
    b.step(6)
    for i, d in enumerate(data):
        s = P.Sampler(*d[:3], d[3], 200, 1.0, 0.5, kmax=16, seed=3, chain_id=i,
                      engine=P.ENGINE_TILE_BF16)
        s.step(6)
        assert P.dpmm_debug_engine(b.chain(i).ctx) == (i > 0)
        for x, y in zip(s.get_state(), b.chain(i).get_state()):
            np.testing.assert_array_equal(x, y)
        s.close()
    b.close()
