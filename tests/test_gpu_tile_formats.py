"""Dense-tile engine: BF16 hi + lo operands (any range of log theta, their error
against FP64), second planes of large counts, and the item order's edges (tiles in
pairs or alone, one, two or an odd number of chunks), scores against FP64."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# hi + lo against the FP32 value: two roundings to BF16's eight bits, 2^-18, and as
# much for the two products' sum
EPS = 2.0 ** -17


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
def test_scores(P, N, D, K):
    rng = np.random.default_rng([N, D, K])
    X = sparse(N, D, min(1.0, 40.0 / D), rng)
    logtheta = np.log(rng.dirichlet(np.full(D, 0.3), size=3 * K) + 1e-30)
    check_scores(P, X, K, logtheta, EPS)


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
    """Counts above 255: few, in many items of a CTA (more than the second
    planes' stages), in nearly every item."""
    rng = np.random.default_rng([N, big])
    X = sparse(N, D, min(1.0, 40.0 / D), rng, big=big)
    logtheta = np.log(rng.dirichlet(np.full(D, 0.3), size=3 * K) + 1e-30)
    check_scores(P, X, K, logtheta, EPS)


@pytest.mark.parametrize("N", [700, 38989])
@pytest.mark.parametrize("density", [0.33, 0.5, 0.9])
def test_second_planes_of_long_segments(P, N, density):
    """Segments so long that a producer set has one stage (four sets, then two) or two sets
    have two: the second plane takes the set's next stage, or the same one again."""
    rng = np.random.default_rng([N, int(100 * density)])
    D, K = 140, 40
    X = sparse(N, D, density, rng, big=N)
    logtheta = np.log(rng.dirichlet(np.full(D, 0.3), size=3 * K) + 1e-30)
    check_scores(P, X, K, logtheta, EPS)


@pytest.mark.parametrize("N,D,K", [(300, 200, 5), (20001, 130, 40)])
def test_log_theta_of_any_size(P, N, D, K):
    """A log theta of -1e6 (a hopeless gene of one row) beside ordinary ones, counts
    above 255 among them."""
    rng = np.random.default_rng([N, 9])
    X = sparse(N, D, min(1.0, 40.0 / D), rng, big=60, top=3000)
    logtheta = np.log(rng.dirichlet(np.full(D, 0.3), size=3 * K) + 1e-30)
    logtheta[1, 3] = -1e6
    check_scores(P, X, K, logtheta, EPS)


def test_chain_of_small_beta(P):
    """beta = 1e-4: drawn log theta values reach -1e5; the chain
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


def operand_errors(P, N, D, K, lib, seed):
    """(tile scores less the 64-bit sums of the same FP32 centred values, that
    difference for exactly summed BF16 hi + lo operands), own cluster and the
    difference of its two sub-clusters; per cell."""
    from scipy.sparse import csr_matrix
    from paper_1812_10048_gb300 import synth
    ds = synth.make_dataset(N, D, K, gamma=0.05, lib_mu=np.log(lib), lib_sigma=0.3, seed=seed)
    X = csr_matrix((ds.data.astype(np.float64), ds.indices, ds.indptr), shape=(N, D))
    s = P.Sampler(ds.indptr, ds.indices, ds.data, N, D, 1.0, 0.1, kmax=64, seed=seed,
                  engine=P.ENGINE_TILE_BF16)
    s.set_state(ds.labels, np.random.default_rng(seed).integers(0, 2, N).astype(np.uint8), K, 1)
    P.dpmm_draw_params(s.ctx)
    L = P.dpmm_get_params(s.ctx, K, D)[1]
    got = P.dpmm_debug_tile_scores(s.ctx, N, K).astype(np.float64)
    s.close()
    order = np.concatenate([np.arange(0, 3 * K, 3),
                            np.stack([np.arange(1, 3 * K, 3), np.arange(2, 3 * K, 3)], 1).ravel()])
    L = L[order]
    # m_u as the kernel forms it: four FP32 sums of every fourth row
    q = []
    for j in range(4):
        acc = np.zeros(D, np.float32)
        for r in range(j, 3 * K, 4):
            acc = acc + L[r]
        q.append(acc)
    d = L - ((q[0] + q[1]) + (q[2] + q[3])) / np.float32(3 * K)
    hi = to_bf16(d)
    lo = to_bf16(d - hi)
    err = got - X @ d.astype(np.float64).T
    model = X @ (hi.astype(np.float64) + lo - d).T
    c, at = ds.labels, np.arange(N)
    out = []
    for e in (err, model):
        out.append((e[at, c], e[at, K + 2 * c] - e[at, K + 2 * c + 1]))
    return out


def to_bf16(x):
    b = np.ascontiguousarray(x, np.float32).view(np.uint32).astype(np.uint64)
    b = (b + 0x7FFF + ((b >> 16) & 1)) & 0xFFFF0000          # nearest, ties to even
    return b.astype(np.uint32).view(np.float32)


@pytest.mark.parametrize("N,D,K,lib", [(4000, 3000, 3, 3000.0), (4000, 1000, 12, 1000.0)])
def test_score_error_is_that_of_the_operands(P, N, D, K, lib):
    """The error against 64 bits is the hi + lo operands' own: the FP32 accumulator adds
    little to it even where few clusters meet many counts (scores of 1e4 and more)."""
    (own, diff), (own_model, diff_model) = operand_errors(P, N, D, K, lib, 31)

    def rms(x):
        return np.sqrt(np.mean(x * x))
    print("rms own %.3e (operands %.3e), difference %.3e (operands %.3e)"
          % (rms(own), rms(own_model), rms(diff), rms(diff_model)))
    assert rms(own) <= 2.0 * rms(own_model)
    assert rms(diff) <= 2.0 * rms(diff_model)


def test_label_step_after_a_local_iteration_of_small_beta(P):
    """beta = 3e-5: theta-bar redrawn by a local iteration after ordinary parameters were
    set holds values below -65,504; the label step that follows agrees with FP64."""
    from oracle.sampler import Sampler as OracleSampler, sufficient_stats
    from paper_1812_10048_gb300 import synth
    from .parity import bf16_bound, check_assign, decisions_from_oracle
    K, beta = 4, 3e-5
    ds = synth.make_dataset(1500, 400, K, gamma=0.1, lib_mu=np.log(800.0), lib_sigma=0.5, seed=3)
    sub = np.random.default_rng(1).integers(0, 2, ds.N)
    o = OracleSampler(ds.indptr, ds.indices, ds.data, ds.N, ds.D, 1.0, beta, seed=5, kmax=32)
    o.set_state(ds.labels, sub, K, t=3, m=1)
    s = P.Sampler(ds.indptr, ds.indices, ds.data, ds.N, ds.D, 1.0, beta, kmax=32, seed=5,
                  engine=P.ENGINE_TILE_BF16, local_iters=2)
    s.set_state(ds.labels, sub.astype(np.uint8), K, 3, 1)
    S = s.stats()[1].astype(np.float64)
    rows = np.concatenate([S.sum(1, keepdims=True), S], 1).reshape(3 * K, ds.D) + 0.5
    logtheta = np.log(rows / rows.sum(1, keepdims=True))
    logpi = np.log(np.full(K + 1, 1.0 / (K + 1)))
    P.dpmm_set_params(s.ctx, logpi, logtheta)
    P.dpmm_assign(s.ctx)
    P.dpmm_local_gibbs(s.ctx, 1)
    state = s.get_state()
    assert state[2] == K
    logpi, logtheta = (x.astype(np.float64) for x in P.dpmm_get_params(s.ctx, K, ds.D))
    assert logtheta.min() < -65504
    o.set_state(*state[:3], t=state[3], m=state[4])
    ref = decisions_from_oracle(o, logpi, logtheta, bf16_bound(o.X.astype(np.float64), logtheta))
    P.dpmm_assign(s.ctx)
    lab, sb, Kg, t, m = s.get_state()
    nsub, Ssub, sq = s.stats()
    check_assign(ref, K, Kg, lab, sb, sq, o.seed, o.chain_id, state[3])
    on, oS = sufficient_stats(o.X, lab, sb, Kg)
    np.testing.assert_array_equal(nsub, on)
    np.testing.assert_array_equal(Ssub, oS)
    s.close()
