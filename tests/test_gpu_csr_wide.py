"""CSR label kernel.  With the cluster table in slabs (K > 32, or tables beyond
shared memory): slab widths from one to sixteen float4s, several slabs, odd
kmax (no 16-byte table rows), unpacked counts, rows around the pieces a warp
holds, fewer cells than blocks, tables that fit not even one slab.  With the
tables held (K <= 32): the edges of each number of lanes an entry, rows past the
registers.  Every label and sub-label against the FP64 decision."""

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


@pytest.mark.parametrize("N,D,K,kmax,longest,big", [
    (900, 200, 60, 64, 200, 0),       # one slab of sixteen float4s
    (900, 1000, 64, 64, 300, 0),      # two of eight
    (900, 1000, 41, 131, 257, 0),     # kmax not a multiple of four
    (5000, 1000, 33, 64, 129, 0),     # 32 cells a warp and more
    (120, 3000, 50, 64, 400, 0),      # fewer cells than blocks, slabs of four
    (700, 6000, 45, 48, 100, 0),      # slabs of two
    (700, 12000, 34, 64, 100, 0),     # slabs of one
    (700, 12000, 7, 16, 100, 0),      # K <= 32 with a table beyond shared memory
    (400, 16000, 40, 64, 100, 0),     # no slab fits: from global memory
    (900, 1000, 64, 64, 300, 70000),  # unpacked entries
    # K <= 32 with the tables in shared memory: one to eight lanes an entry
    (900, 333, 1, 1, 300, 0),
    (900, 333, 4, 5, 257, 0),
    (900, 333, 5, 7, 300, 0),
    (900, 333, 8, 8, 256, 0),
    (900, 333, 9, 33, 300, 0),
    (120, 333, 16, 16, 300, 0),       # fewer cells than blocks
    (900, 333, 17, 19, 300, 0),
    (900, 1000, 32, 32, 300, 0),      # the sub-cluster table stays in global memory
    (900, 333, 3, 4, 300, 70000),     # unpacked entries
    (900, 333, 7, 8, 300, 70000),
    (900, 333, 13, 16, 300, 70000),
    (900, 333, 27, 32, 300, 70000),
    (160000, 50, 6, 8, 33, 0),        # more than 1,024 cells a block
])
def test_labels_match_fp64(P, N, D, K, kmax, longest, big):
    from scipy.sparse import csr_matrix
    from .parity import assert_decisions, fp32_bound, fp64_decisions
    rng = np.random.default_rng([N, D, K])
    length = rng.integers(0, longest + 1, size=N)
    length[:8] = [0, 1, 31, 32, 33, min(longest, 127), min(longest, 128), longest]
    indptr = np.concatenate([[0], np.cumsum(length)]).astype(np.int32)
    idx = np.concatenate([rng.choice(D, l, replace=False) for l in length]).astype(np.int32)
    val = rng.integers(0, 7, size=idx.size).astype(np.int32)
    if big:
        val[rng.integers(0, val.size, 5)] = big
    lab = np.arange(N) % K
    sub = rng.integers(0, 2, N).astype(np.uint8)
    s = P.Sampler(indptr, idx, val, N, D, 1.0, 0.5, kmax=kmax, seed=4, chain_id=3,
                  engine=P.ENGINE_CSR_FP32)
    s.set_state(lab, sub, K, t=2)
    nsub, _, _ = s.stats()
    P.dpmm_draw_params(s.ctx)
    logpi, logtheta = P.dpmm_get_params(s.ctx, K, D)
    P.dpmm_assign(s.ctx)
    got_lab, got_sub, Kg, _, _ = s.get_state()
    n2, S2, _ = s.stats()
    s.close()
    X = csr_matrix((val.astype(np.float64), idx.copy(), indptr), shape=(N, D))
    th = logtheta.astype(np.float64)
    ref = fp64_decisions(X, np.arange(N), logpi.astype(np.float64), th, lab, sub,
                         nsub.astype(np.int64), K, 4, 3, 2, fp32_bound(X, th))
    keep = np.bincount(ref["lab"], minlength=K) > 0
    assert Kg == keep.sum()
    pre = np.nonzero(keep)[0][got_lab]
    n = np.stack([np.bincount(ref["lab"][ref["sub"] == r], minlength=K) for r in (0, 1)], 1)
    reset = (n.sum(1) >= 2) & (n.min(1) == 0)          # these redraw their sub-labels
    got_sub = np.where(reset[ref["lab"]], ref["sub"], got_sub)
    assert_decisions(ref, pre, got_sub)
    np.testing.assert_array_equal(n2.sum(1), np.bincount(got_lab, minlength=Kg))
    tot = np.zeros((Kg, D), np.int64)
    rows = np.repeat(got_lab, length)
    np.add.at(tot, (rows, idx), val)
    np.testing.assert_array_equal(S2.astype(np.int64).sum(1), tot)


@pytest.mark.parametrize("engine", ["csr", "tile"])
@pytest.mark.parametrize("D,K", [(300, 5), (300, 40), (300, 70), (20001, 5), (20001, 40)])
@pytest.mark.parametrize("value", [np.nan, -np.inf])
def test_scores_without_an_order(P, engine, D, K, value):
    """Parameters that leave a cell no finite score (every form of the label step): it
    takes cluster 0 of the table, and the statistics follow."""
    rng = np.random.default_rng(D + K)
    N = 300
    idx = np.sort(rng.integers(0, D // 8, size=(N, 8)) + np.arange(8) * (D // 8), axis=1)
    csr = (np.arange(0, 8 * N + 1, 8, dtype=np.int32), idx.astype(np.int32).ravel(),
           np.ones(8 * N, np.int32))
    s = P.Sampler(*csr, N, D, 1.0, 0.5, kmax=80, seed=3,
                  engine=P.ENGINE_CSR_FP32 if engine == "csr" else P.ENGINE_TILE_BF16)
    s.set_state(np.arange(N) % K, np.zeros(N, np.uint8), K, 1)
    P.dpmm_set_params(s.ctx, np.zeros(K + 1, np.float32),
                      np.full((3 * K, D), value, np.float32))
    P.dpmm_assign(s.ctx)
    labels, sub, Kn, _, _ = s.get_state()
    assert Kn == 1 and not labels.any()
    assert s.stats()[0].sum() == N and s.stats()[1].sum() == 8 * N
    s.close()
