"""Cluster statistics of the log ML counted in shared memory: sizes around the
kernel's edges (one or several cluster groups, rows longer than a warp's batch,
ragged flush tails, empty rows and clusters), totals of 2^32 and more, and the
range of beta, against the FP64 oracle."""

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


def matrix(N, D, K, rng, longest):
    length = rng.integers(1, min(D, longest) + 1, size=N)
    length[3::7] = 0
    indptr = np.concatenate([[0], np.cumsum(length)]).astype(np.int32)
    idx = np.concatenate([rng.permutation(D)[:l] for l in length] + [np.zeros(0, int)])
    val = rng.integers(0, 40, size=idx.size)
    labels = rng.integers(0, K, size=N)
    labels[labels == K // 2] = 0                      # an empty cluster
    return indptr, idx.astype(np.int32), val.astype(np.int32), labels.astype(np.int32)


def both(P, arrs, N, D, K, la, lb):
    """Value and gradients from the allocation-free call and from LogML."""
    import torch
    dev = [torch.from_numpy(a).cuda() for a in arrs]
    lbt, gb = torch.from_numpy(lb).cuda(), torch.empty(D, dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    v, ga = P.dpmm_logml_grad_noalloc(*dev[:3], N, D, dev[3], K, la, lbt, gb)
    h = P.LogML(*arrs[:3], N, D, arrs[3], K)
    gb2 = np.empty(D, np.float32)
    v2, ga2 = h.forward(la, lb), h.backward(la, lb, gb2)
    h.close()
    assert (v2, ga2) == (v, ga)                       # the same kernels, block order fixed
    np.testing.assert_array_equal(gb.cpu().numpy(), gb2)
    return v, ga, gb2


def check(got, arrs, N, D, K, la, lb):
    from oracle.logml import cluster_stats, log_ml, log_ml_grad
    n, S = cluster_stats(*arrs[:3], N, D, arrs[3], K)
    ref = log_ml(n, S, la, lb.astype(np.float64))
    ga, gb = log_ml_grad(n, S, la, lb.astype(np.float64))
    # FP64 sums of at most K D terms of both signs, none above |lgamma(total)|
    assert abs(got[0] - ref) <= 1e-12 * abs(ref) + 1e-9
    assert abs(got[1] - ga) <= 1e-9 * max(1.0, abs(ga))
    np.testing.assert_allclose(got[2], gb, rtol=2e-4, atol=1e-3)


@pytest.mark.parametrize("N,D,K,longest", [
    (1, 1, 1, 1),            # a single counter
    (129, 63, 3, 63),        # a ragged flush tail (189 words)
    (700, 1025, 5, 900),     # rows over the 256 entries a warp loads at once
    (3000, 3001, 60, 40),    # four groups of clusters
    (2000, 333, 1024, 30),   # many clusters, two groups
    (300, 65536, 3, 50),     # one cluster's counters do not fit: global memory
])
def test_counts_match_oracle(P, N, D, K, longest):
    rng = np.random.default_rng([N, D, K])
    arrs = matrix(N, D, K, rng, longest)
    lb = (np.log(0.1) + 0.1 * rng.standard_normal(D)).astype(np.float32)
    check(both(P, arrs, N, D, K, 0.3, lb), arrs, N, D, K, 0.3, lb)


def test_total_of_2_to_32_without_a_wrapped_gene(P):
    """One cluster's counts reach 2^32 in all while no gene's do: the exact
    global count answers; a caller may pass one buffer for beta and gradient."""
    import torch
    n, D = 70000, 2
    arrs = [(2 * np.arange(n + 1)).astype(np.int32), np.tile([0, 1], n).astype(np.int32),
            np.full(2 * n, 40000, np.int32), np.zeros(n, np.int32)]
    lb = np.array([-1.0, 0.5], np.float32)
    dev = [torch.from_numpy(a).cuda() for a in arrs]
    buf = torch.from_numpy(lb).cuda()
    torch.cuda.synchronize()
    v, ga = P.dpmm_logml_grad_noalloc(*dev[:3], n, D, dev[3], 1, 0.3, buf, buf)
    check((v, ga, buf.cpu().numpy()), arrs, n, D, 1, 0.3, lb)


@pytest.mark.parametrize("log_beta", [-60.0, -20.0, -2.0, 0.0, 2.7, 9.0, 30.0])
def test_lgamma_forms_over_beta(P, log_beta):
    """Small and large counts at beta from 1e-26 to 1e13."""
    rng = np.random.default_rng(3)
    D, K = 24, 2
    val = np.concatenate([np.arange(1, D + 1), 2 ** np.arange(D) % 65521 + 1]).astype(np.int32)
    arrs = [np.array([0, D, 2 * D], np.int32), np.tile(np.arange(D), 2).astype(np.int32), val,
            np.array([0, 1], np.int32)]
    lb = (log_beta + 0.1 * rng.standard_normal(D)).astype(np.float32)
    got = both(P, arrs, 2, D, K, -0.4, lb)
    from oracle.logml import cluster_stats, log_ml
    from scipy.special import gammaln
    n, S = cluster_stats(*arrs[:3], 2, D, arrs[3], K)
    b = np.exp(lb.astype(np.float64))
    # the oracle subtracts lgammas: its own rounding, a few ulps of the largest
    scale = np.abs(gammaln(b + S)).sum() + K * np.abs(gammaln(b)).sum() + \
        np.abs(gammaln(b.sum() + S.sum(1))).sum()
    assert abs(got[0] - log_ml(n, S, -0.4, lb.astype(np.float64))) <= 4e-15 * scale + 1e-12
