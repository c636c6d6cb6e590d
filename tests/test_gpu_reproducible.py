"""The same inputs and seed give the same bits in every version: CRC-32 of label
steps, parameter draws and chains on inputs made of integers and exact binary
fractions, against recorded ones (tests/golden/chain_crc.txt; a line is written by
`line(P, name)`)."""

import os
import zlib

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "chain_crc.txt")

# name: (kind, N, D, K, entries a row, largest count)
CASES = {
    "assign_13": ("assign", 5003, 1237, 13, 60, 9),
    "assign_40_large_counts": ("assign", 2501, 700, 40, 50, 3000),
    "assign_3_deep": ("assign", 1300, 3000, 3, 700, 300),
    "draw_2048": ("draw", 900, 2048, 5, 40, 9),
    "draw_2049": ("draw", 900, 2049, 5, 40, 9),
    "draw_5003": ("draw", 900, 5003, 5, 40, 9),
    "draw_9001": ("draw", 900, 9001, 3, 40, 9),
    "draw_32738": ("draw", 900, 32738, 3, 40, 9),
    "draw_70001": ("draw", 300, 70001, 2, 40, 9),
    "local_5003": ("local", 900, 5003, 5, 40, 9),
    "chain_400": ("chain", 1500, 400, 6, 50, 40),
    "chain_5003": ("chain", 900, 5003, 4, 200, 40),
    "csr_chain_400": ("csr", 1500, 400, 6, 50, 40),
}


@pytest.fixture(scope="module")
def P():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1812_10048_gb300 import build
    build.build()
    import paper_1812_10048_gb300 as P
    return P


def mix(x):
    """A 32-bit integer hash (multiply and xor-shift)."""
    x = np.asarray(x, np.uint64)
    for m in (0x7FEB352D, 0x846CA68B):
        x = ((x ^ (x >> np.uint64(16))) * np.uint64(m)) & np.uint64(0xFFFFFFFF)
    return x ^ (x >> np.uint64(15))


def matrix(N, D, K, per_row, top):
    """CSR whose cells of cluster k prefer the genes k mod K; (csr, labels, sub-labels)."""
    lab = (mix(np.arange(N)) % np.uint64(K)).astype(np.int64)
    lab[:K] = np.arange(K)
    rows, cols, vals = [], [], []
    for i in range(N):
        h = mix(np.arange(2 * per_row, dtype=np.uint64) + np.uint64(i * 7919 + 17))
        u = (h % np.uint64(D)).astype(np.int64)
        half = per_row // 2                       # half of the entries on the cluster's genes
        u[:half] = np.minimum(u[:half] // K * K + lab[i], D - 1)
        u = np.unique(u[:per_row])
        x = 1 + (mix(u.astype(np.uint64) * np.uint64(31) + np.uint64(i)) % np.uint64(9))
        big = mix(u.astype(np.uint64) + np.uint64(i * 13)) % np.uint64(50) == 0
        x = np.where(big, 1 + mix(u.astype(np.uint64) + np.uint64(i)) % np.uint64(top), x)
        rows.append(u.size)
        cols.append(u)
        vals.append(x)
    indptr = np.concatenate([[0], np.cumsum(rows)]).astype(np.int32)
    sub = (mix(np.arange(N) + 5) % np.uint64(2)).astype(np.uint8)
    return (indptr, np.concatenate(cols).astype(np.int32), np.concatenate(vals).astype(np.int32),
            lab, sub)


def crc(arrays):
    c = 0
    for a in arrays:
        c = zlib.crc32(np.ascontiguousarray(a).tobytes(), c)
    return c


def line(P, name):
    kind, N, D, K, per_row, top = CASES[name]
    *csr, lab, sub = matrix(N, D, K, per_row, top)
    s = P.Sampler(*csr, N, D, 1.0, 0.5, kmax=64, seed=11, chain_id=3,
                  local_iters=2 if kind == "local" else 1,
                  engine=P.ENGINE_CSR_FP32 if kind == "csr" else P.ENGINE_TILE_BF16
                  if kind == "assign" else P.ENGINE_AUTO)
    s.set_state(lab, sub, K, 4)
    if kind == "assign":
        # log theta in steps of 1 / 256 (exact in FP32)
        h = mix(np.arange(3 * K * D, dtype=np.uint64)).reshape(3 * K, D)
        logtheta = -(h % np.uint64(4096)).astype(np.float32) / 256
        P.dpmm_set_params(s.ctx, np.full(K + 1, -2.0, np.float32), logtheta)
        P.dpmm_assign(s.ctx)
    elif kind == "draw":
        P.dpmm_draw_params(s.ctx)
    elif kind == "local":
        s.sweep(1)
        lab, sub, K = s.get_state()[:3]
    else:
        s.step(12)
    if kind in ("draw", "local"):
        out = list(P.dpmm_get_params(s.ctx, K, D)) + list(s.get_state()[:2])
    else:
        st = s.get_state()
        out = [st[0], st[1], np.array(st[2:], np.int64)] + list(s.stats())
    s.close()
    return "%s %08x" % (name, crc(out))


@pytest.mark.parametrize("name", list(CASES))
def test_same_bits_as_recorded(P, name):
    with open(GOLDEN) as f:
        assert line(P, name) in f.read().split("\n")
