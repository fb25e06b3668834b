"""Small batches run with a block per query (beam_block_kernel): ids and scores equal those of a warp
per query bit for bit, over widths, degrees, beams, encodings, metrics, budgets, descriptors and
graphs with repeated neighbours between parents."""
import numpy as np
import pytest
import torch

from gpu_util import t

pytestmark = pytest.mark.gpu


def _setup(lv, n, D, d, bits, R, metric, m, seed):
    rng = np.random.default_rng(seed)
    c = rng.standard_normal((12, D))
    X = (c[rng.integers(0, 12, n)] + 0.5 * rng.standard_normal((n, D))).astype(np.float32)
    Q = (c[rng.integers(0, 12, m)] + 0.5 * rng.standard_normal((m, D))).astype(np.float32)
    P = np.linalg.qr(rng.standard_normal((D, d)))[0].T.astype(np.float32)
    # every second neighbour near, the rest random: parents share many neighbours
    adj = np.concatenate([(np.arange(n)[:, None] + 1 + np.arange(R // 2)) % n, rng.integers(0, n, (n, R - R // 2))], 1)
    adj[rng.random((n, R)) < 0.1] = -1
    return lv.Index(0, metric=metric).encode(t(X), t(P), bits, 8).set_graph(t(adj.astype(np.int32)), 3), t(Q), t(P)


@pytest.mark.parametrize("n,D,d,bits,R,metric", [
    (2000, 64, 16, 8, 32, 0), (2000, 64, 40, 8, 64, 1), (3000, 200, 160, 8, 64, 0), (1500, 256, 240, 8, 33, 0),
    (1500, 256, 224, 8, 17, 1), (2000, 128, 30, 4, 128, 0), (2000, 400, 350, 4, 50, 0), (70, 16, 8, 8, 128, 0),
])
@pytest.mark.parametrize("W,L,k,r,hops", [(1, 1, 1, 1, 0), (1, 50, 10, 50, 0), (2, 31, 5, 0, 7), (2, 128, 100, 128, 64),
                                          (2, 300, 10, 290, 0), (1, 512, 33, 512, 40)])
def test_block_equals_warp(n, D, d, bits, R, metric, W, L, k, r, hops):
    import paper_2312_16335_gb300 as lv
    idx, Q, P = _setup(lv, n, D, d, bits, R, metric, 37, seed=n + D + R + L)
    kw = dict(k=k, L=L, rerank=r, max_hops=hops, width=W)
    a = idx.search(Q, P, **kw)
    b = idx.search(Q, P, queries_per_warp=1, **kw)
    assert idx.sync_status() == 0
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])


def test_block_descriptors_and_bad_queries():
    import paper_2312_16335_gb300 as lv
    idx, Q, P = _setup(lv, 2000, 64, 24, 8, 64, 0, 60, seed=5)
    rng = np.random.default_rng(1)
    L = rng.integers(1, 201, 60)
    kk = np.minimum(L, rng.integers(1, 60, 60))
    desc = t(np.stack([kk, L, rng.integers(0, L + 1), rng.integers(0, 90, 60)], 1).astype(np.int32))
    Q[7, 3] = float("nan")
    Q[11] = 0.0
    Q[12] *= 1e30
    a = idx.search(Q, P, k=60, L=200, rerank=200, desc=desc, width=2)
    b = idx.search(Q, P, k=60, L=200, rerank=200, desc=desc, width=2, queries_per_warp=1)
    assert idx.sync_status() == 0
    ok = torch.arange(60, device="cuda") != 7  # the scores of a query with NaN order nothing
    assert torch.equal(a[0][ok], b[0][ok]) and torch.equal(a[1][ok], b[1][ok])
    assert bool(((a[0] >= -1) & (a[0] < 2000)).all())
