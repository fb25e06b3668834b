"""Float32 search where the parents of a round share most of their neighbours: every id comes once, the answers
are the exact ones when the beam holds the whole database, and no launch shape changes them.  Dimensions on
both sides of the scorer's sizes (128, 256, 512, 768 and 1024 floats a record).  Scores within D 2^-23 of ||q|| ||x||
(float32 products and sums)."""
import numpy as np
import pytest
import torch

from gpu_util import t

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [100, 128, 129, 512, 768, 769, 1000])
@pytest.mark.parametrize("W", [1, 2, 3, 4])
@pytest.mark.parametrize("metric", [0, 1])
def test_shared_neighbours(D, W, metric):
    import paper_2312_16335_gb300 as lv
    n, R, m = 400, 32, 25
    rng = np.random.default_rng(D + W)
    X = rng.standard_normal((n, D)).astype(np.float32)
    Q = rng.standard_normal((m, D)).astype(np.float32)
    hubs = rng.permutation(n)[:24]  # in every row: most ids of a round come from several parents
    adj = np.stack([np.concatenate([hubs, (i + 1 + np.arange(8)) % n]) for i in range(n)]).astype(np.int32)
    idx = lv.Index(0, metric=metric).encode_fp32(t(X)).set_graph(t(adj), 5)
    exact = Q.astype(np.float64) @ X.astype(np.float64).T
    if metric:
        exact = 2 * exact - (X.astype(np.float64) ** 2).sum(1)
    tol = 2 * D * 2.0 ** -23 * np.linalg.norm(Q, axis=1)[:, None] * np.linalg.norm(X, axis=1).max()
    if metric:
        tol = tol + D * 2.0 ** -23 * (X.astype(np.float64) ** 2).sum(1).max()
    ids, sc = idx.search(t(Q), None, k=n, L=n, width=W)
    assert idx.sync_status() == 0
    a, s = ids.cpu().numpy(), sc.cpu().numpy()
    assert (np.sort(a, 1) == np.arange(n)).all()  # every id, once
    assert (np.abs(np.take_along_axis(exact, a, 1) - s) <= tol).all() and (np.diff(s, axis=1) <= 0).all()
    for L in (20, 33, 64):
        want = idx.search(t(Q), None, k=10, L=L, width=W)
        shapes = [dict(visited_bits=16), dict(hash_slots=256), dict(warps_per_block=2)]
        if W % 2 == 0:
            shapes.append(dict(warps_per_query=2))
        for kw in shapes:
            got = idx.search(t(Q), None, k=10, L=L, width=W, **kw)
            assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1]), (L, kw)
        assert all(len(set(r)) == 10 for r in want[0].tolist())
