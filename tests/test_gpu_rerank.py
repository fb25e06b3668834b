"""The rerank kernel at its edges (groups of four records shared by four warps, a two-stage ring,
top k by rounds or by ranks) against the FP64 scores of the beam's own candidates.

The candidates are the beam itself (the same search without rerank, k = L).  Tolerance: scores within
1e-4 ||q|| ||x|| (24-bit fixed-point query, float32 sums), as for every rerank; two candidates closer
than twice that may change places."""
import numpy as np
import pytest
import torch

from gpu_util import t

pytestmark = pytest.mark.gpu

N = 700


def _index(lv, D, sbits, metric, seed):
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((N, D)).astype(np.float32)
    X /= np.linalg.norm(X, axis=1, keepdims=True)
    Q = rng.standard_normal((9, D)).astype(np.float32)
    d = min(D, 24)
    P = np.linalg.qr(rng.standard_normal((D, d)))[0].T.astype(np.float32)
    adj = np.stack([np.concatenate([[(i + 1) % N], rng.choice(N, 31, replace=False)]) for i in range(N)]).astype(np.int32)
    idx = lv.Index(0, metric=metric).encode(t(X), t(P), 8, sbits)
    idx.set_graph(t(adj), 0)
    if sbits == 16:
        dec = X.astype(np.float16).astype(np.float64)
        norms = (dec ** 2).sum(1)
    else:
        rec = idx.secondary_records().cpu().numpy()
        co = (D + 15) // 16 * 16
        cst = np.ascontiguousarray(rec[:, co:co + 16]).view(np.float32).astype(np.float64)
        mean = lv.leanvec_column_mean(t(X)).cpu().numpy().astype(np.float64)
        dec = mean + cst[:, 1:2] + cst[:, 0:1] * rec[:, :D].astype(np.float64)
        norms = (X.astype(np.float64) ** 2).sum(1)
    return idx, t(Q), t(P), Q.astype(np.float64), dec, norms


@pytest.mark.parametrize("D,sbits,metric", [(17, 8, 0), (512, 8, 0), (528, 8, 1), (1008, 8, 0), (40, 16, 0), (1024, 16, 1)])
@pytest.mark.parametrize("r,k", [(1, 1), (3, 3), (4, 2), (5, 5), (17, 10), (64, 32), (65, 33), (128, 128), (509, 100), (512, 20)])
def test_rerank_edges(D, sbits, metric, r, k):
    import paper_2312_16335_gb300 as lv
    idx, Q, P, Qd, dec, norms = _index(lv, D, sbits, metric, seed=D + r)
    beam = idx.search(Q, P, k=r, L=r, rerank=0)[0].cpu().numpy()
    ids, sc = (x.cpu().numpy() for x in idx.search(Q, P, k=k, L=r, rerank=r, ldo=k + 3))
    assert idx.sync_status() == 0
    assert (ids[:, k:] == -1).all() and np.isneginf(sc[:, k:]).all()
    tol = 1e-4 * np.linalg.norm(Qd, axis=1)[:, None] * np.sqrt(norms.max()) * (2 if metric else 1)
    for j in range(Q.shape[0]):
        cand = beam[j][beam[j] >= 0]
        exact = dec[cand] @ Qd[j]
        if metric:
            exact = 2 * exact - norms[cand]
        got, s = ids[j, :k], sc[j, :k]
        m = min(k, len(cand))
        assert (got[m:] == -1).all() and len(set(got[:m])) == m and set(got[:m]) <= set(cand)
        pos = {int(c): i for i, c in enumerate(cand)}
        e = np.array([exact[pos[int(g)]] for g in got[:m]])
        assert np.abs(s[:m] - e).max() <= tol[j]
        assert (np.diff(s[:m]) <= 0).all()
        assert np.sort(exact)[::-1][m - 1] <= e.min() + 2 * tol[j]
