"""A score that is not a number counts as -infinity in every launch shape of the search and in the rerank: such
records come last, by id among themselves, and all shapes give the same answers bit for bit.  The records with
such scores are rows with an infinite entry, in the primaries, in the secondaries, or in both, and all of them
for a query with NaN."""
import numpy as np
import pytest
import torch

from gpu_util import t

pytestmark = pytest.mark.gpu

N, D = 200, 64


def _index(lv, bits, metric, seed, entry):
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((N, D)).astype(np.float32)
    P = np.linalg.qr(rng.standard_normal((D, 24)))[0].T.astype(np.float32)
    Y = X @ P.T
    bad_p, bad_s = np.array([3, 50, 51, 199]), np.array([0, 51, 77])
    mu_p, mu_s = Y.mean(0), X.mean(0)
    Y[bad_p, 5] = np.inf
    X[bad_s, 7] = -np.inf
    adj = np.stack([rng.choice(N, 31, replace=False) for _ in range(N)])
    adj = np.concatenate([(np.arange(N)[:, None] + 1) % N, adj], 1).astype(np.int32)
    idx = lv.Index(0, metric=metric)
    idx.set_primary(t(Y), t(mu_p), bits, D).set_secondary(t(X), t(mu_s))
    if metric:  # a primary's squared norm is its original row's
        bad_p = np.union1d(bad_p, bad_s)
    idx.set_graph(t(adj), entry)
    Q = rng.standard_normal((20, D)).astype(np.float32)
    Q[4, 9] = np.nan
    Q[5] = np.nan
    return idx, t(Q), t(P), bad_p, bad_s


@pytest.mark.parametrize("bits,metric", [(8, 0), (8, 1), (4, 0), (4, 1)])
@pytest.mark.parametrize("L,k,entry,W", [(200, 200, 0, 1), (200, 20, 3, 2), (60, 60, 51, 2), (60, 10, 0, 1)])
@pytest.mark.parametrize("rerank", [False, True])
def test_scores_that_are_no_numbers(bits, metric, L, k, entry, W, rerank):
    import paper_2312_16335_gb300 as lv
    idx, Q, P, bad_p, bad_s = _index(lv, bits, metric, L + bits, entry)
    kw = dict(k=k, L=L, rerank=L if rerank else 0, width=W, max_hops=2 * N)
    ids, sc = idx.search(Q, P, **kw)
    shapes = [dict(queries_per_warp=1), dict(queries_per_warp=2), dict(visited_bits=16), dict(warps_per_block=4, hash_slots=512)]
    if W == 2:
        shapes.append(dict(warps_per_query=2))
    for s in shapes:
        a, b = idx.search(Q, P, **kw, **s)
        assert torch.equal(a, ids) and torch.equal(b, sc), s
    assert idx.sync_status() == 0
    ids, sc = ids.cpu().numpy(), sc.cpu().numpy()
    bad = set((bad_s if rerank else bad_p).tolist())
    assert not np.isnan(sc).any()
    for j in range(Q.shape[0]):
        n = (ids[j] >= 0).sum()
        assert len(set(ids[j][:n])) == n and (np.diff(sc[j][:n][np.isfinite(sc[j][:n])]) <= 0).all()
        isbad = np.array([j in (4, 5) or i in bad for i in ids[j][:n]])
        assert (np.isneginf(sc[j][:n]) == isbad).all()
        last = ids[j][:n][isbad]
        assert (np.diff(isbad.astype(int)) >= 0).all() and (np.diff(last) > 0).all()
        if L == N and k == N:
            assert set(last) == (set(range(N)) if j in (4, 5) else bad)
