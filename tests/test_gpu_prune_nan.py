"""Graph build over a store with records whose pair scores are no numbers (rows with an infinite entry): such a
member ranks last in a pruning pool, wherever it came from.  With an alpha under which nothing covers
anything, every node whose pool holds R ordinary members therefore keeps none of the others."""
import numpy as np
import pytest

from gpu_util import t

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,bits", [(32, 8), (40, 4), (300, 8)])
@pytest.mark.parametrize("metric,alpha", [(0, 1e-6), (1, 1e6)])
@pytest.mark.parametrize("batch", [700, 128])
def test_scores_that_are_no_numbers_rank_last(d, bits, metric, alpha, batch):
    import paper_2312_16335_gb300 as lv
    n, R = 700, 8
    rng = np.random.default_rng(d + batch)
    X = rng.standard_normal((n, d)).astype(np.float32)
    X /= np.linalg.norm(X, axis=1, keepdims=True)
    mean = X.mean(0)
    bad = rng.choice(n, 60, replace=False)
    X[bad, rng.integers(0, d, 60)] = np.inf
    idx = lv.Index(0, metric=metric).set_primary(t(X), t(mean), bits, d)
    idx.build_graph(R=R, L_build=64, alpha=alpha, passes=2, batch=batch, rule=0)
    adj, _ = idx.get_graph()
    assert idx.sync_status() == 0
    adj = adj.cpu().numpy()
    assert ((adj >= -1) & (adj < n)).all()
    for v in range(n):
        row = adj[v][adj[v] >= 0]
        assert v not in row and len(set(row.tolist())) == len(row)
    good = np.setdiff1d(np.arange(n), bad)
    assert not np.isin(adj[good], bad).any()
