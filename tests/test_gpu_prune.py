"""The prune kernel at its edges, through the graph build against the oracle, bit for bit: records of
16 and 17 code chunks (a thread or four lanes per record), pools of one member and of several words,
targets with more new sources than a small pool holds, lists of one and of the largest size."""
import numpy as np
import pytest

import oracle
import workloads
from gpu_util import t

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,bits,R,Lb,alpha,batch,rule", [
    (300, 256, 8, 16, 32, 1.0, 300, 0),    # 16 chunks: a thread per record
    (300, 272, 8, 16, 32, 1.0, 300, 0),    # 17 chunks: four lanes per record
    (260, 530, 4, 8, 20, 1.02, 100, 1),    # 17 chunks of LVQ-4
    (600, 12, 8, 6, 16, 1.0, 600, 0),    # one batch: hubs take more than R + 32 sources
    (500, 300, 8, 6, 16, 1.0, 500, 0),     # the same with long records
    (400, 20, 8, 1, 1, 1.0, 64, 0),        # single-member pools and lists
    (700, 20, 8, 128, 200, 0.9, 350, 0),   # R = 128, pools of up to 328
    (33, 40, 8, 31, 33, 1.3, 33, 1),       # everything within one word
])
def test_prune_edges(n, d, bits, R, Lb, alpha, batch, rule):
    import paper_2312_16335_gb300 as lv
    rng = np.random.default_rng(n + d)
    means = rng.standard_normal((5, d))
    Y = workloads.unit_rows(means[rng.integers(0, 5, n)] + 0.3 * rng.standard_normal((n, d)))
    mu = oracle.mean_fp32(Y)
    g_ref, e_ref = oracle.vamana_build(oracle.lvq_encode(Y, mu, bits), R=R, L_build=Lb, alpha=alpha, passes=2, batch=batch,
                                       seed=7, rule=rule)
    idx = lv.Index(0).set_primary(t(Y), t(mu), bits, d)
    idx.build_graph(R=R, L_build=Lb, alpha=alpha, passes=2, batch=batch, seed=7, rule=rule)
    idx.sync_status()
    g, e = idx.get_graph()
    assert e == e_ref
    np.testing.assert_array_equal(g.cpu().numpy(), g_ref)


def test_prune_rewritten_list_once():
    """A list that the launch for few sources made longer counts as one of few sources still: here a target
    of 12 neighbours or so gains a list which, with its sources again, is longer than a small pool, and
    which must not take back the sources that the pruning left out."""
    import paper_2312_16335_gb300 as lv
    n, d, R = 3000, 32, 48
    rng = np.random.default_rng(n + d)
    means = rng.standard_normal((3, d))
    Y = workloads.unit_rows(means[rng.integers(0, 3, n)] + rng.standard_normal((n, d)))
    mu = oracle.mean_fp32(Y)
    kw = dict(R=R, L_build=64, alpha=0.9, passes=2, batch=1500, seed=7, rule=0)
    g_ref, e_ref = oracle.vamana_build(oracle.lvq_encode(Y, mu, 8), **kw)
    idx = lv.Index(0).set_primary(t(Y), t(mu), 8, d)
    idx.build_graph(**kw)
    idx.sync_status()
    g, e = idx.get_graph()
    assert e == e_ref
    np.testing.assert_array_equal(g.cpu().numpy(), g_ref)
