"""Reverse edges pruned by one launch (pools of up to 40 KB) and by two, on both sides of that line, against the
oracle bit for bit: lists that gain more than 32 sources, lists that a first launch rewrites, LVQ-4."""
import numpy as np
import pytest

import oracle
import workloads
from gpu_util import t

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,bits,R,Lb,alpha,batch,rule", [
    (2500, 32, 8, 48, 64, 0.9, 1250, 0),   # 448 slots of 48 bytes: 27 KB, one launch
    (2500, 64, 8, 48, 64, 0.9, 1250, 0),   # of 80 bytes: 41 KB, two
    (2500, 96, 8, 48, 64, 0.9, 1250, 0),   # of 112 bytes: 55 KB, two
    (1500, 60, 8, 32, 64, 1.02, 1500, 1),  # 384 slots of 80 bytes: 35 KB, one
    (1500, 90, 8, 32, 64, 1.02, 1500, 1),  # of 112 bytes: 47 KB, two
    (900, 100, 4, 16, 32, 1.0, 900, 0),    # 320 slots of 80 bytes, one
])
def test_prune_launches(n, d, bits, R, Lb, alpha, batch, rule):
    import paper_2312_16335_gb300 as lv
    rng = np.random.default_rng(n + d)
    means = rng.standard_normal((3, d))
    Y = workloads.unit_rows(means[rng.integers(0, 3, n)] + rng.standard_normal((n, d)))
    mu = oracle.mean_fp32(Y)
    kw = dict(R=R, L_build=Lb, alpha=alpha, passes=2, batch=batch, seed=7, rule=rule)
    g_ref, e_ref = oracle.vamana_build(oracle.lvq_encode(Y, mu, bits), **kw)
    idx = lv.Index(0).set_primary(t(Y), t(mu), bits, d)
    idx.build_graph(**kw)
    idx.sync_status()
    g, e = idx.get_graph()
    assert e == e_ref
    np.testing.assert_array_equal(g.cpu().numpy(), g_ref)
