"""The initial random graph at its edges, through a one-pass build in one batch against the oracle: rows
that hold every other node, rows of less than, exactly and more than 32 draws, the largest degree."""
import numpy as np
import pytest

import oracle
import workloads
from gpu_util import t

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 9, 32, 33, 65, 129, 130, 250])
@pytest.mark.parametrize("R", [1, 31, 32, 33, 64, 128])
def test_initial_graph(n, R):
    import paper_2312_16335_gb300 as lv
    rng = np.random.default_rng(n + R)
    Y = workloads.unit_rows(rng.standard_normal((n, 16)))
    mu = oracle.mean_fp32(Y)
    g_ref, e_ref = oracle.vamana_build(oracle.lvq_encode(Y, mu, 8), R=R, L_build=R, alpha=1.0, passes=1, batch=n, seed=n)
    idx = lv.Index(0).set_primary(t(Y), t(mu), 8, 16)
    idx.build_graph(R=R, L_build=R, alpha=1.0, passes=1, batch=n, seed=n)
    idx.sync_status()
    g, e = idx.get_graph()
    assert e == e_ref
    np.testing.assert_array_equal(g.cpu().numpy(), g_ref)
