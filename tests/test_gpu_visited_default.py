"""The visited cache that a search picks by itself (16-bit tags for long walks over LVQ records) against
one of 32-bit ids: the same ids and scores on both sides of the rule's lines, and at the sizes where the
number of tags changes."""
import numpy as np
import pytest
import torch

from test_gpu_block_search import _setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,metric,R", [(8, 0, 64), (8, 1, 33), (4, 0, 128)])
@pytest.mark.parametrize("L", [113, 114, 128, 129, 156, 157, 256, 257, 320, 330, 352, 400, 512])
def test_default_cache_equals_ids(bits, metric, R, L):
    import paper_2312_16335_gb300 as lv
    idx, Q, P = _setup(lv, 6000, 96, 48, bits, R, metric, 80, seed=L + bits)
    for W, T, hops in ((1, 1, 0), (1, 1, 129), (2, 2, 0)):
        kw = dict(k=min(L, 100), L=L, rerank=L, max_hops=hops, width=W, warps_per_query=T)
        a = idx.search(Q, P, queries_per_warp=1, **kw)
        b = idx.search(Q, P, visited_bits=32, **kw)
        assert idx.sync_status() == 0
        assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
