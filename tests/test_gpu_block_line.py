"""Both sides of the line between a block per query and a warp per query (six queries per SM): the same ids and
scores as a warp per query."""
import pytest
import torch

from test_gpu_block_search import _setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,metric,L,W", [(8, 0, 128, 2), (4, 0, 512, 2), (8, 1, 512, 1), (4, 1, 40, 1)])
def test_block_line(bits, metric, L, W):
    import paper_2312_16335_gb300 as lv
    line = 6 * torch.cuda.get_device_properties(0).multi_processor_count
    idx, Q, P = _setup(lv, 4000, 96, 48, bits, 64, metric, line + 1, seed=L + bits)
    for m in (line - 1, line, line + 1):
        kw = dict(k=10, L=L, rerank=L, width=W)
        a = idx.search(Q[:m].contiguous(), P, **kw)
        b = idx.search(Q[:m].contiguous(), P, queries_per_warp=1, **kw)
        assert idx.sync_status() == 0
        assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
