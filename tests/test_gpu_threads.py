"""Four threads search four indexes of two very different sizes at the same time, each on its own stream.  They launch
the same kernels with different amounts of shared memory: every call succeeds and every answer is the one a
single thread gets."""
import threading

import pytest
import torch

from test_gpu_block_search import _setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [dict(), dict(queries_per_warp=1), dict(queries_per_warp=2)])
@pytest.mark.parametrize("bits,sbits,sizes", [(8, 8, ((1000, 512), (32, 32))), (4, 16, ((1000, 512), (32, 32))),
                                              (8, 16, ((1000, 512), (800, 224)))])
def test_threads_and_sizes(bits, sbits, sizes, kw):
    import paper_2312_16335_gb300 as lv
    jobs = []
    for D, L in sizes * 2:
        idx, Q, P = _setup(lv, 1500, D, 24, bits, 32, 0, 4, seed=D)
        if sbits == 16:
            adj, entry = idx.get_graph()
            X = torch.randn(1500, D, device="cuda", generator=torch.Generator(device="cuda").manual_seed(D))
            idx.encode(X, P, bits, 16).set_graph(adj, entry)
        args = dict(k=10, L=L, rerank=L, max_hops=8, **kw)
        jobs.append((idx, Q, P, args, idx.search(Q, P, **args)))
    torch.cuda.synchronize()
    errors, wrong, go = [], [], threading.Barrier(4)

    def work(idx, Q, P, args, want):
        out = tuple(torch.empty_like(x) for x in want)
        with torch.cuda.stream(torch.cuda.Stream()):
            go.wait()
            for _ in range(4000):
                try:
                    idx.search(Q, P, out=out, **args)
                except lv.LeanVecError as e:
                    errors.append(str(e))
            torch.cuda.current_stream().synchronize()
            wrong.append(not all(torch.equal(a, b) for a, b in zip(out, want)))

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for x in threads:
        x.start()
    for x in threads:
        x.join()
    assert not errors, (len(errors), errors[0])
    assert wrong == [False] * 4
