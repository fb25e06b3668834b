"""The rerank's bounded wait: a query whose record copies are given up on has no answer at all (-1, -infinity)
and the status says so, however many of the block's warps it concerns; else the answers are the FP64 ranking's.

Records are LVQ-8 with delta 2^-8, lower 0, a zero mean and integer queries of entries up to 4.  Tolerance: a
query entry's fixed point is off by 2^-22 at most (half of 4 / 8388607), which 255 2^-8 multiplies D times; and
twelve float32 roundings of sums below S = 4 255 2^-8 D, 2^-24 S each.
"""
import ctypes

import numpy as np
import pytest
import torch

import kernel_unit
from gpu_util import t

pytestmark = pytest.mark.gpu

TIMEOUT = 4  # ST_TIMEOUT


def _run(lib, rec, stride, chunks, Q, cand, cand_n, k, tries):
    m, D = Q.shape
    ids = torch.full((m, k), -7, dtype=torch.int32, device="cuda")
    sc = torch.full((m, k), float("nan"), device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    mean = torch.zeros(D, device="cuda")
    p = lambda a: ctypes.c_void_p(a.data_ptr())
    rc = lib.rerank_unit(p(rec), ctypes.c_int64(stride), chunks, 8, 0, p(Q), ctypes.c_int64(m), D, p(mean), p(cand),
                         p(cand_n), cand.shape[1], k, p(ids), p(sc), k, p(status), tries,
                         ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0
    torch.cuda.synchronize()
    return ids.cpu().numpy(), sc.cpu().numpy(), int(status.item())


@pytest.mark.parametrize("nr,k", [(512, 10), (509, 100), (37, 37), (5, 3), (1, 1)])
def test_no_time_to_wait(nr, k):
    lib = kernel_unit.load("rerank_unit")
    n, D, m = 20000, 784, 300
    chunks, stride = D // 16, 800
    rng = np.random.default_rng(nr)
    codes = rng.integers(0, 256, (n, D), dtype=np.uint8)
    rec = np.zeros((n, stride), np.uint8)
    rec[:, :D] = codes
    rec[:, D:D + 4] = np.frombuffer(np.float32(2.0 ** -8).tobytes(), np.uint8)
    Q = rng.integers(-4, 5, (m, D)).astype(np.float32)
    Q[:, 0] = 4
    cand = np.stack([rng.choice(n, nr, replace=False) for _ in range(m)]).astype(np.int32)
    cand_n = np.full(m, nr, np.int32)
    cand_n[7] = 0   # no candidate to wait for
    cand_n[9] = -1  # a query that is not for the rerank
    args = (lib, t(rec), stride, chunks, t(Q), t(cand), t(cand_n), k)
    ids, sc, status = _run(*args, 1000)
    assert status == 0
    tol = 255 * D * 2.0 ** -8 * (2.0 ** -22 + 12 * 4 * 2.0 ** -24)
    for j in range(0, m, 25):
        exact = codes[cand[j]].astype(np.float64) @ Q[j].astype(np.float64) / 256
        pos = {int(c): i for i, c in enumerate(cand[j])}
        got = np.array([exact[pos[int(g)]] for g in ids[j]])
        assert len(set(ids[j].tolist())) == k and np.abs(sc[j] - got).max() <= tol
        assert np.sort(exact)[::-1][k - 1] <= got.min() + 2 * tol
    assert (ids[7] == -1).all() and (ids[9] == -7).all()
    ids, sc, status = _run(*args, 0)
    assert status == TIMEOUT
    others = np.arange(m) != 9
    assert (ids[others] == -1).all() and np.isneginf(sc[others]).all() and (ids[9] == -7).all()
