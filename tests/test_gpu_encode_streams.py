"""Filling an index that holds no store waits for its own stream only; writing a held store again waits for
the work of every stream, which may be searching it."""
import numpy as np
import pytest
import torch

from gpu_util import t

pytestmark = pytest.mark.gpu

CYCLES = 600_000_000  # about 0.3 s on the other stream


def _fill(idx, how, X, P, Y):
    if how == "encode":
        idx.encode(X, P, 8, 8)
    elif how == "encode_fp16":
        idx.encode(X, P, 4, 16)
    else:
        idx.set_primary(Y, None, 8, X.shape[1])
        idx.set_secondary(X)


@pytest.mark.parametrize("metric", [0, 1])
@pytest.mark.parametrize("how", ["encode", "encode_fp16", "set"])
def test_new_stores_do_not_wait_for_other_streams(how, metric):
    import paper_2312_16335_gb300 as lv
    rng = np.random.default_rng(3)
    X = t(rng.standard_normal((3000, 96)).astype(np.float32))
    P = t(np.linalg.qr(rng.standard_normal((96, 32)))[0].T.astype(np.float32))
    Y = X @ P.T
    first = lv.Index(0, metric=metric)
    _fill(first, how, X, P, Y)  # loads the kernels and sizes the scratch pool
    new = lv.Index(0, metric=metric)
    mine, other, done = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.Event()
    torch.cuda.synchronize()
    with torch.cuda.stream(other):
        torch.cuda._sleep(CYCLES)
        done.record()
    with torch.cuda.stream(mine):
        _fill(new, how, X, P, Y)
    assert not done.query()
    with torch.cuda.stream(mine):
        _fill(first, how, X, P, Y)  # its stores are held
    assert done.query()
    assert torch.equal(new.primary_records()[:, :32], first.primary_records()[:, :32])
    assert torch.equal(new.primary_mean(), first.primary_mean())
