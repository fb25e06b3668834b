"""Encoding at its edges: codes next to rounding halves and of rows that are not ordinary numbers, column
means at the edges of a chunk and of its unrolled loads, and an index that is encoded again and again."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import t, unpack_records

pytestmark = pytest.mark.gpu


def _rows(dim, levels, rng):
    rows = []
    for delta in (1.0, 0.25, 0.1, 3e-3, 7.7e6, 1e-30):  # codes within a few units in the last place of a half
        q = (rng.integers(0, levels, dim) + 0.5) * np.float64(delta)
        r = q.astype(np.float32)
        r = (r.view(np.int32) + rng.integers(-3, 4, dim, dtype=np.int32)).view(np.float32)
        r[0], r[-1] = 0.0, np.float32(delta) * np.float32(levels)
        rows += [r, -r, r + np.float32(delta)]
    rows += [np.full(dim, 0.125), np.arange(dim) * 1e-45, np.arange(dim) * 1e-41, rng.standard_normal(dim) * 1e-38,
             rng.uniform(-1.7e38, 1.7e38, dim), rng.uniform(-3.4e38, 3.4e38, dim)]
    return np.stack([np.asarray(r, np.float32) for r in rows])


@pytest.mark.parametrize("dim", [4, 60, 192, 196, 256, 260, 512, 516, 768, 772, 1024])
@pytest.mark.parametrize("bits", [4, 8])
def test_codes_near_halves(dim, bits):
    """Rows read in 16-byte pieces and rows that start on another boundary take different kernels: the same
    records, byte for byte, also with infinities and NaN in a row; the oracle's codes where all is finite."""
    import paper_2312_16335_gb300 as lv
    rng = np.random.default_rng(dim + bits)
    Y = _rows(dim, 2 ** bits - 1, rng)
    odd = np.repeat(rng.standard_normal((1, dim)).astype(np.float32), 5, 0)
    odd[0, 1], odd[1, 2], odd[2, 0], odd[3, :2], odd[4, 3] = np.inf, -np.inf, np.nan, (np.inf, -np.inf), 3e38
    for mean in (np.zeros(dim, np.float32), rng.standard_normal(dim).astype(np.float32)):
        Z = np.concatenate([Y, odd])
        buf = torch.zeros(Z.size + 1, device="cuda")
        buf[1:] = t(Z).reshape(-1)
        a = lv.leanvec_lvq_encode(t(Z), t(mean), bits)
        b = lv.leanvec_lvq_encode(buf[1:].view(Z.shape), t(mean), bits)
        assert torch.equal(a, b)
        fin = np.arange(len(Y) - 1)  # the last row's range is above the largest float32
        codes, delta, lower, *_ = unpack_records(a.cpu().numpy()[fin], dim, bits)
        ref = oracle.lvq_encode(Y[fin], mean, bits)
        np.testing.assert_array_equal(delta, ref.delta)
        np.testing.assert_array_equal(lower, ref.lower)
        np.testing.assert_array_equal(codes, ref.codes)


@pytest.mark.parametrize("n,dim", [(n, d) for n in (1, 7, 9, 57, 64, 65, 121, 129, 2047, 2048, 2049, 4096 + 61)
                                   for d in (4, 33, 132)] + [(57 * 2048 + 1, 8), (56 * 2048, 5), (113 * 2048 - 1, 516),
                                                             (153 * 2048 + 127, 132), (2048, 39000)])
def test_column_mean_edges(n, dim):
    """Rounding to float32 (2^-24, doubled) and the compensated float32 sums of at most 256 rows
    (256 x 2^-24 x 2^-24 x 256 = 2^-32 of the mean magnitude)."""
    import paper_2312_16335_gb300 as lv
    X = np.random.default_rng(n + dim).standard_normal((n, dim)).astype(np.float32)
    X[:, 0] += 100.0
    got = lv.leanvec_column_mean(t(X)).cpu().numpy()
    X = X.astype(np.float64)
    assert (np.abs(got - X.mean(0)) <= 2.0 ** -23 * np.abs(X.mean(0)) + 2.0 ** -32 * np.abs(X).mean(0)).all()


def test_encode_again():
    """An index that is encoded again holds what a new one does: the same and other sizes, encodings of
    either store, and stores set one by one in between."""
    import paper_2312_16335_gb300 as lv
    rng = np.random.default_rng(0)
    for metric in (0, 1):
        idx = lv.Index(0, metric=metric)
        for n, D, d, pb, sb in [(500, 64, 16, 8, 8), (500, 64, 16, 8, 8), (500, 64, 16, 4, 8), (500, 64, 16, 8, 16),
                                (300, 64, 16, 8, 8), (700, 64, 16, 8, 8), (700, 96, 40, 8, 8), (500, 64, 16, 8, 8)]:
            X, B = t(rng.standard_normal((n, D)).astype(np.float32)), t(rng.standard_normal((d, D)).astype(np.float32))
            new = lv.Index(0, metric=metric).encode(X, B, pb, sb)
            adj = t(rng.integers(0, n, (n, 16)).astype(np.int32))
            for again in range(2):
                idx.encode(X, B, pb, sb).set_graph(adj, 1)
                new.set_graph(adj, 1)
                assert torch.equal(idx.primary_records(), new.primary_records())
                assert torch.equal(idx.secondary_records(), new.secondary_records())
                assert torch.equal(idx.primary_mean(), new.primary_mean())
                a, b = (i.search(X[:50].contiguous(), B, k=5, L=20, rerank=20) for i in (idx, new))
                assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
                Y = t(rng.standard_normal((n, d)).astype(np.float32))
                for i in (idx, new):
                    i.set_primary(Y, None, pb, D)
                assert torch.equal(idx.primary_records(), new.primary_records())
                new = lv.Index(0, metric=metric).encode(X, B, pb, sb)
