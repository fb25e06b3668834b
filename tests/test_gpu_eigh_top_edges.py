"""The leading eigenpairs at the sizes where the reduction's storage changes (rows in shared memory and
their slots per thread, then global memory), for spread, repeated and scaled spectra.  Tolerances: those
of a backward-stable FP64 solver, 1e-11 of ||K|| for eigenvalues, residual and orthonormality."""
import numpy as np
import pytest

from gpu_util import t

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [8, 9, 31, 33, 127, 128, 129, 130, 255, 257, 385, 511, 513, 640, 769, 1023, 1025, 1300,
                               1900])
@pytest.mark.parametrize("kind", ["random", "decay", "repeated", "tiny"])
def test_eigh_top_edges(D, kind):
    import paper_2312_16335_gb300 as lv
    if D > 1100 and kind != "decay":
        pytest.skip("one spectrum for the largest sizes")
    rng = np.random.default_rng(D)
    w = {"random": rng.standard_normal(D), "decay": 1.0 / np.arange(1, D + 1),
         "repeated": np.repeat([3.0, 1.0, -2.0], D)[rng.permutation(3 * D)[:D]], "tiny": 1e-100 * (1 + rng.random(D))}[kind]
    Q = np.linalg.qr(rng.standard_normal((D, D)))[0]
    K = (Q * w) @ Q.T
    K = (K + K.T) / 2
    nout = min(D, 24)
    ev, V = (x.cpu().numpy() for x in lv.leanvec_eigh_top(t(K), nout))
    scale = np.abs(w).max()
    assert np.abs(ev - np.sort(w)[::-1][:nout]).max() <= 1e-11 * scale
    assert np.abs(V @ V.T - np.eye(nout)).max() <= 1e-11
    assert np.abs(K @ V.T - V.T * ev).max() <= 1e-11 * scale
