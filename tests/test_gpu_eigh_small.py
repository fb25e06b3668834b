"""The one-launch Jacobi eigen-decomposition (matrices of up to 256 rows) and the path above it at the
edges of their ranges: odd sizes, both thread layouts, repeated and widely spread eigenvalues, scales
far outside float32.  Tolerances: the bounds of a backward-stable FP64 solver, 1e-11 of ||K|| for the
residual and the eigenvalues and 1e-11 for orthonormality."""
import numpy as np
import pytest

from gpu_util import t

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [2, 3, 5, 16, 33, 127, 128, 129, 130, 255, 256, 258])
@pytest.mark.parametrize("kind", ["random", "spread", "repeated", "tiny", "huge"])
def test_eigh_edges(D, kind):
    import paper_2312_16335_gb300 as lv
    rng = np.random.default_rng(D)
    Q = np.linalg.qr(rng.standard_normal((D, D)))[0]
    w = {"random": rng.standard_normal(D), "spread": 10.0 ** np.linspace(0, -14, D),
         "repeated": np.repeat([3.0, 1.0, -2.0], D)[rng.permutation(3 * D)[:D]],
         "tiny": 1e-120 * (1 + rng.random(D)), "huge": 1e150 * rng.standard_normal(D)}[kind]
    K = (Q * w) @ Q.T
    K = (K + K.T) / 2
    ev, V = (x.cpu().numpy() for x in lv.leanvec_eigh(t(K)))
    scale = np.abs(w).max()
    assert (np.diff(ev) <= 0).all()
    assert np.abs(ev - np.sort(w)[::-1]).max() <= 1e-11 * scale
    assert np.abs(V @ V.T - np.eye(D)).max() <= 1e-11
    assert np.abs(K @ V.T - V.T * ev).max() <= 1e-11 * scale
    j = np.abs(V).argmax(1)
    assert (V[np.arange(D), j] > 0).all()
