"""The polar factor of the Frank-Wolfe step on ill-conditioned matrices, against a host FP64 SVD.

One iteration from zero gives A = the leading eigenvectors of K_X and B = the polar factor of A K_Q K_X.
With K_X diagonal and K_Q of integers that matrix is exact in float32 (A is a permutation, every entry one
product of an integer below 2^13 and a number of 7 bits times a power of two), so only the factor's own
arithmetic counts: (C C^T)^(-1/2) C through the FP64 eigenvalues of C C^T, whose relative error at the
smallest one is D 2^-53 kappa^2 (product and decomposition), hence D 2^-52 kappa^2 for the factor, and 2^-24 for
its float32 entries, which are at most 1.  Rows of B B^T - I add up sqrt(D) times that twice."""
import numpy as np
import pytest

from gpu_util import t

pytestmark = pytest.mark.gpu


def _diagonal_rows(ex, mult):
    """Rows whose second moment is diag(2^ex mult) exactly: entry j from copies of one-hot rows."""
    rows = []
    for j, (e, m) in enumerate(zip(ex, mult)):
        k, c = int(e) - 6, int(round(64 * m))
        rows += [(j, 2.0 ** (k // 2))] * (c if k % 2 == 0 else 2 * c)
    X = np.zeros((len(rows), len(ex)), np.float32)
    for i, (j, v) in enumerate(rows):
        X[i, j] = v
    return X


@pytest.mark.parametrize("D", [16, 24, 64])
@pytest.mark.parametrize("span", [0, 5, 10, 14, 17])
def test_polar_factor_of_ill_conditioned_matrices(D, span):
    import paper_2312_16335_gb300 as lv
    rng = np.random.default_rng(span + D)
    X = _diagonal_rows(np.round(np.linspace(0, -span, D)), 1 + np.arange(D)[::-1] / 64.0)
    Q = rng.integers(-2, 3, (40 * D, D)).astype(np.float32)
    A, B, _ = lv.leanvec_fit_ood(t(X), t(Q), D, method=lv.FIT_FW, max_iter=1)
    A, B = A.cpu().numpy().astype(np.float64), B.cpu().numpy().astype(np.float64)
    KX, KQ = X.astype(np.float64).T @ X, Q.astype(np.float64).T @ Q
    assert np.abs(KQ).max() < 2 ** 13
    assert np.array_equal(A, np.eye(D)[np.argsort(-np.diag(KX), kind="stable")])
    u, s, vt = np.linalg.svd(A @ KQ @ KX)
    kappa = s[0] / s[-1]
    assert kappa < 3e5  # below the cut at 1e-12 of the largest eigenvalue of C C^T
    tol = D * 2.0 ** -52 * kappa ** 2 + 2.0 ** -24
    assert np.abs(B - u @ vt).max() <= tol
    assert np.abs(B @ B.T - np.eye(D)).max() <= 2 * np.sqrt(D) * tol
