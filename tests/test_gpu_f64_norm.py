"""FP64 fit, ||v' - V b'||: the two ways it is formed (the difference ||v'||^2 - b'^T b', or the
rows with a third reduction), where each must be taken.

V diag(sigma) is built from v' - V b' and its norm, so with svd_form the columns of T have unit
norm whatever V looks like: their squares are 150 terms of relative rounding 2^-53 and the norm
another sum of the same kind, some 300 x 2^-53 = 3e-14 in the worst case, so 1e-12 is the bar.
"""
import numpy as np
import pytest

import oracle
from test_gpu_f64 import ANG, SIG, dist, fit64, gp  # noqa: F401  (gp is the fixture)

pytestmark = pytest.mark.gpu


def share(X, lock):
    """b'^T b' / ||v'||^2 of every iteration of every component, and the loss of V's orthonormality."""
    K = len(lock)
    R, V, U = X.copy(), np.zeros((X.shape[0], K)), np.zeros((X.shape[1], K))
    out = []
    for k in range(K):
        v = R[:, k]
        out.append([])
        for _ in range(lock[k]):
            u = R.T @ v
            u = u - U[:, :k] @ (U[:, :k].T @ u)
            u /= np.linalg.norm(u)
            v = R @ u
            b = V[:, :k].T @ v
            out[-1].append(float(b @ b / (v @ v)))
            v = v - V[:, :k] @ b
            lam = np.linalg.norm(v)
            v = v / lam
        V[:, k], U[:, k] = v, u
        R = R - lam * np.outer(v, u)
    return out, float(np.abs(V.T @ V - np.eye(K)).max())


@pytest.mark.parametrize("decades,n1,it,seed", [(6, 130, 10, 0), (6, 130, 10, 4), (8, 120, 20, 2)])
def test_norm_where_score_directions_are_dependent(gp, decades, n1, it, seed):  # noqa: F811
    """n1 components of one iteration each on a graded matrix, then twelve of more: V is no longer
    orthonormal (1e-9 and more off), so ||v'||^2 - b'^T b' is not ||v' - V b'||^2."""
    X = np.triu(np.random.default_rng(seed).standard_normal((150, 150))) * 10.0 ** np.linspace(-decades, 0, 150)
    lock = [1] * n1 + [it] * 12
    g = fit64(gp, X, len(lock), "gs", iters_lock=lock, svd_form=1)
    found = g["info"]["found"]
    assert found > n1
    V = g["T"][:, :found]
    G = V.T @ V
    assert np.abs(G - np.diag(np.diag(G))).max() > 1e-10  # what the case is about
    np.testing.assert_allclose(np.linalg.norm(V, axis=0), 1.0, rtol=0, atol=1e-12)


def test_norm_of_unconverged_components(gp):  # noqa: F811
    """Components of few iterations leave b' large: the rows are summed, at a component's last
    iteration and before it, with V orthonormal; the oracle's bars of test_gpu_f64.py hold."""
    g0 = np.random.default_rng(1)
    L, Z = np.linalg.qr(g0.standard_normal((400, 150)))[0], np.linalg.qr(g0.standard_normal((150, 150)))[0]
    X = (L * (100 * 0.85 ** np.arange(150))) @ Z.T
    lock = [1] * 10 + [4, 1, 3, 1, 5, 2, 6, 1, 2, 3]
    sh, loss = share(X, lock)
    assert loss < 1e-13
    assert any(s[-1] > 0.3 for s in sh) and any(max(s[:-1], default=0) > 0.3 for s in sh)
    g = fit64(gp, X, len(lock), "gs", iters_lock=lock, svd_form=1)
    ref = oracle.fit(X, len(lock), tol=1e-10, max_iter=2000, algo="gs", iters_lock=lock)
    assert g["info"]["found"] == ref.found == len(lock)
    np.testing.assert_allclose(g["lam"], ref.lam, rtol=SIG)
    for k in range(len(lock)):
        assert dist(g["T"][:, k], ref.T[:, k]) <= ANG, k
        assert dist(g["P"][:, k], ref.P[:, k]) <= ANG, k
