"""Block fit: the order of its iterations (locked, capped, stopped by the tolerance, dependent
columns found late) and its inputs (centring, both layouts).

Parity with the FP64 oracle at the bars of test_gpu_block.py.
"""
import numpy as np
import pytest

import oracle
import synth
from parity_helpers import angle, clusters, sigma_ok, subspace_angle
from test_gpu_block import gp  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu


def run(gp, X32, K, b, layout="row", **kw):  # noqa: F811
    import torch

    M, N = X32.shape
    Xd = torch.from_numpy(np.ascontiguousarray(X32)).cuda()
    if layout == "col":
        Xd = Xd.t().contiguous().t()
    with gp.Handle(M, N, K) as h:
        r = h.fit_block(Xd, K, block=b, want_R=True, **kw)
        torch.cuda.synchronize()
        return dict(T=r.T.cpu().numpy().astype(np.float64), P=r.P.cpu().numpy().astype(np.float64),
                    lam=r.lam.cpu().numpy(), iters=r.iters.cpu().numpy(), R=r.R.cpu().numpy().astype(np.float64),
                    status=r.status, info=r.info)


def check(g, X32, K, b, lock):
    ref = oracle.block_fit(X32.astype(np.float64), K, b, tol=1e-6, max_iter=1000, iters_lock=lock)
    assert g["info"]["found"] == ref.found == K and list(g["iters"]) == list(lock)
    assert sigma_ok(g["lam"], ref.lam).all(), (g["lam"], ref.lam)
    for grp in clusters(ref.lam, 1e-3, floor=1e-2):
        if len(grp) == 1:
            assert angle(g["P"][:, grp[0]], ref.P[:, grp[0]]) <= 1e-3, grp
            assert angle(g["T"][:, grp[0]], ref.T[:, grp[0]]) <= 1e-3, grp
        else:
            assert subspace_angle(g["P"][:, grp], ref.P[:, grp]) <= 1e-3, grp
    assert np.abs(g["P"].T @ g["P"] - np.eye(K)).max() <= 1e-5
    assert np.linalg.norm(g["R"] - ref.R) <= 1e-5 * np.linalg.norm(X32.astype(np.float64))


def planted():
    return synth.planted(500, 200, 10.0, 0.85, 0.01, 44).X.astype(np.float32)


@pytest.mark.parametrize("its", [(1, 1, 1), (1, 2, 3), (3, 1, 2), (2, 5, 1)])
def test_locked_blocks(gp, its):  # noqa: F811
    X = planted()
    lock = [its[k // 4] for k in range(10)]
    g = run(gp, X, 10, 4, iters_lock=lock, tol=10.0, max_iter=1)  # the lock decides, not these
    assert g["status"] == 0
    check(g, X, 10, 4, lock)


@pytest.mark.parametrize("n", [1, 2, 3])
def test_capped_blocks(gp, n):  # noqa: F811
    X = planted()
    g = run(gp, X, 10, 4, tol=1e-12, max_iter=n)
    assert g["status"] == 4
    check(g, X, 10, 4, [n] * 10)


@pytest.mark.parametrize("tol", [10.0, 0.2, 0.05, 1e-2, 1e-3])
def test_loose_tolerances(gp, tol):  # noqa: F811
    """Stops after one to a few iterations, whether the next half step waited for the test or not;
    the counts are the oracle's own, within one for rounding of the Ritz values."""
    X = planted()
    g = run(gp, X, 10, 4, tol=tol, max_iter=100)
    assert g["status"] == 0
    free = oracle.block_fit(X.astype(np.float64), 10, 4, tol=tol, max_iter=100)
    assert np.abs(g["iters"] - free.iters).max() <= (0 if tol > 1 else 1), (g["iters"], free.iters)
    check(g, X, 10, 4, g["iters"])


@pytest.mark.parametrize("layout", ["row", "col"])
@pytest.mark.parametrize("center", [0, 1, 2])
def test_centring_and_layouts(gp, center, layout):  # noqa: F811
    X = planted() + np.float32(3.0)
    g = run(gp, X, 6, 3, layout=layout, center=center, tol=1e-6, max_iter=500)
    X64 = X.astype(np.float64)
    Xc = X64 - X64.mean(axis=center - 1, keepdims=True) if center else X64
    assert g["status"] == 0
    check(g, Xc.astype(np.float32), 6, 3, g["iters"])


def late(eps):
    """Rank 3, sigma (1, a, a) with a = 2^-23: two start columns that contain the large direction
    only eps-fold, so the iterate's columns become dependent (singular values 1 and a) a few steps on."""
    a = np.float32(2.0**-23)
    X = np.zeros((40, 6), dtype=np.float32)
    X[0, 5] = 1.0
    X[1, 0], X[2, 1] = a, a
    X[0, 0], X[0, 1] = np.float32(eps) * a * a, np.float32(0.5 * eps) * a * a
    return X


def dependent_by(X, b, cap):
    """Iterations of the first block before its columns are dependent (a pivot of a Gram matrix at most 1e-12
    of its largest diagonal entry), at most cap; None if they are not by then."""
    R = X.astype(np.float64)

    def qr(A):
        for _ in range(2):
            G = A.T @ A
            S = np.linalg.cholesky(G + 1e-30 * G.max() * np.eye(b)).T
            if not (np.diag(S) ** 2 > 1e-12 * np.diag(G).max()).all():
                return None
            A = A @ np.linalg.inv(S)
        return A

    U = qr(R.T @ R[:, :b])
    for j in range(cap):
        V = None if U is None else qr(R @ U)
        if V is None:
            return j
        U = qr(R.T @ V)
    return None


@pytest.mark.parametrize("eps,after", [(1e-3, 1), (1e-6, 1), (1e-12, 1), (1e-20, 2)])
def test_columns_found_dependent_after_some_iterations(gp, eps, after):  # noqa: F811
    X = late(eps)
    assert dependent_by(X, 2, 5) == after
    for cap in (1, 2, 3, 4):
        g = run(gp, X, 2, 2, tol=1e-6, max_iter=cap)
        if cap <= after:  # the block ended before
            assert (g["status"], g["info"]["found"]) == (4, 2), cap
            assert list(g["iters"]) == [cap] * 2 and g["lam"][0] > 0
        else:
            assert (g["status"], g["info"]["found"]) == (5, 0), cap
            for key in ("T", "P", "lam", "iters"):
                assert not g[key].any(), (cap, key)
            assert np.array_equal(g["R"], X.astype(np.float64))
        lock = run(gp, X, 2, 2, iters_lock=[cap] * 2)
        assert lock["status"] == (0 if cap <= after else 5), cap
