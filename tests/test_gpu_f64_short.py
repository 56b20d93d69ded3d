"""FP64 sweep for short rows (at most 256 doubles, 32 rows a chunk), at the edges of its warps'
four rows, its chunks, its ring of three and its shares of the column sums (iteration-locked
against the FP64 oracle, at the bars of test_gpu_f64.py).
"""
import numpy as np
import pytest

from test_gpu_f64 import check, fit64, gp  # noqa: F401  (gp is the fixture)

pytestmark = pytest.mark.gpu

# (rows, columns, K, CTAs): rows per CTA 1 to 4, 5, 31 to 33, 64 to 65, 96 to 97, 129, and some 300 with two CTAs
SHAPES = [(2, 1, 1, 0), (300, 2, 2, 0), (610, 3, 2, 0), (761, 31, 7, 0), (4711, 33, 5, 0), (4865, 4, 3, 0),
          (5017, 63, 6, 0), (9729, 64, 9, 0), (9881, 65, 4, 0), (14593, 34, 33, 0), (14745, 129, 5, 0),
          (19609, 8, 3, 0), (601, 255, 11, 2), (97, 256, 12, 1), (700, 257, 4, 2), (1216, 200, 60, 8)]


@pytest.mark.parametrize("algo", ["gs", "nipals"])
@pytest.mark.parametrize("shape", SHAPES, ids=[f"{m}x{n}k{k}g{c}" for m, n, k, c in SHAPES])
def test_short_rows(gp, algo, shape):  # noqa: F811
    M, N, K, ctas = shape
    g = np.random.default_rng(M * 100003 + N)
    if N < 8:
        X = g.standard_normal((M, N))
    else:  # K well-separated directions and noise
        L, Z = np.linalg.qr(g.standard_normal((M, K)))[0], np.linalg.qr(g.standard_normal((N, K)))[0]
        X = (L * (5.0 * 0.9 ** np.arange(K))) @ Z.T + 1e-4 * g.standard_normal((M, N))
    out = fit64(gp, X, K, algo, tol=1e-9, max_iter=200, grid_ctas=ctas)
    assert out["status"] in ((0, 4) if N < 8 else (0,))  # random columns: close singular values
    check(out, X, K, algo, tol=1e-9, max_iter=200)


def test_zero_start_column_of_short_rows(gp):  # noqa: F811
    """A zero column behind the first component: the sweep is repeated with the column of largest norm."""
    g = np.random.default_rng(5)
    X = g.standard_normal((5000, 12)) * 0.8 ** np.arange(12)
    X[:, 1] = 0.0
    out = fit64(gp, X, 3, "gs", tol=1e-9, max_iter=500)
    check(out, X, 3, "gs", tol=1e-9, max_iter=500)
    X[:, 0] = 0.0
    out = fit64(gp, X, 3, "gs", tol=1e-9, max_iter=500)
    check(out, X, 3, "gs", tol=1e-9, max_iter=500)
