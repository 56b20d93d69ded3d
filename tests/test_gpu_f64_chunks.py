"""FP64 sweep at the edges of its chunks: rows left over in the last chunk of a CTA, odd row
lengths, and row lengths that leave room for three chunks of four, two or one rows or for a
single chunk (iteration-locked against the FP64 oracle, at the bars of test_gpu_f64.py).
"""
import numpy as np
import pytest

from test_gpu_f64 import check, fit64, gp  # noqa: F401  (gp is the fixture)

pytestmark = pytest.mark.gpu

SHAPES = [(761, 1, 1), (761, 2, 2), (1367, 33, 4), (1216, 255, 5), (1825, 129, 34), (1217, 2055, 3), (761, 3601, 3),
          (460, 5801, 2), (308, 8191, 2)]


@pytest.mark.parametrize("algo", ["gs", "nipals"])
@pytest.mark.parametrize("shape", SHAPES, ids=[f"{m}x{n}k{k}" for m, n, k in SHAPES])
def test_chunk_edges(gp, algo, shape):  # noqa: F811
    M, N, K = shape
    g = np.random.default_rng(M * 100003 + N)
    if N < 8:
        X = g.standard_normal((M, N))
    else:  # K well-separated directions and noise
        L, R = np.linalg.qr(g.standard_normal((M, K)))[0], np.linalg.qr(g.standard_normal((N, K)))[0]
        X = (L * (5.0 * 0.9 ** np.arange(K))) @ R.T + 1e-4 * g.standard_normal((M, N))
    out = fit64(gp, X, K, algo, tol=1e-9, max_iter=200)
    assert out["status"] == 0
    check(out, X, K, algo, tol=1e-9, max_iter=200)
