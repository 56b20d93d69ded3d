"""Column means of the centring step, at the edges of the chunks and blocks its kernels take.

With `want_R` the fit returns X - mean = R + t p^T (K = 1), so R + T P^T is compared with
the FP64 centred matrix.  Bar: the centred value is rounded to FP32 once, t and p once each,
and the deflation's fma and the scale of t once more; each is at most 2^-24 of |x - mean| or
|t p|, six in all, so 8 x 2^-24 x (max |x - mean| + max |t p|).  A mean off by one row's
share at a chunk edge (an offset of 100 / M and more) is thousands of times that.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gp():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("CUDA device required")
    import paper_0811_1081_gb300 as m

    m.load()
    return m


@pytest.mark.parametrize("layout", ["row", "col"])
@pytest.mark.parametrize("M,N", [(1, 1), (2, 33), (63, 32), (64, 31), (65, 1), (129, 130), (4097, 65), (9001, 3)])
def test_column_means(gp, layout, M, N):
    import torch

    g = np.random.default_rng(M * 10007 + N)
    X = (g.standard_normal((M, N)) + 100.0).astype(np.float32)
    X64 = X.astype(np.float64)
    Xc = X64 - X64.mean(axis=0, keepdims=True)
    Xd = torch.from_numpy(X).cuda()
    if layout == "col":
        Xd = Xd.t().contiguous().t()
    with gp.Handle(M, N, 1) as h:
        r = h.fit(Xd, 1, tol=1e-6, max_iter=3, center=1, want_R=True)
        torch.cuda.synchronize()
        tp = r.T.cpu().numpy().astype(np.float64) @ r.P.cpu().numpy().astype(np.float64).T
        back = r.R.cpu().numpy().astype(np.float64) + tp
    bar = 8 * 2.0**-24 * (np.abs(Xc).max() + np.abs(tp).max())
    assert np.abs(back - Xc).max() <= bar
