"""Column means: every entry point adds in the same order, and both forms are right at the lines
between them.

Columns of ones with +-2^55 in them have FP64 sums that depend on the order (one is below half an
ulp of 2^55), so two orders give different means and different fits.
"""
import ctypes

import numpy as np
import pytest

from test_gpu_colmean import gp  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu


def noalloc(gp, Xd, K, center, ctas):  # noqa: F811
    """gspca_fit_noalloc through the C ABI (the binding does not pass grid_ctas)."""
    import torch

    M, N = Xd.shape
    layout, ldx = gp._layout_of(Xd)
    T = torch.empty((K, M), device="cuda").t()
    P = torch.empty((K, N), device="cuda").t()
    lam = torch.empty(K, device="cuda", dtype=torch.float64)
    R = torch.empty((N, M), device="cuda").t()
    o, keep = gp._opts(center=center, grid_ctas=ctas)
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    st = gp.load().gspca_fit_noalloc(None, ptr(Xd), layout, int(ldx), M, N, K, 1e-6, 3, gp._ALGOS["gs"], ptr(T), ptr(P),
                                     ptr(lam), None, ptr(R), ctypes.byref(o))
    del keep
    torch.cuda.synchronize()
    return st, [t.cpu().numpy() for t in (T, P, lam, R)]


@pytest.mark.parametrize("layout", ["row", "col"])
@pytest.mark.parametrize("M,N,ctas", [(8, 64, 0), (300, 90, 0), (700, 40, 0), (3000, 40, 2), (2100, 600, 4)])
def test_entry_points_add_in_the_same_order(gp, layout, M, N, ctas):  # noqa: F811
    import torch

    r = np.random.default_rng(M + N)
    X = (1.0 + 1e-3 * r.standard_normal((M, N))).astype(np.float32)
    for c in range(N):  # as many +2^55 as -2^55
        i = r.permutation(M)[: 2 * max(1, M // 50)]
        X[i[::2], c] = 2.0**55
        X[i[1::2], c] = -(2.0**55)
    Xd = torch.from_numpy(X).cuda()
    if layout == "col":
        Xd = Xd.t().contiguous().t()
    for center in (0, 1):
        with gp.Handle(M, N, 1) as h:
            a = h.fit(Xd, 1, tol=1e-6, max_iter=3, center=center, want_R=True, grid_ctas=ctas)
            torch.cuda.synchronize()
            ref = [t.cpu().numpy() for t in (a.T, a.P, a.lam, a.R)]
        st, got = noalloc(gp, Xd, 1, center, ctas)
        assert st == a.status
        for x, y in zip(ref, got):
            assert np.array_equal(x, y), center


@pytest.mark.parametrize("layout", ["row", "col"])
@pytest.mark.parametrize("M,N", [(64, 2049), (65, 2049), (512, 2051), (513, 2051), (16385, 30), (512, 511), (513, 511), (513, 513), (2048, 512), (2049, 512),
                                 (2049, 999), (2049, 1001), (20001, 1000), (641, 2050), (4099, 35)])
def test_column_means_at_the_lines(gp, layout, M, N):  # noqa: F811
    """At the bar of test_gpu_colmean.py, whose reasoning holds for these sizes as well."""
    import test_gpu_colmean as t

    t.test_column_means(gp, layout, M, N)
