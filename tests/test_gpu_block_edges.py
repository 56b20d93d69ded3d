"""Block power iteration at the edges of its small kernels, against the FP64 oracle at the bars
of test_gpu_block.py: the narrowest, odd and widest blocks (the eigensolver's pairs, the
factorisation's rows), fewer rows than CTAs and rows past a staged chunk (Gram matrix), and data
whose squares leave FP32's range (the small kernels scale by powers of two).
"""
import numpy as np
import pytest

import oracle
import synth
from parity_helpers import angle, clusters, sigma_ok, subspace_angle
from test_gpu_block import fit_block, gp  # noqa: F401  (gp is the fixture)

pytestmark = pytest.mark.gpu

CASES = [(40, 33, 1, 1, 0.8, 1.0), (100, 90, 7, 2, 0.85, 1.0), (300, 129, 33, 32, 0.9, 1.0), (16513, 40, 31, 31, 0.9, 1.0),
         (700, 300, 9, 3, 0.85, 1e-15), (700, 300, 9, 3, 0.85, 1e15)]


@pytest.mark.parametrize("case", CASES, ids=[f"{c[0]}x{c[1]}k{c[2]}b{c[3]}s{c[5]:g}" for c in CASES])
def test_block_edges(gp, case):  # noqa: F811
    M, N, K, b, ratio, scale = case
    X32 = (synth.planted(M, N, 10.0, ratio, 0.01, (98, M, N)).X * scale).astype(np.float32)
    g = fit_block(gp, X32, K, b)
    assert g["status"] in (0, 4) and g["info"]["found"] == K
    ref = oracle.block_fit(X32.astype(np.float64), K, b, tol=1e-6, max_iter=1000, iters_lock=g["iters"])
    assert ref.found == K
    assert sigma_ok(g["lam"], ref.lam).all(), (g["lam"], ref.lam)
    for grp in clusters(ref.lam, 1e-3, floor=1e-2):
        if len(grp) == 1:
            assert angle(g["P"][:, grp[0]], ref.P[:, grp[0]]) <= 1e-3, grp
            assert angle(g["T"][:, grp[0]], ref.T[:, grp[0]]) <= 1e-3, grp
        else:
            assert subspace_angle(g["P"][:, grp], ref.P[:, grp]) <= 1e-3, grp
    assert np.abs(g["P"].T @ g["P"] - np.eye(K)).max() <= 1e-5
    assert np.linalg.norm(g["R"] - ref.R) <= 1e-5 * np.linalg.norm(X32.astype(np.float64))
