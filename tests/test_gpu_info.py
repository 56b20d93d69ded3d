"""The per-call record (gspca_info): what it says of the launch and of the bytes."""
import numpy as np
import pytest

from test_gpu_f64 import fit64, gp  # noqa: F401  (gp is the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("algo", ["gs", "nipals"])
def test_f64_algorithmic_bytes(gp, algo):  # noqa: F811
    """R once per pass (one more pass per component than iterations) and written by a deflation;
    GS: V for b' every iteration and for the new column at a component's end, W once and U twice
    an iteration (the last iteration's two are the component's start's)."""
    M, N, lock = 500, 120, [7, 6, 9, 5]
    X = np.random.default_rng(2).standard_normal((M, N))
    b = fit64(gp, X, len(lock), algo, iters_lock=lock)["info"]["alg_bytes"]
    want = sum((it + 1 + (k > 0)) * M * N for k, it in enumerate(lock))
    if algo == "gs":
        want += sum((it + 1) * M * k + 3 * it * N * k for k, it in enumerate(lock))
    assert b == 8 * want


def test_block_launch_shape(gp):  # noqa: F811
    """A block fit reports the Gram kernel's launch, grid and block."""
    import os
    import re

    import torch

    src = open(os.path.join(os.path.dirname(gp.__file__), "csrc", "block_kernels.cuh")).read()
    const = {n: int(v) for n, v in re.findall(r"constexpr int (kGram\w+) = (\d+);", src)}
    X = torch.from_numpy(np.random.default_rng(2).standard_normal((300, 60)).astype(np.float32)).cuda()
    with gp.Handle(300, 60, 4) as h:
        info = h.fit_block(X, 4, block=2, tol=1e-3, max_iter=5).info
    assert (info["grid_ctas"], info["block_threads"]) == (const["kGramCtas"], const["kGramThreads"])
