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
