"""Block fit: a block that stops on a loose tolerance does not pay for the half step after.

(Wide blocks go ahead of the test from the second iteration on; theirs hides the half step.)
The launches of a fit that stops by its tolerance after n iterations are those of a fit capped at
n: nothing was enqueued behind the last test.
"""
import numpy as np
import pytest

import synth
from test_gpu_block import gp  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tol,n,block", [(10.0, 1, 3), (10.0, 1, 6), (0.5, 2, 3), (0.2, 2, 3)])
def test_no_launches_behind_the_stop(gp, tol, n, block):  # noqa: F811
    import torch

    X = torch.from_numpy(synth.planted(500, 200, 10.0, 0.6, 0.01, 45).X.astype(np.float32)).cuda()
    with gp.Handle(500, 200, 6) as h:
        a = h.fit_block(X, 6, block=block, tol=tol, max_iter=50)
        b = h.fit_block(X, 6, block=block, tol=1e-12, max_iter=n)
        torch.cuda.synchronize()
        assert a.status == 0 and b.status == 4
        assert a.iters.tolist() == b.iters.tolist() == [n] * 6
        assert torch.equal(a.T, b.T) and torch.equal(a.lam, b.lam)
    assert a.info["kernel_launches"] == b.info["kernel_launches"]
