"""The dense FP64 inverse of a coarsest level, alone: a matrix of at most 64
rows is a smoothed-aggregation hierarchy of one level, whose V-cycle applies
the inverse.  Sizes at the edges of the column deal (16 blocks) and of a
warp; off-diagonal entries dominate, so rows are exchanged."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 31, 32, 33, 50, 64])
def test_dense_inverse_against_lu(n):
    import torch
    from paper_2501_11767_gb300 import chnss
    rng = np.random.default_rng(n)
    A = rng.uniform(-1, 1, (n, n))
    A[np.arange(n), np.arange(n)] *= 1e-3                       # the diagonal is stored and non-zero, not the pivot
    b = rng.uniform(-1, 1, n)
    dev = lambda a, t: torch.as_tensor(a, dtype=t, device="cuda")   # noqa: E731
    h = chnss.Amg(dev(np.arange(0, n * n + 1, n), torch.int32), dev(np.tile(np.arange(n), n), torch.int32),
                  dev(A.ravel(), torch.float64), 0)
    assert len(h.levels()) == 1
    x = h.vcycle(dev(b, torch.float64)).cpu().numpy()
    ref = np.linalg.solve(A, b)
    # backward error of elimination with row exchanges, growth below 2 n on such matrices
    tol = 4 * n * n * np.finfo(float).eps * np.linalg.cond(A)
    assert np.linalg.norm(x - ref) <= tol * np.linalg.norm(ref)
