"""The launch count (chnss_profile.launches) around a smoothed-aggregation
handle: making one counts the kernels that ran, not those recorded into its
graphs; a replay counts its graph's kernels."""
import numpy as np
import pytest

from paper_2501_11767_gb300 import chnss, inputs

pytestmark = pytest.mark.gpu


def test_create_counts_what_ran():
    import torch
    ctx = chnss.Context(chnss.Mesh(4), inputs.default_params())   # any context reads the library's count
    n = 50                                                        # one level: the diagonal, then the numeric setup
    A = np.eye(n) * 4 - np.eye(n, k=1) - np.eye(n, k=-1)
    r, c = np.nonzero(A)
    dev = lambda a, t: torch.as_tensor(a, dtype=t, device="cuda")   # noqa: E731
    rp = dev(np.concatenate([[0], np.cumsum(np.bincount(r))]), torch.int32)
    col, val = dev(c, torch.int32), dev(A[r, c], torch.float64)
    count = lambda: ctx.profile_read()["launches"]   # noqa: E731
    c0 = count()
    h = chnss.Amg(rp, col, val, 0)
    c1 = count()
    h.update(val)
    c2 = count()
    h.vcycle(torch.ones(n, dtype=torch.float64, device="cuda"))
    c3 = count()
    numeric, cycle = c2 - c1, c3 - c2
    assert numeric > 20 and cycle == 3            # ten power steps of three; copy in, inverse, copy out
    assert c1 - c0 == numeric + 1
