"""The cluster kernel of the P1 coarse levels at the sizes where its line
deal, halos and coarsest-level forms change: one-block hierarchies only (10,
14), spread levels down to an odd one solved by Chebyshev steps (34 -> 17),
dense coarsest levels of 9^2 to 15^2 cells (18, 26, 30, 44), the largest
meshes handled whole (64 in FP64, 128 in FP32)."""
import numpy as np
import pytest

from oracle.step import Oracle
from paper_2501_11767_gb300 import chnss, inputs
from solve_compare import compare_solves, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [10, 14, 18, 26, 30, 34, 44, 64])
def test_iterates_match_oracle(n):
    p = inputs.default_params()
    st = inputs.initial_state(n, seed=n)
    ref, rinfo = Oracle(n, p).step(st)
    out, info, _ = chnss.Context(chnss.Mesh(n), p).step(chnss.state_to_device(st))
    compare_solves(chnss.state_to_numpy(out), info, ref, rinfo, st, p, lambda q: Oracle(n, q))


@pytest.mark.parametrize("n", [60, 104, 128])
def test_mixed_precision_close_to_fp64(n):
    """Outer residual 1e-10: the mixed step within 1e-6 of the FP64 one (the
    library's mixed-precision gate), with the preconditioners' rounding moving
    no Krylov count by more than two."""
    mesh = chnss.Mesh(n)
    st = chnss.state_to_device(inputs.initial_state(n, seed=n))
    p = inputs.default_params()
    p.update(rtol=1e-10)
    ref, rinfo, _ = chnss.Context(mesh, p).step(st)
    p.update(precision=1, ortho=1)
    got, info, _ = chnss.Context(mesh, p).step(st)
    for name in ("ch_p", "ch_N", "ch_s", "ac", "ns"):
        assert abs(info[name]["iters"] - rinfo[name]["iters"]) <= 2, name
    a, b = chnss.state_to_numpy(got), chnss.state_to_numpy(ref)
    for key in ("phi", "Phi_v", "v", "p"):
        assert rel(a[key], b[key]) <= 1e-6, key
    assert np.isfinite(a["mu"]).all()
