"""The cluster kernel of the velocity hierarchy's coarse levels at the sizes
where its line deal and coarsest-level forms change: one block's levels alone
(8, 14), a spread level over one-block ones (16, 24, 32, 48), a dense coarsest
level spread over the blocks (20 -> 5^2), the 25^2 coarsest level alone (50),
FP32 and BF16 values, enclosed and open top.  Against the FP64 step (launches
only) at an outer residual of 1e-10: the library's mixed-precision gate, and
no Oseen count moved by more than rounding does (FP32: 2; BF16 values: 6)."""
import pytest

from paper_2501_11767_gb300 import chnss, inputs
from solve_compare import rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("top_bc", [0, 1])
@pytest.mark.parametrize("n", [8, 14, 16, 20, 24, 32, 48, 50])
def test_mixed_oseen_against_fp64(n, top_bc):
    mesh = chnss.Mesh(n, top_bc=top_bc)
    st = chnss.state_to_device(inputs.initial_state(n, seed=n))
    p = inputs.default_params()
    p.update(rtol=1e-10, top_bc=top_bc)
    ref, rinfo, _ = chnss.Context(mesh, p).step(st)
    ref = chnss.state_to_numpy(ref)
    for precision, moved in ((1, 2), (2, 6)):
        p.update(precision=precision, ortho=1)
        got, info, _ = chnss.Context(mesh, p).step(st)
        assert abs(info["ns"]["iters"] - rinfo["ns"]["iters"]) <= moved, precision
        got = chnss.state_to_numpy(got)
        assert rel(got["v"], ref["v"]) <= 1e-6 and rel(got["p"], ref["p"]) <= 1e-6, precision
