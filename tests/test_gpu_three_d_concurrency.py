"""chnss3_set_step_concurrency(0) runs one kernel at a time: the captured 3D
preconditioners have no branches, also when the setting changes after they
were captured, and the step's result stays the same bit for bit."""
import pytest

from paper_2501_11767_gb300 import chnss, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    return torch


@pytest.mark.parametrize("extra", [{"precision": 1}, {"precision": 0, "mobility_kind": 1},
                                   {"precision": 1, "inner_rtol": 1e-3, "inner_maxit": 5}])
def test_switch_sets_the_branches(torch, extra):
    n = 4
    p = inputs.default_params()
    p.update(alpha=[1e-2] * 4, **extra)
    st = chnss.state_to_device(inputs.initial_state_3d(n, seed=3))
    ctx = chnss.Context3(n, p)
    branched, serial = [2, 2, 2, 1, 2], [1] * 5
    assert [ctx.debug_prec_branches(g) for g in range(5)] == [0] * 5
    outs = []
    for on, want in ((True, branched), (False, serial), (True, branched)):
        ctx.set_step_concurrency(on)
        out, info, _ = ctx.step(st)
        got = [ctx.debug_prec_branches(g) for g in range(5)]
        assert got == want, (on, got)
        outs.append((out, {k: v["iters"] for k, v in info.items()}))
    for out, iters in outs[1:]:
        assert iters == outs[0][1]
        for k in out:
            assert torch.equal(out[k], outs[0][0][k]), k
