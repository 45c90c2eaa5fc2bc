"""What the tracing counts: the bytes of the fine velocity sweeps (a sweep
that forms its first iterate reads no vector for it), and the whole cycles
that one cluster launch takes as coarse levels."""
import numpy as np
import pytest

from paper_2501_11767_gb300 import chnss, inputs

pytestmark = pytest.mark.gpu


def _profiled_solve(n, precision, sys):
    import torch
    p = inputs.default_params()
    p.update(precision=precision, ortho=1 if precision else 0)
    ctx = chnss.Context(chnss.Mesh(n), p)
    ctx.assemble(chnss.state_to_device(inputs.initial_state(n)))
    ctx.profile_enable(True)
    b = np.random.default_rng(1).standard_normal(ctx.system_size(sys))
    b[2 * ctx.mesh.N2:] = 0.0
    _, info, _ = ctx.solve(sys, torch.as_tensor(b, device="cuda"))
    return ctx, ctx.profile_read()["kinds"], info["iters"]


@pytest.mark.parametrize("precision,value", [(0, None), (1, 4), (2, 2)])
def test_velocity_sweep_bytes(precision, value):
    n = 64
    ctx, kinds, iters = _profiled_solve(n, precision, chnss.SYS_NS)
    nnz = len(ctx.export_csr(chnss.MAT_A)[1]) // 4
    N2 = ctx.mesh.N2
    fine = kinds["mg_velocity_spmv_fine"]
    assert fine["launches"] >= 8 * iters and fine["launches"] % 8 == 0      # degree 4: 3 + residual + 4
    cycles = fine["launches"] // 8
    # vectors of the three steps from zero, the residual, the four steps after the correction: out, u, b, dinv
    # (and w) each; a stencil's first step has no u, its second no w
    if value is None:     # FP64, 2x2-block SELL
        want = 8 * (nnz * 36.0 + 4.0 * (N2 + 1)) + (4 + 5 + 5 + 3 + 4 + 15) * 2.0 * N2 * 8
    else:
        want = 8 * 2.0 * nnz * value + (3 + 4 + 5 + 3 + 4 + 15) * 2.0 * N2 * 4
    assert fine["bytes"] == pytest.approx(cycles * want, rel=1e-12)
    assert kinds["mg_velocity_coarse_levels"]["launches"] == cycles


def test_whole_cycles_of_a_cluster_are_timed():
    _, kinds, iters = _profiled_solve(16, 1, chnss.SYS_NS)
    assert kinds["mg_velocity_spmv_fine"]["launches"] == 0
    assert kinds["mg_velocity_coarse_levels"]["launches"] >= iters
    assert kinds["mg_velocity_coarse_levels"]["ms"] > 0
    assert kinds["mg_p1_coarse_levels"]["launches"] >= iters                 # K_p
    _, kinds, iters = _profiled_solve(16, 0, chnss.SYS_AC)
    assert kinds["mg_p1_coarse_levels"]["launches"] >= iters
