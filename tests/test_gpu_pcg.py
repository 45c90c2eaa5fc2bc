"""The mass solve's two-kernel conjugate gradients: against a sparse LU at
meshes whose rows end inside a block and fill more than one grid pass, on a
zero, an infinite and a huge right-hand side, and with the solution over the
right-hand side (relative tolerance 1e-12; the scaled mass matrix has
condition number below 8)."""
import numpy as np
import pytest
import scipy.sparse as sp
import scipy.sparse.linalg as spla

from paper_2501_11767_gb300 import chnss, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 4, 20, 34, 256, 1024])
def test_mass_solve_against_lu(n):
    import torch
    ctx = chnss.Context(chnss.Mesh(n), inputs.default_params())
    ctx.assemble(chnss.state_to_device(inputs.initial_state(n)))
    rp, col, val = ctx.export_csr(chnss.MAT_M)
    M = sp.csr_matrix((val, col, rp)).tocsc()
    b = np.random.default_rng(n).standard_normal(M.shape[0])
    x, info, _ = ctx.solve(chnss.SYS_MU_A, torch.as_tensor(b, device="cuda"))
    assert info["converged"] and info["rel_residual"] <= 1e-12
    r = M @ x.cpu().numpy() - b
    assert np.linalg.norm(r) <= 1.1e-12 * np.linalg.norm(b)
    if n <= 256:
        ref = spla.spsolve(M, b)
        assert np.linalg.norm(x.cpu().numpy() - ref) <= 8 * 1.1e-12 * np.linalg.norm(ref)


def test_special_right_hand_sides():
    import torch
    ctx = chnss.Context(chnss.Mesh(16), inputs.default_params())
    ctx.assemble(chnss.state_to_device(inputs.initial_state(16)))
    b = torch.zeros(ctx.mesh.N1, dtype=torch.float64, device="cuda")
    x, info, st = ctx.solve(chnss.SYS_MU_A, b)
    assert st == 0 and info["iters"] == 0 and not x.any()
    b += 1e140
    x, info, st = ctx.solve(chnss.SYS_MU_A, b)
    assert st == 0 and info["converged"]
    b[3] = float("inf")
    _, info, st = ctx.solve(chnss.SYS_MU_A, b, check=False)
    assert st == 6 and not info["converged"]             # CHNSS_ERR_NAN
