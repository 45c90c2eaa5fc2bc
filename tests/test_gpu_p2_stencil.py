"""The velocity operator's stencil form at the sizes where its cells, masks
and open-top rows can go wrong: the Oseen solution for a right-hand side that
is non-zero on the walls too, its residual recomputed from the exported CSR
blocks.  (Sums of at most 19 blocks in FP64: the recomputed residual differs
from the solver's by rounding only.)"""
import numpy as np
import pytest
import scipy.sparse as sp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lxy", [(1.0, 1.0), (2.0, 0.75)])
@pytest.mark.parametrize("top_bc", [0, 1])
@pytest.mark.parametrize("n", [2, 4, 6, 10, 16, 22, 34])
def test_oseen_residual_from_exported_blocks(n, top_bc, lxy):
    import torch
    from paper_2501_11767_gb300 import chnss, inputs
    mesh = chnss.Mesh(n, *lxy, top_bc=top_bc)
    N1, N2 = mesh.N1, mesh.N2
    rng = np.random.default_rng(100 * n + top_bc)
    for precision in (0, 1, 2):
        p = inputs.default_params()
        p.update(top_bc=top_bc, precision=precision, ortho=1 if precision else 0)
        ctx = chnss.Context(mesh, p)
        st = inputs.initial_state(n, seed=3)
        st["v"] = 0.02 * rng.standard_normal(2 * N2)
        ctx.assemble(chnss.state_to_device(st))
        b = rng.standard_normal(2 * N2 + N1)
        if top_bc == 0:
            b[2 * N2:] -= b[2 * N2:].mean()          # enclosed flow: the pressure rows sum to zero
        x, info, _ = ctx.solve(chnss.SYS_NS, torch.as_tensor(b, device="cuda"))
        assert info["converged"]
        rp, col, val = ctx.export_csr(chnss.MAT_A)
        A = sp.csr_matrix((val, col, rp), shape=(2 * N2, 2 * N2))
        rp, col, val = ctx.export_csr(chnss.MAT_B)
        B = sp.csr_matrix((val, col, rp), shape=(N1, 2 * N2))
        v, q = np.split(x.cpu().numpy(), [2 * N2])
        r = b - np.concatenate([A @ v + B.T @ q, B @ v])
        assert np.linalg.norm(r) <= (p["rtol"] + 1e-12) * np.linalg.norm(b)
