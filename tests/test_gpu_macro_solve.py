"""The macro CG with its rows resident in registers, at the edges of its plans: one block or several (2D: 128
rows, 3D: 64), 8, 4 or 2 lanes per row, a last block with few rows, every row fixed but one; and the general
kernel beyond it.  Against a sparse direct solve of the oracle's assembled system."""
import numpy as np
import pytest
import scipy.sparse.linalg as spl

import synth
from oracle import material as mat
from oracle.macro import MacroMesh

pytestmark = pytest.mark.gpu


# rows: 4, 128 (one block), 144 (several, 8 lanes), 1098, 4794 (4 lanes), 9800 (2 lanes), 20604 (general);
# 3D: 24, 60 (one block), 72 (8 lanes), 3549 (4 lanes), 6591 (2 lanes)
@pytest.mark.parametrize("n_el", [(1, 1), (7, 7), (8, 7), (60, 8), (46, 50), (69, 69), (100, 101), (1, 1, 1), (4, 1, 1),
                                  (2, 1, 3), (6, 12, 12), (12, 12, 12)])
def test_macro_solve_matches_direct_solve(n_el):
    import torch

    import paper_1908_08292_gb300 as fe

    d = len(n_el)
    mesh = MacroMesh(n_el)
    lam, mu = mat.lame(3.0, 0.3)
    F = synth.random_F(521, mesh.n_qp, d, 0.05)
    P, A = mat.P_of_F(F, lam, mu), mat.A_of_F(F, lam, mu)
    f_ref, K_ref = mesh.assemble(P, A)
    dev = torch.device("cuda:0")
    fixed = np.nonzero(np.isclose(mesh.X[:, 0], 0.0))[0]
    dofs = (fixed[:, None] * d + np.arange(d)).reshape(-1).astype(np.int32)
    for dirichlet in (dofs, np.arange(1, mesh.n_dof, dtype=np.int32)):  # the plane x = 0; all dofs but one
        with fe.Context(d, "fp64") as ctx:
            ctx.macro_create(n_el)
            ctx.macro_set_dirichlet(dirichlet, np.zeros(dirichlet.size))
            _, _, nr, nnz = ctx.macro_csr()
            f, du = (torch.full((nr,), 3.0, dtype=torch.float64, device=dev) for _ in range(2))
            K = torch.full((nnz,), 3.0, dtype=torch.float64, device=dev)
            info = torch.zeros(3, dtype=torch.float64, device=dev)
            ctx.macro_assemble(torch.tensor(P.reshape(-1, d * d), device=dev),
                               torch.tensor(A.reshape(-1, d ** 4), device=dev), f, K)
            ctx.macro_solve(K, f, du, info, rtol=1e-13, max_it=20000)
            torch.cuda.synchronize()
            du, info = du.cpu().numpy(), info.cpu().numpy()
            short = torch.zeros(3, dtype=torch.float64, device=dev)
            ctx.macro_solve(K, f, torch.zeros(nr, dtype=torch.float64, device=dev), short, rtol=1e-13, max_it=1)
            short = short.cpu().numpy()
        free = np.setdiff1d(np.arange(mesh.n_dof), dirichlet)
        ref = np.zeros(mesh.n_dof)
        ref[free] = spl.spsolve(K_ref.tocsc()[free][:, free], -f_ref[free]) if free.size > 1 else -f_ref[0] / K_ref[0, 0]
        assert info[2] == 0 and abs(info[0] - np.linalg.norm(f_ref[free])) <= 1e-12 * info[0]
        assert np.all(du[dirichlet] == 0)
        # CG stops at 1e-13 of the preconditioned residual; times the square root of the condition number
        assert np.abs(du - ref).max() <= 1e-8 * np.abs(ref).max()
        if info[1] > 1:
            assert short[1] == 1 and short[2] == 1  # the cap
