"""A macro load of 1e-150: the inner products of the CG run out of the normal numbers (their reciprocals would
overflow) before it has converged.  It ends as it does at ordinary scales."""
import numpy as np
import pytest
import scipy.sparse.linalg as spl

import synth
from oracle import material as mat
from oracle.macro import MacroMesh

pytestmark = pytest.mark.gpu


# one block, 8, 4 and 2 lanes per row, the kernel for larger meshes; 3D
@pytest.mark.parametrize("n_el", [(4, 4), (30, 30), (46, 50), (69, 69), (100, 101), (6, 12, 12)])
def test_macro_load_of_1e_minus_150(n_el):
    import torch

    import paper_1908_08292_gb300 as fe

    d, dev = len(n_el), torch.device("cuda:0")
    mesh = MacroMesh(n_el)
    lam, mu = mat.lame(3.0, 0.3)
    F = synth.random_F(911, mesh.n_qp, d, 0.05)
    f_ref, K_ref = mesh.assemble(mat.P_of_F(F, lam, mu), mat.A_of_F(F, lam, mu))
    dofs = (np.nonzero(np.isclose(mesh.X[:, 0], 0.0))[0][:, None] * d + np.arange(d)).reshape(-1).astype(np.int32)
    free = np.setdiff1d(np.arange(mesh.n_dof), dofs)
    ref = np.zeros(mesh.n_dof)
    ref[free] = spl.spsolve(K_ref.tocsc()[free][:, free], -f_ref[free])
    with fe.Context(d, "fp64") as ctx:
        ctx.macro_create(n_el)
        ctx.macro_set_dirichlet(dofs, np.zeros(dofs.size))
        rowptr, col, nr, nnz = ctx.macro_csr()
        f = torch.zeros(nr, dtype=torch.float64, device=dev)
        K = torch.zeros(nnz, dtype=torch.float64, device=dev)
        ctx.macro_assemble(torch.tensor(mat.P_of_F(F, lam, mu).reshape(-1, d * d), device=dev),
                           torch.tensor(mat.A_of_F(F, lam, mu).reshape(-1, d ** 4), device=dev), f, K)
        du = torch.zeros(nr, dtype=torch.float64, device=dev)
        info = torch.zeros(3, dtype=torch.float64, device=dev)
        f *= 1e-150
        ctx.macro_solve(K, f, du, info, rtol=1e-6, max_it=20000)
        torch.cuda.synchronize()
        du, info = du.cpu().numpy(), info.cpu().numpy()
    assert info[2] == 0
    # the smallest number is 1e-324, so the sums resolve a reduction of the residual to 1e-11 or so at best; asked for
    # is 1e-6, times the square root of the condition number (below 1e3)
    assert np.abs(du * 1e150 - ref).max() <= 1e-3 * np.abs(ref).max()
