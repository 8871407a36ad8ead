"""The macro CG whose blocks exchange words, when a wait for one runs out: the kernel returns, says so, and leaves
nothing that could pass for a result; the next solve on the same context is an ordinary one.  The wait is cut short by
a limit of zero cycles, with which a block gives up on the first word that is not there yet."""
import numpy as np
import pytest
import scipy.sparse.linalg as spl

import synth
from oracle import material as mat
from oracle.macro import MacroMesh

pytestmark = pytest.mark.gpu


# 2D: 8, 4 and 2 lanes per row; 3D; the last a mesh of one block, which waits for nobody
@pytest.mark.parametrize("n_el,waits", [((30, 30), True), ((46, 50), True), ((69, 69), True), ((6, 12, 12), True),
                                        ((7, 7), False)])
def test_wait_that_runs_out_is_reported(n_el, waits):
    import torch

    import paper_1908_08292_gb300 as fe

    d = len(n_el)
    mesh = MacroMesh(n_el)
    lam, mu = mat.lame(3.0, 0.3)
    F = synth.random_F(531, mesh.n_qp, d, 0.05)
    P, A = mat.P_of_F(F, lam, mu), mat.A_of_F(F, lam, mu)
    f_ref, K_ref = mesh.assemble(P, A)
    fixed = np.nonzero(np.isclose(mesh.X[:, 0], 0.0))[0]
    dofs = (fixed[:, None] * d + np.arange(d)).reshape(-1).astype(np.int32)
    free = np.setdiff1d(np.arange(mesh.n_dof), dofs)
    ref = np.zeros(mesh.n_dof)
    ref[free] = spl.spsolve(K_ref.tocsc()[free][:, free], -f_ref[free])
    dev = torch.device("cuda:0")
    with fe.Context(d, "fp64") as ctx:
        ctx.macro_create(n_el)
        ctx.macro_set_dirichlet(dofs, np.zeros(dofs.size))
        _, _, nr, nnz = ctx.macro_csr()
        f = torch.zeros(nr, dtype=torch.float64, device=dev)
        K = torch.zeros(nnz, dtype=torch.float64, device=dev)
        ctx.macro_assemble(torch.tensor(P.reshape(-1, d * d), device=dev),
                           torch.tensor(A.reshape(-1, d ** 4), device=dev), f, K)
        with pytest.raises(fe.FehmmError):
            ctx.macro_set_wait_limit(-1)
        for limit in (1 << 32, 0, 1 << 32, 0, 1 << 32):
            du = torch.zeros(nr, dtype=torch.float64, device=dev)
            info = torch.full((3,), 7.0, dtype=torch.float64, device=dev)
            ctx.macro_set_wait_limit(limit)
            ctx.macro_solve(K, f, du, info, rtol=1e-13, max_it=20000)
            torch.cuda.synchronize()
            norm, _, status = info.cpu().numpy()
            if waits and limit == 0:
                assert status == 3 and np.isnan(norm)
                continue
            assert status == 0 and abs(norm - np.linalg.norm(f_ref[free])) <= 1e-12 * norm
            # CG stops at 1e-13 of the preconditioned residual; times the square root of the condition number
            assert np.abs(du.cpu().numpy() - ref).max() <= 1e-8 * np.abs(ref).max()
