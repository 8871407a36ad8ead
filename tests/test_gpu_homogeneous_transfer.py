"""Transfer solves whose right-hand side is nothing but rounding, or exactly zero, from a start value that is not: a
homogeneous RVE with the kept solutions of another deformation.  Such a point converges like any other."""
import numpy as np
import pytest

import synth
from gpu_harness import rel_err
from oracle import material as mat

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("dim,n", [(2, 2), (2, 4), (2, 8), (2, 18), (2, 24), (3, 2), (3, 4)])
def test_homogeneous_rve_from_kept_transfer_solutions(dim, n, precision):
    import torch

    import paper_1908_08292_gb300 as fe

    n_qp, dev = 60, torch.device("cuda:0")
    lam, mu = mat.lame(1.0, 0.3)
    with fe.Context(dim, precision) as ctx:
        ctx.add_rves([n], [np.zeros(n ** dim, np.uint8)], [[1.0]], [[0.3]])
        ctx.bind_qps(np.zeros(n_qp, dtype=np.int32))
        Fs = synth.random_F(901, n_qp, dim, 0.1)
        Fs[::7] = np.eye(dim) * 1.5  # exact in binary: L is exactly zero
        for k in range(4):
            F = torch.tensor(Fs.reshape(n_qp, dim * dim), device=dev)
            P = torch.zeros(n_qp, dim * dim, dtype=torch.float64, device=dev)
            A = torch.zeros(n_qp, dim ** 4, dtype=torch.float64, device=dev)
            st = torch.full((n_qp,), -1, dtype=torch.int32, device=dev)
            ctx.rve_solve(F, P, A, st)
            torch.cuda.synchronize()
            st, P, A = st.cpu().numpy(), P.cpu().numpy(), A.cpu().numpy()
            assert np.all(st == 0), (k, np.nonzero(st)[0], st[st != 0])
            for q in range(n_qp):
                tol = 1e-10 if precision == "fp64" else 1e-5
                assert rel_err(P[q], mat.P_of_F(Fs[q], lam, mu), 1e-3) < tol
                assert rel_err(A[q], mat.A_of_F(Fs[q], lam, mu), 1e-3) < tol
            Fs = Fs[np.roll(np.arange(n_qp), 1)] if k % 2 else Fs + 0.01 * (synth.random_F(902 + k, n_qp, dim, 1.0) - np.eye(dim))
            Fs[::5] = np.eye(dim) * 1.25
