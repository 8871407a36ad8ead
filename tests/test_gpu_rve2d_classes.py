"""2D batches of many grid sizes: every size has a launch of its own (block shape, scratch and work
queue of its size; the multigrid grids 6, 8, 12, 16, 24, 32 in mixed precision a kernel with the size
compiled in), forked beside each other.  All even sizes 2..32 in one call, through the whole-batch and
through the device-list entry, against the FP64 oracle point by point; and a size alone gives the same
bits as in the batch."""
import numpy as np
import pytest

import synth
from gpu_harness import gpu_batch, rel_err
from oracle.rve import PeriodicRVE

pytestmark = pytest.mark.gpu

SIZES = list(range(2, 33, 2))
TOL = {"fp64": 1e-10, "mixed": 1e-5}
STRICT = dict(newton_rtol=1e-13, newton_atol=1e-15, cg_rtol=1e-8, cond_rtol=1e-11)


def rves():
    u = synth.uniform(811, np.arange(len(SIZES)), 4)
    phases = [synth.phase_from_inclusions(n, 2, [u[k, :2]], [0.2 + 0.15 * u[k, 2]]) for k, n in enumerate(SIZES)]
    E = np.array([[1.0, 5.0 + 40.0 * u[k, 3]] for k in range(len(SIZES))])
    return phases, E, np.full((len(SIZES), 2), 0.3)


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_every_size_in_one_call(precision):
    import torch

    import paper_1908_08292_gb300 as fe

    phases, E, nu = rves()
    qp_rve = np.array([5, 15, 0, 3, 7, 11, 2, 15, 1, 4, 6, 8, 9, 10, 12, 13, 14, 3], dtype=np.int32)
    n_qp = len(qp_rve)
    Fs = synth.random_F(812, n_qp, 2, 0.1)
    opts = STRICT if precision == "fp64" else {}
    refs = [PeriodicRVE(SIZES[r], 2, phases[r], E[r], nu[r]).solve(F, rtol=1e-14, atol=1e-16)
            for r, F in zip(qp_rve, Fs)]
    dev = torch.device("cuda:0")
    with fe.Context(2, precision, **opts) as ctx:
        ctx.add_rves(SIZES, phases, E, nu)
        ctx.bind_qps(qp_rve)
        F = torch.tensor(Fs.reshape(n_qp, 4), dtype=torch.float64, device=dev)
        out = []
        for subset in (None, [1, 2, 3, 8, 12, 15, 17]):
            P = torch.full((n_qp, 4), 7.0, dtype=torch.float64, device=dev)
            A = torch.full((n_qp, 16), 7.0, dtype=torch.float64, device=dev)
            st = torch.full((n_qp,), -1, dtype=torch.int32, device=dev)
            if subset is None:
                ctx.rve_solve(F, P, A, st, flags=fe.SOLVE_FROM_COMMITTED)
            else:
                lst = torch.tensor(subset, dtype=torch.int32, device=dev)
                cnt = torch.tensor([len(subset)], dtype=torch.int32, device=dev)
                ctx.rve_solve_list(F, P, A, st, None, fe.SOLVE_FROM_COMMITTED, lst, cnt)
            torch.cuda.synchronize()
            out.append((P.cpu().numpy(), A.cpu().numpy(), st.cpu().numpy()))
    for q in range(n_qp):
        assert out[0][2][q] == 0
        assert rel_err(out[0][0][q], refs[q]["P"], 1e-3) < TOL[precision]
        assert rel_err(out[0][1][q], refs[q]["A"], 1e-3) < TOL[precision]
        if q in (1, 2, 3, 8, 12, 15, 17):  # the list entry: the same solves
            for k in range(3):
                np.testing.assert_array_equal(out[1][k][q], out[0][k][q])
        else:
            assert out[1][2][q] == -1 and np.all(out[1][0][q] == 7.0) and np.all(out[1][1][q] == 7.0)
    one = gpu_batch(2, precision, [SIZES[3]], [phases[3]], [E[3]], [nu[3]], [0, 0], Fs[[3, 17]], **opts)
    np.testing.assert_array_equal(one["P"].reshape(2, 4), out[0][0][[3, 17]])
    np.testing.assert_array_equal(one["A"].reshape(2, 16), out[0][1][[3, 17]])
