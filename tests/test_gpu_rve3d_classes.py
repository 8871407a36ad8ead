"""3D batches of several grid sizes (a launch per size, forked beside each other) and of more points than SMs
(two smaller blocks per SM), through the whole-batch and the device-list entry, both laws and couplings."""
import numpy as np
import pytest

import synth
from gpu_harness import gpu_batch, rel_err
from oracle.kubc import DirichletRVE
from oracle.rve import PeriodicRVE

pytestmark = pytest.mark.gpu

SIZES = [2, 3, 4, 5, 6, 7, 8]
TOL = {"fp64": 1e-10, "mixed": 1e-5}
STRICT = dict(newton_rtol=1e-13, newton_atol=1e-15, cg_rtol=1e-9, cond_rtol=1e-11)


def rves():
    u = synth.uniform(831, np.arange(len(SIZES)), 4)
    phases = [synth.sphere_rve(n, 1, 0.1 + 0.2 * u[k, 3], u[k, None, :3]) for k, n in enumerate(SIZES)]
    return phases, np.tile([1.0, 10.0], (len(SIZES), 1)), np.full((len(SIZES), 2), 0.3)


@pytest.mark.parametrize("precision,law,bc", [("mixed", 0, 0), ("mixed", 1, 1), ("fp64", 0, 0)])
def test_every_small_size_in_one_call(precision, law, bc):
    import torch

    import paper_1908_08292_gb300 as fe

    phases, E, nu = rves()
    qp_rve = np.array([6, 0, 3, 1, 5, 2, 4, 6, 2], dtype=np.int32)
    n_qp = len(qp_rve)
    Fs = synth.random_F(832, n_qp, 3, 0.06)
    opts = dict(STRICT if precision == "fp64" else {}, law=law, bc=bc)
    dev = torch.device("cuda:0")
    with fe.Context(3, precision, **opts) as ctx:
        ctx.add_rves(SIZES, phases, E, nu)
        ctx.bind_qps(qp_rve)
        F = torch.tensor(Fs.reshape(n_qp, 9), dtype=torch.float64, device=dev)
        out = []
        for subset in (None, [0, 2, 6, 8]):
            P = torch.full((n_qp, 9), 7.0, dtype=torch.float64, device=dev)
            A = torch.full((n_qp, 81), 7.0, dtype=torch.float64, device=dev)
            st = torch.full((n_qp,), -1, dtype=torch.int32, device=dev)
            if subset is None:
                ctx.rve_solve(F, P, A, st, flags=fe.SOLVE_FROM_COMMITTED)
            else:
                ctx.rve_solve_list(F, P, A, st, None, fe.SOLVE_FROM_COMMITTED,
                                   torch.tensor(subset, dtype=torch.int32, device=dev),
                                   torch.tensor([len(subset)], dtype=torch.int32, device=dev))
            torch.cuda.synchronize()
            out.append((P.cpu().numpy(), A.cpu().numpy(), st.cpu().numpy()))
    for q, r in enumerate(qp_rve):
        if bc:
            if law:
                continue  # no oracle for both: the list entry below, and the other parametrisations
            ref = DirichletRVE(SIZES[r], 3, phases[r], E[r], nu[r]).solve(Fs[q], rtol=1e-14, atol=1e-16)
        else:
            ref = PeriodicRVE(SIZES[r], 3, phases[r], E[r], nu[r]).solve(Fs[q], rtol=1e-14, atol=1e-16)
        assert rel_err(out[0][0][q], ref["P"], 1e-3) < TOL[precision]
        assert rel_err(out[0][1][q], ref["A"], 1e-3) < TOL[precision]
    assert np.all(out[0][2] == 0)
    for q in range(n_qp):
        if q in (0, 2, 6, 8):
            assert out[1][2][q] == 0
            assert rel_err(out[1][0][q], out[0][0][q], 1e-3) < TOL[precision]
            assert rel_err(out[1][1][q], out[0][1][q], 1e-3) < TOL[precision]
        else:
            assert out[1][2][q] == -1 and np.all(out[1][1][q] == 7.0)


@pytest.mark.parametrize("law", [0, 1])
def test_more_points_than_sms(law):
    """330 points of 4^3 and 8^3: two blocks of 256 threads per SM; a few of them again in a call of their own
    (512 threads)."""
    phases, E, nu = rves()
    n_qp = 330
    qp_rve = np.where(np.arange(n_qp) % 3 == 0, 6, 2)
    Fs = synth.random_F(833, n_qp, 3, 0.06)
    big = gpu_batch(3, "mixed", SIZES, phases, E, nu, qp_rve, Fs, flags=4, law=law)
    some = np.array([0, 1, 2, 3, 151, 152, 153, 327, 328, 329])
    small = gpu_batch(3, "mixed", SIZES, phases, E, nu, qp_rve[some], Fs[some], flags=4, law=law)
    assert np.all(big["status"] == 0) and np.all(small["status"] == 0)
    for k, q in enumerate(some):
        assert rel_err(big["P"][q], small["P"][k], 1e-3) < 1e-9  # both within the Newton tolerance
        assert rel_err(big["A"][q], small["A"][k], 1e-3) < 1e-6  # FP32 tangent
        assert abs(big["W"][q] - small["W"][k]) < 1e-12


@pytest.mark.parametrize("size", [3, 4, 5, 6, 7])
def test_block_shapes_of_small_grids(size):
    """A grid's block has the threads its element passes fill evenly: 128 to 448, other shapes with more points than
    SMs (up to four blocks of 128 per SM at 4^3).  A few points of such a batch again in a call of their own."""
    phases, E, nu = rves()
    k = SIZES.index(size)
    n_qp = 330
    Fs = synth.random_F(834, n_qp, 3, 0.06)
    big = gpu_batch(3, "mixed", [size], [phases[k]], E[k:k + 1], nu[k:k + 1], np.zeros(n_qp, dtype=np.int32), Fs)
    some = np.array([0, 1, 153, 328, 329])
    small = gpu_batch(3, "mixed", [size], [phases[k]], E[k:k + 1], nu[k:k + 1], np.zeros(5, dtype=np.int32), Fs[some])
    assert np.all(big["status"] == 0) and np.all(small["status"] == 0)
    for m, q in enumerate(some):
        assert rel_err(big["P"][q], small["P"][m], 1e-3) < 1e-9  # both within the Newton tolerance
        assert rel_err(big["A"][q], small["A"][m], 1e-3) < 1e-6  # FP32 tangent
    ref = PeriodicRVE(size, 3, phases[k], E[k], nu[k]).solve(Fs[329], rtol=1e-14, atol=1e-16)
    assert rel_err(big["P"][329], ref["P"], 1e-3) < TOL["mixed"] and rel_err(big["A"][329], ref["A"], 1e-3) < TOL["mixed"]
