"""The FP64-mode 2D kernel at the edges of its thread layout: one degree of freedom per thread up to 16 x 16, two up to
22 x 22 (stencil rows in registers), four beyond (rows in block scratch); a block's smallest shape (four warps) with
and without idle lanes; multigrid levels in shared memory up to 24 x 24, in block scratch at 32 x 32.  Both laws and
both preconditioners, against the FP64 oracle at the tolerance of FP64 mode, then once more with kept transfer
solutions."""
import ctypes

import numpy as np
import pytest

import synth
from gpu_harness import gpu_batch, rel_err
from oracle.rve import PeriodicRVE

pytestmark = pytest.mark.gpu

SIZES = [2, 6, 8, 10, 12, 16, 18, 22, 24, 32]
TOL = 1e-10  # the FP64-mode tolerance of the other parity tests
STRICT = dict(newton_rtol=1e-13, newton_atol=1e-15, cg_rtol=1e-8, cond_rtol=1e-11)


@pytest.mark.parametrize("precond", [1, 0])
@pytest.mark.parametrize("law", ["nh", "svk"])
def test_layout_edges(law, precond):
    import torch

    import paper_1908_08292_gb300 as fe

    u = synth.uniform(821, np.arange(len(SIZES)), 4)
    phases = [synth.phase_from_inclusions(n, 2, [u[k, :2]], [0.2 + 0.15 * u[k, 2]]) for k, n in enumerate(SIZES)]
    E = np.array([[1.0, 3.0 + 10.0 * u[k, 3]] for k in range(len(SIZES))])
    nu = np.full((len(SIZES), 2), 0.3)
    n_qp = len(SIZES)
    F1 = synth.random_F(822, n_qp, 2, 0.05)
    F2 = F1 + 0.01 * (synth.random_F(823, n_qp, 2, 1.0) - np.eye(2))
    dev = torch.device("cuda:0")
    with fe.Context(2, "fp64", law=1 if law == "svk" else 0, precond=precond, transfer_warm=1, **STRICT) as ctx:
        ctx.add_rves(SIZES, phases, E, nu)
        ctx.bind_qps(np.arange(n_qp, dtype=np.int32))
        for Fs in (F1, F2):
            F = torch.tensor(Fs.reshape(n_qp, 4), dtype=torch.float64, device=dev)
            P = torch.zeros(n_qp, 4, dtype=torch.float64, device=dev)
            A = torch.zeros(n_qp, 16, dtype=torch.float64, device=dev)
            W = torch.zeros(n_qp, dtype=torch.float64, device=dev)
            st = torch.full((n_qp,), -1, dtype=torch.int32, device=dev)
            ctx.rve_solve(F, P, A, st, None, W, flags=4)
            torch.cuda.synchronize()
            for q, n in enumerate(SIZES):
                ref = PeriodicRVE(n, 2, phases[q], E[q], nu[q], law=law).solve(Fs[q], rtol=1e-14, atol=1e-16)
                assert int(st[q]) == 0, n
                assert rel_err(P[q].cpu().numpy(), ref["P"], 1e-3) < TOL, n
                assert rel_err(A[q].cpu().numpy(), ref["A"], 1e-3) < TOL, n
                assert abs(float(W[q]) - ref["W"]) <= TOL * max(abs(ref["W"]), 1e-3), n


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n", [6, 10])
def test_collapsed_point_is_reported(precision, n):
    """det F = 1e-50, below the range of the residual's FP32 reciprocal: the point fails, as with det F <= 0, and does
    not disturb its neighbour in the batch.  n = 6: two lanes per element, n = 10 one."""
    phase = synth.phase_from_inclusions(n, 2, [[0.5, 0.5]], [0.25])
    Fs = np.stack([1e-25 * np.eye(2), np.array([[1.02, 0.01], [0.0, 0.99]])])
    out = gpu_batch(2, precision, [n], [phase], [[1.0, 10.0]], [[0.3, 0.3]], [0, 0], Fs)
    ref = PeriodicRVE(n, 2, phase, [1.0, 10.0], [0.3, 0.3]).solve(Fs[1], rtol=1e-14, atol=1e-16)
    assert out["status"][0] != 0 and out["status"][1] == 0
    assert rel_err(out["P"][1], ref["P"], 1e-3) < 1e-5  # default tolerances in both modes


@pytest.mark.parametrize("precond", [1, 0])
@pytest.mark.parametrize("n", [4, 6, 10, 12, 14, 16])
def test_noalloc_preconditioners(n, precond):
    """The no-allocation entry on grids with a multigrid hierarchy (6, 12, 16) and without, by either option."""
    import torch

    import paper_1908_08292_gb300 as fe
    dev = torch.device("cuda:0")
    n_qp = 3
    E, nu = np.array([1.0, 25.0]), np.array([0.3, 0.3])
    u = synth.uniform(841, np.arange(n_qp), 3)
    phases = [synth.phase_from_inclusions(n, 2, [u[q, :2]], [0.2 + 0.1 * u[q, 2]]) for q in range(n_qp)]
    table = np.zeros((n_qp, 4, 2))
    table[:, :2, 0] = E * nu / ((1 + nu) * (1 - 2 * nu))
    table[:, :2, 1] = E / (2 * (1 + nu))
    opt = fe.Options()
    assert fe.lib().fehmm_default_options(ctypes.byref(opt), 2, fe.PREC_FP64) == 0
    for k, v in dict(STRICT, precond=precond).items():
        setattr(opt, k, v)
    Fs = synth.random_F(842, n_qp, 2, 0.1)
    t = dict(phase=torch.tensor(np.stack(phases), dtype=torch.uint8, device=dev), lame=torch.tensor(table, device=dev),
             w=torch.zeros(n_qp, 2 * n * n, dtype=torch.float64, device=dev), F=torch.tensor(Fs.reshape(n_qp, 4), device=dev),
             P=torch.zeros(n_qp, 4, dtype=torch.float64, device=dev), A=torch.zeros(n_qp, 16, dtype=torch.float64, device=dev),
             st=torch.full((n_qp,), -1, dtype=torch.int32, device=dev), it=torch.zeros(n_qp, 4, dtype=torch.int32, device=dev))
    p = {k: ctypes.c_void_p(v.data_ptr()) for k, v in t.items()}
    rc = fe.lib().fehmm_rve2d_solve_fp64_noalloc(n_qp, n, 1, p["phase"], p["lame"], p["w"], p["F"], p["P"], p["A"], p["st"],
                                                 p["it"], ctypes.byref(opt),
                                                 ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0
    torch.cuda.synchronize()
    for q in range(n_qp):
        ref = PeriodicRVE(n, 2, phases[q], E, nu).solve(Fs[q], rtol=1e-14, atol=1e-16)
        assert int(t["st"][q]) == 0
        assert rel_err(t["P"][q].cpu().numpy(), ref["P"], 1e-3) < TOL
        assert rel_err(t["A"][q].cpu().numpy(), ref["A"], 1e-3) < TOL
