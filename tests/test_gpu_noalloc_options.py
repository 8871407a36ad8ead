"""The multigrid options of the no-allocation entry: the same damping and reuse of levels as in a context's FP64 solve,
to the same iteration counts; options that name no damping at all; and the way from multigrid to block-Jacobi."""
import ctypes

import numpy as np
import pytest

import synth
from gpu_harness import gpu_batch, rel_err
from oracle.rve import PeriodicRVE

pytestmark = pytest.mark.gpu

TOL = 1e-10  # the FP64-mode tolerance of the other parity tests
STRICT = dict(newton_rtol=1e-13, newton_atol=1e-15, cg_rtol=1e-8, cond_rtol=1e-11)
E, NU = np.array([1.0, 6.0]), np.array([0.3, 0.3])


def problem(n, n_qp, amplitude):
    u = synth.uniform(871, np.arange(n_qp), 3)
    phases = [synth.phase_from_inclusions(n, 2, [u[q, :2]], [0.2 + 0.1 * u[q, 2]]) for q in range(n_qp)]
    return phases, synth.random_F(872, n_qp, 2, amplitude)


def noalloc(n, phases, Fs, **options):
    import torch

    import paper_1908_08292_gb300 as fe
    dev = torch.device("cuda:0")
    n_qp = len(Fs)
    table = np.zeros((n_qp, 4, 2))
    table[:, :2, 0] = E * NU / ((1 + NU) * (1 - 2 * NU))
    table[:, :2, 1] = E / (2 * (1 + NU))
    opt = fe.Options()
    assert fe.lib().fehmm_default_options(ctypes.byref(opt), 2, fe.PREC_FP64) == 0
    for k, v in dict(STRICT, **options).items():
        setattr(opt, k, v)
    t = dict(phase=torch.tensor(np.stack(phases), dtype=torch.uint8, device=dev), lame=torch.tensor(table, device=dev),
             w=torch.zeros(n_qp, 2 * n * n, dtype=torch.float64, device=dev), F=torch.tensor(Fs.reshape(n_qp, 4), device=dev),
             P=torch.zeros(n_qp, 4, dtype=torch.float64, device=dev), A=torch.zeros(n_qp, 16, dtype=torch.float64, device=dev),
             status=torch.full((n_qp,), -1, dtype=torch.int32, device=dev),
             iters=torch.zeros(n_qp, 4, dtype=torch.int32, device=dev))
    rc = fe.lib().fehmm_rve2d_solve_fp64_noalloc(n_qp, n, 1, *(ctypes.c_void_p(v.data_ptr()) for v in t.values()),
                                                 ctypes.byref(opt),
                                                 ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0
    torch.cuda.synchronize()
    return {k: t[k].cpu().numpy() for k in ("P", "A", "status", "iters")}


@pytest.mark.parametrize("omega,reuse", [(0.7, 1), (0.7, 0), (0.4, 1), (0.55, 0)])
@pytest.mark.parametrize("n", [6, 8, 12, 16])
def test_damping_and_reuse_as_in_a_context(n, omega, reuse):
    phases, Fs = problem(n, 4, 0.08)
    got = noalloc(n, phases, Fs, mg_omega=omega, mg_reuse=reuse)
    ref = gpu_batch(2, "fp64", [n] * 4, phases, [E] * 4, [NU] * 4, np.arange(4), Fs, mg_omega=omega, mg_reuse=reuse,
                    transfer_warm=0, **STRICT)
    assert np.all(got["status"] == 0) and np.all(ref["status"] == 0)
    np.testing.assert_array_equal(got["iters"], ref["iters"])  # the same kernel with the same settings
    for q in range(4):
        assert rel_err(got["P"][q], ref["P"][q], 1e-3) < TOL and rel_err(got["A"][q], ref["A"][q], 1e-3) < TOL


@pytest.mark.parametrize("omega", [0.0, -0.5, 1.0, 3.0, float("nan")])
def test_no_damping_is_block_jacobi(omega):
    phases, Fs = problem(8, 3, 0.08)
    got, ref = noalloc(8, phases, Fs, mg_omega=omega), noalloc(8, phases, Fs, precond=0)
    for k in ref:
        np.testing.assert_array_equal(got[k], ref[k])


def test_multigrid_gives_way_to_block_jacobi():
    """A cap of 64 PCG iterations and a tolerance of 1e-150, which none of them meets: every Newton correction is tried
    with the levels kept from the last tangent (from the second on), with fresh ones at the damping 0.7, 0.35, 0.175 and
    0.0875, and then with block-Jacobi, whose step is taken.  Newton converges to the oracle's solution.  So do the
    transfer's four solves with that cap and tolerance (the first once more, for the kept levels), which the status
    reports."""
    phases, Fs = problem(8, 3, 0.02)
    capped = noalloc(8, phases, Fs, max_cg=64, cg_rtol=1e-150)
    transfer = noalloc(8, phases, Fs, max_cond_cg=64, cond_rtol=1e-150)
    assert np.all(capped["status"] == 0) and np.all(transfer["status"] == 5)
    np.testing.assert_array_equal(capped["iters"][:, 1], 64 * (5 + 6 * (capped["iters"][:, 0] - 1)))
    assert np.all(transfer["iters"][:, 2] == 64 * (1 + 4 * 5)) and np.all(transfer["iters"][:, 3] == 64 * 5)
    for q in range(3):
        ref = PeriodicRVE(8, 2, phases[q], E, NU).solve(Fs[q], rtol=1e-14, atol=1e-16)
        for got in (capped, transfer):
            assert rel_err(got["P"][q], ref["P"], 1e-3) < TOL and rel_err(got["A"][q], ref["A"], 1e-3) < TOL


@pytest.mark.parametrize("cap", [1, 3, 12, 63])
def test_a_low_cap_truncates(cap):
    """Below 64 a cap that binds is the caller's truncation: no correction and no transfer solve takes more iterations
    than it, as with block-Jacobi."""
    phases, Fs = problem(8, 3, 0.02)
    for precond in (0, 1):
        newton = noalloc(8, phases, Fs, max_cg=cap, cg_rtol=1e-150, max_newton=5, precond=precond)
        transfer = noalloc(8, phases, Fs, max_cond_cg=cap, cond_rtol=1e-150, precond=precond)
        np.testing.assert_array_equal(newton["iters"][:, 1], cap * newton["iters"][:, 0])
        assert np.all(transfer["status"] == 5) and np.all(transfer["iters"][:, 2] == 4 * cap)
