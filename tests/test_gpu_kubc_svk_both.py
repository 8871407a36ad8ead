"""St. Venant-Kirchhoff law and KUBC coupling together against the FP64 oracle: the multigrid grids and others, 2D and
3D, both precisions and preconditioners."""
import numpy as np
import pytest

import synth
from gpu_harness import gpu_batch, rel_err
from oracle.kubc import DirichletRVE

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-10, "mixed": 1e-5}  # the tolerances of the other parity tests
STRICT = {2: dict(newton_rtol=1e-13, newton_atol=1e-15, cg_rtol=1e-8, cond_rtol=1e-11),
          3: dict(newton_rtol=1e-13, newton_atol=1e-15, cg_rtol=1e-9, cond_rtol=1e-11)}


@pytest.mark.parametrize("precond", [1, 0])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("d,sizes", [(2, [2, 6, 10, 16, 24]), (3, [2, 3, 4, 5, 6, 7, 8])])
def test_svk_with_kubc(d, sizes, precision, precond):
    u = synth.uniform(891, np.arange(len(sizes)), 4)
    phases = [synth.phase_from_inclusions(n, d, [u[k, :d]], [0.2 + 0.15 * u[k, 3]]) for k, n in enumerate(sizes)]
    E, nu = np.tile([1.0, 10.0], (len(sizes), 1)), np.full((len(sizes), 2), 0.3)
    Fs = synth.random_F(892, len(sizes), d, 0.08)
    out = gpu_batch(d, precision, sizes, phases, E, nu, np.arange(len(sizes)), Fs, flags=4, law=1, bc=1, precond=precond,
                    **(STRICT[d] if precision == "fp64" else {}))
    for q, n in enumerate(sizes):
        ref = DirichletRVE(n, d, phases[q], E[q], nu[q], law="svk").solve(Fs[q], rtol=1e-14, atol=1e-16)
        assert out["status"][q] == 0, n
        assert rel_err(out["P"][q], ref["P"], 1e-3) < TOL[precision], n
        assert rel_err(out["A"][q], ref["A"], 1e-3) < TOL[precision], n
        assert abs(out["W"][q] - ref["W"]) <= TOL[precision] * max(abs(ref["W"]), 1e-3), n
