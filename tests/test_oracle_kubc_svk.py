"""Pins of the KUBC RVE oracle with the St. Venant-Kirchhoff law: a homogeneous RVE is the pointwise law, and Pbar =
dWbar/dFbar, Abar = dPbar/dFbar by finite differences of whole solves."""
import numpy as np
import pytest

import synth
from oracle import material as mat
from oracle.kubc import DirichletRVE


@pytest.mark.parametrize("d", [2, 3])
def test_homogeneous_is_the_pointwise_law(d):
    n = 4
    F = synth.random_F(881, 1, d, 0.15)[0]
    out = DirichletRVE(n, d, np.zeros(n ** d, np.uint8), [2.0, 2.0], [0.3, 0.3], law="svk").solve(F)
    lam, mu = mat.lame(2.0, 0.3)
    assert out["status"] == 0 and out["newton_iters"] == 0
    np.testing.assert_allclose(out["P"], mat.svk_P(F, lam, mu), atol=1e-13)
    np.testing.assert_allclose(out["A"], mat.svk_A(F, lam, mu), atol=1e-12)


@pytest.mark.parametrize("d,n", [(2, 6), (3, 3)])
def test_stress_and_tangent_are_derivatives(d, n):
    phase = synth.phase_from_inclusions(n, d, [[0.45, 0.55, 0.5][:d]], [0.3])
    rve = DirichletRVE(n, d, phase, [1.0, 10.0], [0.3, 0.25], law="svk")
    F = synth.random_F(882, 1, d, 0.08)[0]
    out = rve.solve(F, rtol=1e-14)
    assert out["status"] == 0 and out["newton_iters"] > 0
    h = 1e-5
    for k in range(d):
        for m in range(d):
            E = np.zeros((d, d))
            E[k, m] = h
            hi, lo = rve.solve(F + E, rtol=1e-14, tangent=False), rve.solve(F - E, rtol=1e-14, tangent=False)
            assert abs((hi["W"] - lo["W"]) / (2 * h) - out["P"][k, m]) < 1e-8
            np.testing.assert_allclose((hi["P"] - lo["P"]) / (2 * h), out["A"][:, :, k, m], atol=1e-7)
