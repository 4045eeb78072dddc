"""The per-particle kernels' short quotients (reciprocal and residual correction)
against the divisions they fall back to outside 2^-100 .. 2^100: a problem whose
masses, densities, radiation constant, energies E and sources are scaled by a power
of two has the same solution scaled, bit for bit but for the quotients."""
import numpy as np
import pytest

from paper_2001_11606_gb300 import inputs as I
from paper_2001_11606_gb300 import sphrt

pytestmark = pytest.mark.gpu

TIGHT = dict(tol_krylov=1e-14, tol_outer_e=1e-12, tol_outer_E=1e-12, tol_inner_e=1e-14)


@pytest.mark.parametrize("make", [lambda: I.mms_2d(n=24, steps=2), lambda: I.mms_3d_lp(n=10, steps=2),
                                  lambda: I.mms_cgs(1, 60, steps=2)])
@pytest.mark.parametrize("power", [117, -117])
def test_scaled_problem_has_the_scaled_solution(make, power):
    w = make()
    k = 2.0 ** power
    P = w.particles
    got = []
    for s in (1.0, k):
        prm = dict(w.params, **TIGHT)
        prm["a"] = prm["a"] * s
        S = sphrt.Solver(sphrt.config_from_params(prm))
        S.set_particles(P.pos, P.mass * s, P.rho * s, P.h, P.sigma0, P.kind,
                        P.copy_of if np.any(P.kind == I.COPY) else None, w.e0, w.E0 * s)
        for n in (1, 2):
            Qe, QE, ge, gE = w.step_inputs(n)
            S.step(w.dt, Qe * s, QE * s, ge, gE * s)
        e, E, _ = S.get_energies()
        got.append((e, E / s))
    # a quotient is within an ulp of the division; a step takes ~10 of them per
    # particle, and both runs then iterate to 1e-14: far inside 1e-12
    for x, y in zip(*got):
        np.testing.assert_allclose(x, y, rtol=1e-12, atol=0)
