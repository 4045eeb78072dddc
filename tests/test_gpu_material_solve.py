"""The last Newton iteration of the material solve against extended precision.  Loose
tolerances end the solve after its first iteration and the step after its first outer
iteration, so that no later iteration hides the first one's rounding."""
import numpy as np
import pytest

from paper_2001_11606_gb300 import inputs as I
from paper_2001_11606_gb300 import sphrt

pytestmark = pytest.mark.gpu

LOOSE = dict(tol_outer_e=1e9, tol_outer_E=1e9, tol_inner_e=1e9, krylov_start=0)


# Without emission (a = 0) the iteration from any e is e - (r (e - e_old) - P) / r with
# r = rho / dt and P = c sigma E: from a cold e_old = 0 the second one ends at P / r,
# having moved by de.  Its roundings: P, u (relative to u = r de), the quotient and the
# new e: 2^-53 (2 |de| + 2 |e|).  dt = 8: E falls to a ninth, so that |de| ~ 8 |e|; dt =
# 0.003: |de| << |e|, and r's own rounding shows.
@pytest.mark.parametrize("batch", [False, True])
@pytest.mark.parametrize("dim,n", [(2, 40), (3, 12)])
@pytest.mark.parametrize("dt", [8.0, 0.003])
def test_last_iteration_has_full_precision(batch, dim, n, dt):
    P = I.make_lattice(dim, (n,) * dim, 1.0 / n, 5)
    rng = np.random.default_rng(8)
    P.rho = rng.uniform(0.5, 1.5, P.n)
    e0, E0 = np.zeros(P.n), rng.uniform(1.0, 3.0, P.n)
    if batch:
        B = sphrt.Batch(sphrt.default_config(dim=dim, a=0.0, **LOOSE))
        k = B.add(P, e0, E0)
        B.step(dt)
        e, E = B.get_energies(k)
        B.close()
        r = P.rho / dt
    else:
        w = I.Workload("one", P, dict(dim=dim, a=0.0), dt, 1, e0=e0, E0=E0)
        S = sphrt.solver_for(w, **LOOSE)
        _, st = S.step(dt)
        assert st.outer_iters == 1 and st.newton_iters_max == 1
        e, E, _ = S.get_energies()
        S.close()
        r = P.rho * (1.0 / dt)
    m = P.kind == I.INTERIOR
    L = np.longdouble
    want = E.astype(L) / r.astype(L)
    de = np.abs(want - E0.astype(L) / r.astype(L))
    bound = L(2.0) ** -53 * (2 * de + 2 * np.abs(want))
    assert np.max((np.abs(e - want) / bound)[m]) <= 1.0
