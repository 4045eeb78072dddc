"""The next level's sparsity from the rows of A P: coarse rows of a few columns, and of
more than the warp kernel's 512 (the block kernel takes over), each in a solve against
the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_2001_11606_gb300 import inputs as I
from paper_2001_11606_gb300 import sphrt

pytestmark = pytest.mark.gpu

TIGHT = dict(tol_krylov=1e-14, tol_outer_e=1e-12, tol_outer_E=1e-12, tol_inner_e=1e-14)


def _workload(n, h):
    P = I.make_lattice(3, (n,) * 3, 1.0 / n, 4, h_over_dx=h)
    m = I.Manufactured(dim=3)
    e0, E0 = m.fields(P.pos, 0.0)
    return I.Workload("dense", P, dict(dim=3), 0.1, 1, mms=m, e0=e0, E0=E0)


# h = 4.5 spacings: ~1,600 entries a row; the strength threshold sets how small the
# aggregates are, hence how many coarse columns a coarse row has
@pytest.mark.parametrize("n,h,thetas,wide", [(20, 1.5, (0.02,), False),
                                             (18, 4.5, (2.1e-3, 2.2e-3, 2.3e-3, 2.4e-3, 2.5e-3),
                                              True)])
@pytest.mark.parametrize("precision", [0, 1])
def test_coarse_rows_of_any_width(n, h, thetas, wide, precision):
    w = _workload(n, h)
    pb = O.Problem(w.particles, dict(w.params, **TIGHT))
    ins = w.step_inputs(1)
    rc, e, E, _ = pb.step(w.e0, w.E0, w.dt, *ins)
    assert rc == 0
    m = w.particles.kind == I.INTERIOR
    found = False
    for theta in thetas:
        S = sphrt.solver_for(w, **dict(TIGHT, amg_theta=theta, precision=precision))
        S.step(w.dt, *ins)
        info = S.amg_info()
        assert info[0][1] > 600000  # a level that has A P
        found = found or (len(info) > 1 and (not wide or info[1][1] > 512 * info[1][0]))
        eg, Eg, _ = S.get_energies()
        # the parity tests' tolerances
        tol = 1e-8 if precision else 1e-10
        assert np.max(np.abs(eg[m] - e[m]) / e[m]) < tol
        assert np.max(np.abs(Eg[m] - E[m]) / E[m]) < tol
    assert found
