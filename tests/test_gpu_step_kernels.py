"""The kernels that begin and end a step: totals, sources and boundary energy over
particle counts about a block's size, with Dirichlet and with copy ghosts, against
sums of the state that the step was given and returned."""
import numpy as np
import pytest

from paper_2001_11606_gb300 import inputs as I
from paper_2001_11606_gb300 import sphrt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make", [lambda: I.mms_2d(n=4, steps=2), lambda: I.mms_2d(n=16, steps=2),
                                  lambda: I.mms_2d(n=33, steps=2), lambda: I.mms_3d_lp(n=9, steps=2),
                                  lambda: I.mms_cgs(1, 257, steps=2)])
@pytest.mark.parametrize("graphs", [0, 1])
def test_step_energies_are_the_sums_of_the_states(make, graphs):
    w = make()
    P = w.particles
    inner = P.kind == I.INTERIOR
    m, V = P.mass[inner], (P.mass / P.rho)[inner]
    S = sphrt.solver_for(w, graphs=graphs)
    e, E = w.e0, w.E0
    for n in (1, 2):
        Qe, QE, ge, gE = w.step_inputs(n)
        bad = Qe.copy()
        bad[np.flatnonzero(inner)[-1]] = np.nan  # refused, and the state stays
        with pytest.raises(sphrt.SphRtError):
            S.step(w.dt, bad, QE, ge, gE)
        _, st = S.step(w.dt, Qe, QE, ge, gE)
        e1, E1, _ = S.get_energies()
        # sums of N positive terms in two orders: 2 (N + 2) eps relative at most
        tol = 2 * (m.size + 2) * np.finfo(float).eps
        before = np.sum(m * e[inner]) + np.sum(V * E[inner])
        after = np.sum(m * e1[inner]) + np.sum(V * E1[inner])
        terms = w.dt * V * (Qe + QE)[inner]
        assert st.energy_before == pytest.approx(before, rel=tol, abs=0)
        assert st.energy_after == pytest.approx(after, rel=tol, abs=0)
        assert abs(st.source_energy - terms.sum()) <= tol * np.abs(terms).sum()
        e, E = e1, E1
