"""Sliced finest level with dictionaries below, about and above the largest that is
staged in shared memory (43^3 rows; the dictionaries grow with the rows' reach): the
steps of every form run, and close the energy balance."""
import pytest

from paper_2001_11606_gb300 import inputs as I
from paper_2001_11606_gb300 import sphrt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("h", [2.3, 2.5, 2.6, 2.65, 2.7, 2.75, 2.8, 2.85, 2.9])
def test_every_form_steps(h):
    P = I.make_lattice(3, (43, 43, 43), 1.0 / 43, 4, h_over_dx=h)
    m = I.Manufactured(dim=3)
    e0, E0 = m.fields(P.pos, 0.0)
    prm = dict(dim=3, limiter=m.limiter, opacity_exp=float(m.p))
    w = I.Workload("mms", P, prm, 1e-3, 1, mms=m, e0=e0, E0=E0)
    ins = w.step_inputs(1)
    for over in (dict(fine_post_smooth=1), dict(fine_post_smooth=0), dict(precond=1), dict(precond=0),
                 dict(precision=1, fine_post_smooth=0), dict(precision=1, fine_post_smooth=1)):
        S = sphrt.solver_for(w, **over)
        _, st = S.step(w.dt, *ins)
        change = st.energy_after - st.energy_before
        # the solves stop at a relative residual of 1e-8 or less
        assert abs(change - st.source_energy - st.boundary_energy) < 1e-7 * st.energy_before
        S.close()
