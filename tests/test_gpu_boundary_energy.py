"""The energy that crosses the boundary in a step, summed pair by pair from the state
the step returned: Dirichlet couplings on every row, on few rows and on none."""
import numpy as np
import pytest

import oracle as O
from paper_2001_11606_gb300 import inputs as I
from paper_2001_11606_gb300 import sphrt

pytestmark = pytest.mark.gpu


# 4^2: every row has couplings; 24^2 with ghosts on all sides: a band of rows; one side
# only; none
@pytest.mark.parametrize("dim,n,faces", [(2, 4, None), (2, 24, None), (3, 7, None),
                                         (2, 24, [("dirichlet", "reflect"), ("reflect",) * 2]),
                                         (2, 24, [("reflect",) * 2] * 2)])
@pytest.mark.parametrize("limiter", [0, 1])
@pytest.mark.parametrize("graphs", [0, 1])
def test_boundary_energy_is_the_sum_over_the_couplings(dim, n, faces, limiter, graphs):
    P = I.make_lattice(dim, (n,) * dim, 1.0 / n, 7, faces=faces)
    rng = np.random.default_rng(4)
    e0 = 1.0 + 0.2 * np.sin(5.0 * P.pos[:, 0])
    E0 = e0 ** 4
    w = I.Workload("bnd", P, dict(dim=dim, limiter=limiter), 1e-3, 1, e0=e0, E0=E0)
    S = sphrt.solver_for(w, graphs=graphs)
    ge, gE = rng.uniform(0.8, 1.2, P.n), rng.uniform(0.5, 2.0, P.n)
    _, st = S.step(w.dt, None, None, ge, gE)
    D = S.get_properties()["D"]
    _, E, _ = S.get_energies()
    V = P.mass / P.rho
    rp, cols = O.neighbors(P.pos, P.h, P.kind)
    terms = [0.0]
    for i in np.flatnonzero(P.kind == I.INTERIOR):
        for j in cols[rp[i]:rp[i + 1]]:
            if P.kind[j] != I.DIRICHLET:
                continue
            r = np.sqrt(np.sum((P.pos[i] - P.pos[j]) ** 2))
            F = 0.5 * sum(O.kernel(dim, r, hh, 0)[1] for hh in (P.h[i], P.h[j])) / r
            terms.append(-w.dt * V[i] * V[j] * F * (D[i] + D[j]) * (gE[j] - E[i]))
    terms = np.array(terms)
    # a term takes ~30 roundings (its E_j - E_i is one of them), their sum one per term
    tol = (60 + terms.size) * 2.0 ** -53 * np.abs(terms).sum()
    assert abs(st.boundary_energy - terms.sum()) <= tol
    assert (terms.size == 1) == (not np.any(P.kind == I.DIRICHLET))
    S.close()
