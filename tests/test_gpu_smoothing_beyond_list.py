"""Smoothing lengths of supports that hold many times what the list of distances does:
the candidates then pass through the list in several loads, against the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_2001_11606_gb300 import inputs as I
from paper_2001_11606_gb300 import sphrt

pytestmark = pytest.mark.gpu


# ~450 points of the support (about the list's 448), ~1,400 and ~2,800 in 3-D; 2-D; all
# points in few cells
@pytest.mark.parametrize("dim,n,kern,h0,eta", [(3, 8, 1, 4.8, 4.75), (3, 8, 0, 2.4, 4.75),
                                               (3, 10, 1, 6.5, 7.0), (3, 10, 0, 4.6, 8.8),
                                               (2, 30, 1, 14.0, 14.0), (3, 6, 1, 9.0, 8.0)])
def test_lengths_match_oracle_beyond_the_list(dim, n, kern, h0, eta):
    P = I.make_lattice(dim, (n,) * dim, 0.37, seed=13, h_over_dx=h0, support=1.0 if kern else 2.0)
    e = np.ones(P.n)
    w = I.Workload("lat", P, dict(dim=dim, kernel=kern), 1e-3, 1, e0=e, E0=e.copy())
    h_o, it_o = O.smoothing_lengths(P, w.params, eta=eta, tol=1e-12)
    S = sphrt.solver_for(w)
    it = S.adapt_smoothing_lengths(eta=eta, tol=1e-12)
    # both stop at |dh| <= 1e-12 h of a contraction: their ends differ by a few times
    # that at most
    np.testing.assert_allclose(S.get_smoothing_lengths(), h_o, rtol=1e-11, atol=0)
    assert abs(it - it_o) <= 1
    S.close()
