"""The operator's entries bit for bit: B is symmetric to the last bit whatever the
smoothing lengths."""
import numpy as np
import pytest

from paper_2001_11606_gb300 import inputs as I
from paper_2001_11606_gb300 import sphrt

pytestmark = pytest.mark.gpu


def _cloud(dim, n, box, h, seed=3):
    rng = np.random.default_rng(seed)
    pos = rng.uniform(0.0, box, (n, dim))
    kind = np.zeros(n, dtype=np.int32)
    return I.Particles(dim=dim, dx=1.0, counts=(n,), pos=pos, kind=kind,
                       copy_of=np.full(n, -1, dtype=np.int64), mass=np.full(n, 0.8),
                       rho=np.ones(n), h=h(rng, n), sigma0=np.ones(n))


def _entries(P, kern, dt=1e-3, **over):
    e = np.full(P.n, 0.7)
    w = I.Workload("cloud", P, dict(dim=P.dim, kernel=kern), dt, 1, e0=e, E0=e ** 4)
    S = sphrt.solver_for(w, precond=sphrt.PRECOND_JACOBI, **over)
    S.step(dt, raise_on_error=False)  # near coincident points: the solve need not converge
    rp, cols, vals, _, _ = S.get_operator()
    S.close()
    rows = np.repeat(np.arange(P.n), np.diff(rp))
    order = np.lexsort((cols, rows))
    return rows[order], cols[order], vals[order]  # B_ij / V_i, and all V are equal


def _spread(rng, n):
    return rng.uniform(0.7, 1.3, n)


def _adjacent(rng, n):  # neighbouring doubles, of which many share one 1 / h
    h = np.full(n, 1.9)
    for _ in range(4):
        h = np.where(rng.random(n) < 0.5, np.nextafter(h, 2.0), h)
    return h


@pytest.mark.parametrize("dim,n,box", [(1, 300, 40.0), (2, 400, 14.0), (3, 500, 7.0)])
@pytest.mark.parametrize("h", [_spread, _adjacent])
@pytest.mark.parametrize("kern", [0, 1])
def test_operator_is_symmetric_to_the_last_bit(dim, n, box, h, kern):
    rows, cols, vals = _entries(_cloud(dim, n, box, h), kern)
    t = np.lexsort((rows, cols))  # the transposed entries in the same order
    assert np.array_equal(rows, cols[t]) and np.array_equal(cols, rows[t])
    assert vals.size > n and np.array_equal(vals, vals[t])
