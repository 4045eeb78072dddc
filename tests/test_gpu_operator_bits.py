"""The operator's entries bit for bit and at the ends of their range: B is symmetric
to the last bit whatever the smoothing lengths, and particle sets shrunk by a power of
two have the shrunk operator, also where r^2 is no normal FP32 number."""
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


# lengths of 2^-68 leave r^2 ~ 13 bits as an FP32 number, of 2^-80 none; those of 2^68
# overflow FP32's range
@pytest.mark.parametrize("power", [-80, -68, -60, 60, 68])
@pytest.mark.parametrize("kern", [0, 1])
def test_scaled_lengths_scale_the_operator(power, kern):
    P = _cloud(3, 500, 7.0, _spread)
    want = _entries(P, kern)
    s = 2.0 ** power
    Q = I.Particles(dim=3, dx=s, counts=P.counts, pos=P.pos * s, kind=P.kind, copy_of=P.copy_of,
                    mass=P.mass * s ** 3, rho=P.rho, h=P.h * s, sigma0=P.sigma0)
    # V_j F ~ s^-2; dt by s^2 keeps the diagonals in step
    got = _entries(Q, kern, dt=1e-3 * s * s)
    assert np.array_equal(want[0], got[0]) and np.array_equal(want[1], got[1])
    # an entry takes ~30 roundings, and a power of two scales exactly
    assert np.max(np.abs(got[2] * s * s - want[2]) / np.abs(want[2]).max()) <= 60 * 2.0 ** -53
