"""The cell-wise neighbour search at the edges of its work items: cells of one
particle, of exactly and one more than an item's 16, of several items, candidate
counts around multiples of 32, lists with copy ghosts of the row itself; both cell
lists, against the oracle's all-pairs lists (bit for bit) and operator."""
import numpy as np
import pytest

import oracle as O
from paper_2001_11606_gb300 import inputs as I
from paper_2001_11606_gb300 import sphrt

pytestmark = pytest.mark.gpu


def _cloud(dim, n, box, h, seed, spread):
    rng = np.random.default_rng(seed)
    pos = rng.uniform(0.0, box, (n, dim))
    kind = np.zeros(n, dtype=np.int32)
    kind[rng.random(n) < 0.2] = I.DIRICHLET
    kind[0] = I.INTERIOR
    copy = rng.random(n) < 0.15
    copy[0] = False
    kind[copy] = I.COPY
    inner = np.flatnonzero(kind == I.INTERIOR)
    copy_of = np.full(n, -1, dtype=np.int64)
    copy_of[copy] = rng.choice(inner, int(copy.sum()))
    m = rng.uniform(0.5, 1.5, n)
    return I.Particles(dim=dim, dx=1.0, counts=(n,), pos=pos, kind=kind, copy_of=copy_of, mass=m,
                       rho=np.ones(n), h=h * rng.uniform(1.0 - spread, 1.0, n),
                       sigma0=np.ones(n))


# (dim, particles, box, h): one particle a cell; ~16 and ~33 a cell; one cell in all;
# unequal smoothing lengths
@pytest.mark.parametrize("dim,n,box,h,spread", [(3, 300, 9.0, 0.5, 0.0), (3, 430, 6.0, 1.0, 0.3),
                                                (2, 530, 8.0, 1.0, 0.0), (2, 97, 1.0, 2.0, 0.5),
                                                (1, 333, 20.0, 1.0, 0.4), (3, 1, 1.0, 1.0, 0.0)])
@pytest.mark.parametrize("kern", [0, 1])
@pytest.mark.parametrize("cells", [sphrt.CELLS_DENSE, sphrt.CELLS_SORTED])
def test_lists_and_operator_match_oracle(dim, n, box, h, spread, kern, cells):
    P = _cloud(dim, n, box, h, 5 + n, spread)
    e = np.full(n, 0.7)
    prm = dict(dim=dim, kernel=kern)
    w = I.Workload("cloud", P, prm, 1e-3, 1, e0=e, E0=e ** 4)
    S = sphrt.solver_for(w, cell_list=cells, precond=sphrt.PRECOND_JACOBI)
    rp, cols = S.get_neighbors()
    orp, ocols = O.neighbors(P.pos, P.h, P.kind, kernel=kern)
    assert np.array_equal(rp, orp) and np.array_equal(cols, ocols.astype(np.int64))
    S.step(1e-3)
    rp, cols, vals, diag, gb = S.get_operator()
    # row sums of the couplings from the oracle's kernel, pair by pair.  A weight takes
    # ~25 roundings; near coincident points 1/r magnifies none of them (relative errors
    # only), so 1e-13 of the row's absolute sum covers a row of a few hundred.
    V = P.mass / P.rho
    D = S.get_properties()["D"]
    want_gb, want = np.zeros(n), np.zeros((n, n))
    for i in np.flatnonzero(P.kind == I.INTERIOR):
        for j in ocols[orp[i]:orp[i + 1]]:
            r = np.sqrt(np.sum((P.pos[i] - P.pos[j]) ** 2))
            F = 0.5 * sum(O.kernel(dim, r, hh, kern)[1] for hh in (P.h[i], P.h[j])) / r
            wij = -V[j] * (D[i] + D[j]) * F
            if P.kind[j] == I.DIRICHLET:
                want_gb[i] += wij * e[j] ** 4
            else:
                c = j if P.kind[j] == I.INTERIOR else P.copy_of[j]
                if c != i:
                    want[i, c] -= wij
    got = np.zeros((n, n))
    np.add.at(got, (np.repeat(np.arange(n), np.diff(rp)), cols), vals)
    scale = np.abs(want).sum(1).max() + 1e-300
    assert np.max(np.abs(got - want)) <= 1e-13 * scale
    assert np.max(np.abs(gb - want_gb)) <= 1e-13 * (np.abs(want_gb).max() + 1e-300)
