"""The neighbour search over its range of work items and cells: sets whose items are of
one, a few and the most particles (they grow with the particles per SM), and cells that
hold far more particles than one warp orders in shared memory; lists bit for bit as the
oracle's, cell lists alike."""
import numpy as np
import pytest

import oracle as O
from paper_2001_11606_gb300 import inputs as I
from paper_2001_11606_gb300 import sphrt

pytestmark = pytest.mark.gpu


def _cloud(dim, n, box, h, seed, clump=0.0):
    rng = np.random.default_rng(seed)
    pos = rng.uniform(0.0, box, (n, dim))
    pos[rng.random(n) < clump] *= 0.1  # into a tenth of every side
    kind = np.where(rng.random(n) < 0.1, I.DIRICHLET, I.INTERIOR).astype(np.int32)
    kind[0] = I.INTERIOR
    return I.Particles(dim=dim, dx=1.0, counts=(n,), pos=pos, kind=kind,
                       copy_of=np.full(n, -1, dtype=np.int64), mass=np.ones(n), rho=np.ones(n),
                       h=h * rng.uniform(0.8, 1.0, n), sigma0=np.ones(n))


def _check(P, cells, sample=None):
    e = np.ones(P.n)
    w = I.Workload("cloud", P, dict(dim=P.dim), 1e-3, 1, e0=e, E0=e.copy())
    S = sphrt.solver_for(w, cell_list=cells, precond=sphrt.PRECOND_JACOBI)
    rp, cols = S.get_neighbors()
    S.close()
    if sample is None:
        orp, ocols = O.neighbors(P.pos, P.h, P.kind)
        assert np.array_equal(rp, orp) and np.array_equal(cols, ocols)
        return
    rows = np.random.default_rng(1).choice(np.flatnonzero(P.kind == I.INTERIOR), sample, replace=False)
    orp, ocols = O.neighbors_of_rows(P.pos, P.h, rows)
    for k, i in enumerate(rows):
        assert np.array_equal(np.sort(cols[rp[i]:rp[i + 1]]), ocols[orp[k]:orp[k + 1]])


# 24 items of 16 particles an SM: 152 SMs have the longest items from 58,368 particles on
@pytest.mark.parametrize("n,box", [(900, 12.0), (9000, 26.0), (20000, 34.0), (90000, 56.0)])
@pytest.mark.parametrize("cells", [sphrt.CELLS_DENSE, sphrt.CELLS_SORTED])
def test_items_of_every_length(n, box, cells):
    _check(_cloud(3, n, box, 1.1, n), cells, 400)


# one cell of 255 .. 258 particles, of ~3,000; clumps among small cells
@pytest.mark.parametrize("dim,n,box,h,clump", [(2, 255, 1.0, 1.0, 0.0), (2, 256, 1.0, 1.0, 0.0),
                                               (2, 257, 1.0, 1.0, 0.0), (2, 258, 1.0, 1.0, 0.0),
                                               (3, 3000, 1.0, 0.6, 0.0), (1, 1500, 10.0, 2.0, 0.3),
                                               (3, 6000, 20.0, 1.0, 0.6), (2, 9000, 60.0, 1.0, 0.5)])
@pytest.mark.parametrize("cells", [sphrt.CELLS_DENSE, sphrt.CELLS_SORTED])
def test_cells_of_many_particles(dim, n, box, h, clump, cells):
    _check(_cloud(dim, n, box, h, n, clump), cells)
