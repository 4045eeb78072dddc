"""The sliced finest level (from 77,824 particles on 152 SMs) against the oracle:
operator entries, and steps with every preconditioner, both arithmetic forms, both
V-cycles, copy ghosts, a last group that is nearly empty, and a set whose
dictionaries are too large (it stays in CSR rows)."""
import numpy as np
import pytest

import oracle as O
from paper_2001_11606_gb300 import inputs as I
from paper_2001_11606_gb300 import sphrt

pytestmark = pytest.mark.gpu

TIGHT = dict(tol_krylov=1e-14, tol_outer_e=1e-12, tol_outer_E=1e-12, tol_inner_e=1e-14)


def _mms(counts, h=1.5, **kw):
    P = I.make_lattice(len(counts), counts, 1.0 / max(counts), 4, h_over_dx=h)
    m = I.Manufactured(dim=len(counts), **kw)
    e0, E0 = m.fields(P.pos, 0.0)
    prm = dict(dim=len(counts), limiter=m.limiter, opacity_exp=float(m.p))
    return I.Workload("mms", P, prm, 1e-3, 2, mms=m, e0=e0, E0=E0)


def _problem(name):
    if name == "2d":        # 77,841 rows: the last of 305 groups holds 17
        return _mms((279, 279))
    if name == "3d":        # 79,464 rows, temperature-dependent opacity and limiter
        return _mms((44, 43, 42), p=-3.0, limiter=1)
    if name == "reflect":   # copy ghosts fold onto interior columns
        w = I.heating_wave(2, 78400, 5.0, seed=9, steps=2)
        w.params["max_outer"] = 200
        return w
    if name == "periodic":  # the same with energies of one magnitude
        return I.mms_cgs(2, 280)
    return _mms((43, 43, 43), h=2.9)  # ~800 neighbours: dictionaries beyond the cap


CASES = [("2d", dict(precond=0)), ("2d", dict(precond=1, cheb_degree=3)), ("2d", dict()),
         ("2d", dict(precision=1)), ("2d", dict(cheb_degree=2)), ("3d", dict(fine_post_smooth=0)),
         ("3d", dict(precision=1, fine_post_smooth=0, reliable_drop=1e-6)),
         ("3d", dict(graphs=0, amg_rebuild=1)), ("periodic", dict()),
         ("periodic", dict(precision=1, precond=1)), ("wide", dict(precond=0))]
_done = {}


def _oracle(name):
    if name not in _done:
        w = _problem(name)
        pb = O.Problem(w.particles, dict(w.params, **TIGHT))
        e, E = w.e0.copy(), w.E0.copy()
        for n in (1, 2):
            rc, e, E, _ = pb.step(e, E, w.dt, *w.step_inputs(n))
            assert rc == 0
        _done[name] = (w, pb, e, E)
    return _done[name]


@pytest.mark.parametrize("name,over", CASES)
def test_steps_match_oracle(name, over):
    w, pb, e, E = _oracle(name)
    S = sphrt.solver_for(w, **dict(TIGHT, **over))
    for n in (1, 2):
        S.step(w.dt, *w.step_inputs(n))
    eg, Eg, _ = S.get_energies()
    m = w.particles.kind == I.INTERIOR
    # the tolerances of the parity tests: both sides iterate to the same fixed point
    tol = 1e-8 if over.get("precision") else 1e-10
    assert np.max(np.abs(eg[m] - e[m]) / np.abs(e[m])) < tol
    assert np.max(np.abs(Eg[m] - E[m]) / np.abs(E[m])) < tol


@pytest.mark.parametrize("name", ["2d", "3d", "reflect"])
def test_operator_in_row_order(name):
    w = _problem(name)
    S = sphrt.solver_for(w, precond=0, **TIGHT)
    ins = w.step_inputs(1)
    S.step(w.dt, *ins)
    rp, cols, vals, diag, gb = S.get_operator()
    pb = O.Problem(w.particles, w.params)
    props = pb.properties(w.e0, w.E0, w.dt)
    Eg = np.where(w.particles.kind == I.DIRICHLET, ins[3], w.E0)
    arow, acol, aval, adiag, agb = pb.assemble(props, w.dt, Eg)
    n = w.particles.n
    rows = np.repeat(np.arange(n), np.diff(rp))
    orows = np.repeat(np.arange(n), np.diff(arow))
    sparse = pytest.importorskip("scipy.sparse")  # sums duplicate columns of copy ghosts
    A = sparse.csr_matrix((vals, (rows, cols)), shape=(n, n))
    B = sparse.csr_matrix((aval, (orows, acol)), shape=(n, n))
    big = np.abs(adiag).max()
    # entries: ~30 roundings each; diagonals: sums of ~100 of them
    assert np.abs(A - B).max() <= 1e-13 * np.abs(B).max()
    assert np.max(np.abs(diag - adiag)) <= 1e-13 * big
    assert np.max(np.abs(gb - agb)) <= 1e-13 * max(np.abs(agb).max(), 1e-300)
