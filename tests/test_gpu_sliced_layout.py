"""Which layout a particle set runs in, where results alone do not tell: the sets that
the sliced tests rely on are sliced, those beyond the dictionary's cap are not; A P rows
of more entries than shared memory holds; hierarchies rebuilt under a captured graph."""
import numpy as np
import pytest

from paper_2001_11606_gb300 import inputs as I
from paper_2001_11606_gb300 import sphrt
from test_gpu_sliced import _mms, _problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TIGHT = dict(tol_krylov=1e-14, tol_outer_e=1e-12, tol_outer_E=1e-12, tol_inner_e=1e-14)


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def _column_bytes(w, **over):
    """Bytes per stored column of the CG's product sweep: 2 in slices, 4 in CSR rows."""
    S = sphrt.solver_for(w, kernel_timing=1, precond=0, **over)
    S.step(w.dt, *w.step_inputs(1), raise_on_error=False)
    launches, _, by = S.kernel_stats_by_kind()["spmv_pq"]
    n_int, _, nnz = S.sizes()
    S.close()
    return round((by / launches - 56.0 * n_int) / nnz - 8.0)


@pytest.mark.skipif("_sms() > 152", reason="sized for 152 SMs")
@pytest.mark.parametrize("name,want", [("2d", 2), ("3d", 2), ("reflect", 2), ("periodic", 2),
                                       ("wide", 4)])
@pytest.mark.parametrize("precision", [0, 1])
def test_layout_of_the_sliced_tests(name, want, precision):
    assert _column_bytes(_problem(name), precision=precision) == want


@pytest.mark.skipif("_sms() > 152", reason="sized for 152 SMs")
def test_dictionaries_cross_the_cap_once():
    got = [_column_bytes(_mms((43, 43, 43), h=h)) for h in (2.3, 2.5, 2.6, 2.65, 2.7, 2.75, 2.8, 2.85, 2.9)]
    assert got[0] == 2 and got[-1] == 4 and got == sorted(got)


def test_slices_start_at_512_rows_per_sm():
    rows = 512 * _sms()
    n = int(rows ** 0.5)
    for counts in ((n, n), (n, rows // n + 1)):  # just below, just above
        assert _column_bytes(_mms(counts)) == (2 if counts[0] * counts[1] >= rows else 4)


# Particles in pairs a tenth of a spacing apart, ~430 neighbours each: with a strength
# threshold between the pairs' coupling and the next one the aggregates are the pairs, and
# rows of A P have more than the 100 (FP64) and 200 (FP32) entries that shared memory holds
# at once: they are summed in windows.
def _pairs(n, h=2.34):
    P = I.make_lattice(3, (n,) * 3, 1.0 / n, 4, h_over_dx=h, jitter=0.0)
    odd = np.round(P.pos[:, 0] * n - 0.5).astype(int) % 2
    P.pos[:, 0] += np.where(odd, -0.45, 0.45) / n
    m = I.Manufactured(dim=3)
    e0, E0 = m.fields(P.pos, 0.0)
    # dt ~ dx^2: the couplings' share of the diagonal is that of every n
    return I.Workload("pairs", P, dict(dim=3), 0.25 / n ** 2, 1, mms=m, e0=e0, E0=E0)


def _pair_threshold():
    w = _pairs(16)
    S = sphrt.solver_for(w, precond=0)
    S.step(w.dt, *w.step_inputs(1), raise_on_error=False)
    rp, cols, vals, diag, _ = S.get_operator()
    S.close()
    i = np.argmin(np.sum((w.particles.pos - 0.5) ** 2, 1))
    k = slice(rp[i], rp[i + 1])
    c = np.sort(np.abs(vals[k]) / np.sqrt(diag[i] * diag[cols[k]]))
    assert c[-1] > 1.2 * c[-2]
    return 0.5 * (c[-1] + c[-2]), c.size


@pytest.mark.parametrize("precision,most", [(0, 100), (1, 200)])
def test_ap_rows_beyond_shared_memory(precision, most):
    n = int(np.ceil((512 * _sms()) ** (1.0 / 3.0) / 2.0)) * 2
    w = _pairs(n)
    assert _column_bytes(w) == 2
    ins = w.step_inputs(1)
    theta, entries = _pair_threshold()
    assert entries // 2 > most
    got = []
    for over in (dict(precond=0), dict(precision=precision, amg_theta=theta)):
        S = sphrt.solver_for(w, **dict(TIGHT, **over))
        S.step(w.dt, *ins)
        got.append(S.get_energies())
        n_int = S.sizes()[0]
        info = S.amg_info() if over.get("precond") != 0 else []
        S.close()
    assert len(info) > 1 and info[1][0] > 0.49 * n_int  # pairs
    m = w.particles.kind == I.INTERIOR
    tol = 1e-8 if precision else 1e-10  # the parity tests' tolerances
    for a, b in zip(got[0][:2], got[1][:2]):
        assert np.max(np.abs(a[m] - b[m]) / a[m]) < tol


# every step frees the hierarchy's buffers and takes them again
@pytest.mark.parametrize("over", [dict(), dict(fine_post_smooth=0), dict(precision=1),
                                  dict(precision=1, fine_post_smooth=0), dict(cheb_degree=2)])
def test_rebuilt_hierarchies_under_a_captured_graph(over):
    n = int(np.ceil((512 * _sms()) ** 0.5))
    P = I.make_lattice(2, (n, n), 1.0 / n, 4)
    m = I.Manufactured(dim=2, p=-3.0, limiter=1)
    e0, E0 = m.fields(P.pos, 0.0)
    w = I.Workload("mms", P, dict(dim=2, limiter=1, opacity_exp=-3.0), 1e-3, 5, mms=m, e0=e0, E0=E0)
    out = []
    for graphs in (0, 1):
        S = sphrt.solver_for(w, amg_rebuild=1, graphs=graphs, **over)
        for k in range(1, 6):
            S.step(w.dt, *w.step_inputs(k))
        out.append(S.get_energies())
        S.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
