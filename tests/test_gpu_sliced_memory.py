"""The sliced layout where memory is short: whichever allocation of the first step
fails, the step falls back to CSR rows, holds nothing more than a set that was in CSR
rows from the start, and stays there; results are those of that layout, bit for bit."""
import ctypes as C

import numpy as np
import pytest

from paper_2001_11606_gb300 import inputs as I
from paper_2001_11606_gb300 import sphrt

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _workload():
    # the sliced layout starts at 512 rows per SM
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = int(np.ceil(np.sqrt(512 * sms)))
    P = I.make_lattice(2, (n, n), 1.0 / n, 4)
    m = I.Manufactured(dim=2)
    e0, E0 = m.fields(P.pos, 0.0)
    return I.Workload("mms", P, dict(dim=2, tol_krylov=1e-13), 1e-3, 3, mms=m, e0=e0, E0=E0)


def _hook(S, fail_after=-1, refuse_ap=0):
    fn = sphrt.load().sph_rt_test_hook
    fn.restype, fn.argtypes = C.c_int64, [C.c_void_p, C.c_int64, C.c_int32]
    return fn(S._h, fail_after, refuse_ap)


def _column_bytes(S, w):
    """Bytes per stored column of the CG's product sweep: 2 in slices, 4 in CSR rows."""
    launches, _, by = S.kernel_stats_by_kind()["spmv_pq"]
    if launches == 0:  # the CG takes its product from the V-cycle
        return None
    n_int, _, nnz = S.sizes()
    return round((by / launches - 56.0 * n_int) / nnz - 8.0)


@pytest.fixture(scope="module")
def case():
    w = _workload()
    return w, [w.step_inputs(k) for k in (1, 2, 3)]


def _run(case, fail_after=-1, refuse_ap=0, steps=3, **over):
    w, ins = case
    S = sphrt.solver_for(w, kernel_timing=1, **over)
    before = _hook(S, fail_after, refuse_ap)
    out, held = [], []
    for k in range(steps):
        S.step(w.dt, *ins[k])
        out.append(_column_bytes(S, w))
        # the hook's own call ends the countdown: what it did not reach stays alive
        held.append(_hook(S, -1, refuse_ap) - before)
    e, E, _ = S.get_energies()
    S.close()
    return out, held, e, E


def _same(a, b):
    return np.array_equal(a[2], b[2]) and np.array_equal(a[3], b[3])


@pytest.mark.parametrize("over", [dict(precond=0), dict(precond=0, precision=1), dict(),
                                  dict(precision=1)])
def test_any_failed_allocation_falls_back(case, over):
    sliced = _run(case, **over)
    csr = _run(case, fail_after=0, **over)
    assert sliced[0] == [2, 2, 2] and csr[0] == [4, 4, 4]
    seen = set()
    last = 24 if "precond" in over else 150  # past the layout's, or into the AMG set-up's
    for k in range(0, last, 1 if last < 30 else 7):
        got = _run(case, fail_after=k, **over)
        seen.add(got[0][0])
        assert len(set(got[0])) == 1  # the layout of the first step is kept
        assert _same(got, csr if got[0][0] == 4 else sliced)
        assert got[1] == (csr if got[0][0] == 4 else sliced)[1], k
    assert 4 in seen and seen <= {2, 4}


@pytest.mark.parametrize("over", [dict(), dict(precision=1), dict(precision=1, fine_post_smooth=0),
                                  dict(amg_rebuild=1)])
def test_refused_slices_of_ap_take_the_operator_back(case, over):
    csr = _run(case, fail_after=0, **over)
    got = _run(case, refuse_ap=1, **over)
    assert got[0] == csr[0] and _same(got, csr)


def test_operator_read_back_needs_no_device_memory(case):
    w, ins = case
    S = sphrt.solver_for(w, precond=0)
    S.step(w.dt, *ins[0])
    want = S.get_operator()
    _hook(S, 0)
    got = S.get_operator()
    assert all(np.array_equal(a, b) for a, b in zip(want, got))
    S.close()


def test_a_new_set_chooses_again(case):
    w, ins = case
    S = sphrt.solver_for(w, precond=0, kernel_timing=1)
    _hook(S, 0)
    S.step(w.dt, *ins[0])
    assert _column_bytes(S, w) == 4
    S.move_particles(w.particles.pos)
    S.kernel_stats(reset=True)
    S.step(w.dt, *ins[1])
    assert _column_bytes(S, w) == 2
    S.close()
