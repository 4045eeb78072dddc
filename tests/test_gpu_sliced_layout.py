"""Sliced operators whose hierarchies are rebuilt under a captured graph."""
import numpy as np
import pytest

from paper_2001_11606_gb300 import inputs as I
from paper_2001_11606_gb300 import sphrt

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


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
