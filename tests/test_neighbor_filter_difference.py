"""CPU check of the neighbour search's FP32 filter in the form that the cell-wise search
runs (neighbors.cu, neighbor_kernel): d = r^2 - cut in FP32, a hit where d < -band, no hit
where d > band, and the exact FP64 predicate in between and where d is no number."""
import numpy as np
import pytest

from paper_2001_11606_gb300 import inputs as I

BAND = 3e-5  # kNbrBand


def _check(P, rows=300, seed=0):
    n, dim = P.pos.shape
    p3 = np.zeros((n, 3))
    p3[:, :dim] = P.pos
    lo = p3.min(axis=0)
    cell = 2.0 * P.h.max() * (1.0 + 1e-9)
    nc = [(int((p3[:, d].max() - lo[d]) / cell) + 1) if d < dim else 1 for d in range(3)]
    c = np.clip(np.floor((p3 - lo) * (1.0 / cell)).astype(np.int64), 0, np.array(nc) - 1)
    f32 = np.float32
    with np.errstate(over="ignore", under="ignore", invalid="ignore"):
        rel = (p3 - (lo + c * cell)).astype(f32)
        rel[:, dim:] = 0.0
        w = ((2.0 * P.h) * (2.0 * P.h)).astype(f32)
        cellf = f32(cell)
        band = f32(BAND) * cellf * cellf
        pick = np.flatnonzero(P.kind == 0)
        pick = np.random.default_rng(seed).choice(pick, min(rows, pick.size), replace=False)
        decided = 0
        for i in pick:
            o = c - c[i]
            near = np.all(np.abs(o) <= 1, axis=1)
            near[i] = False
            js = np.flatnonzero(near)
            d = (rel[i] - rel[js]) + (-o[js].astype(f32) * cellf)
            d = ((d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]) + d[:, 2] * d[:, 2]) - np.maximum(w[i], w[js])
            assert d.dtype == f32
            dx = p3[i] - p3[js]
            cut = 2.0 * np.maximum(P.h[i], P.h[js])
            exact = dx[:, 0] * dx[:, 0] + dx[:, 1] * dx[:, 1] + dx[:, 2] * dx[:, 2] < cut * cut
            sure = np.abs(d) > band
            assert np.array_equal((d < -band)[sure], exact[sure])
            decided += np.count_nonzero(sure) / max(js.size, 1)
    return decided / pick.size


@pytest.mark.parametrize("make", [
    lambda: I.mms_3d_lp(n=24).particles,
    lambda: I.mms_2d(n=48).particles,
    lambda: I.heating_wave(3, 3000, 5.0, seed=9).particles,
    lambda: I.make_lattice(3, (9, 7, 5), 1.0 / 64, seed=0, jitter=0.0),
])
def test_difference_form_decides_as_the_exact_predicate(make):
    assert _check(make()) > 0.95


# lengths whose squares overflow or leave FP32: every pair takes the exact predicate, or
# is decided alike
@pytest.mark.parametrize("power", [-90, -66, -60, 60, 70])
def test_difference_form_at_the_ends_of_fp32(power):
    P = I.mms_3d_lp(n=10).particles
    P.h = P.h * np.random.default_rng(4).uniform(0.7, 1.3, P.n)
    P.pos, P.h = P.pos * 2.0 ** power, P.h * 2.0 ** power
    _check(P, rows=60)
