"""GPU: the passes carry only the modes that a bin or shell holds.  Plans whose
bins end at a k_x tile's edge, one mode inside or past it, at the Nyquist
frequency and in the cube's corner give the leading bins of a plan that bins
every mode."""
import math

import numpy as np
import pytest

import mockgen
from tests.helpers import to_device

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("N", [64, 60])
def test_leading_bins_do_not_depend_on_the_last(N):
    """Bins centred on integer |n|: with nb bins the passes reach |n| < nb +
    1/2.  The bins' fixed-point sums are rounded at 2^-49 of a bound (at most
    155 of the largest mode power) of each k-space tile, at most 2 N 8 runs of
    them per tile: 1e-9 of the largest bin's power bounds the difference."""
    import paper_1506_02729_gb300 as fkp
    sv = mockgen.survey_small(N=N, assign=2)
    gal, ran = mockgen.catalog(sv, 3)
    g, r = to_device(gal), to_device(ran)
    geom = dict(sv.geometry(), periodic=True)
    kf = 2 * math.pi / sv.L
    full = int(math.ceil(math.sqrt(3) * N / 2))
    ref = fkp.Plan(geom, (0.5 * kf, kf, full)).power(g, r)
    scale = np.nanmax(ref["mono_raw"])
    for nb in (1, 2, 7, 8, 9, N // 2 - 1, N // 2, N // 2 + 1, full - 1):
        got = fkp.Plan(geom, (0.5 * kf, kf, nb)).power(g, r)
        assert np.array_equal(got["nmodes"], ref["nmodes"][:nb]), nb
        for k in ("P0", "P2", "P4", "P4b"):
            assert np.nanmax(np.abs(got[k] - ref[k][:nb])) <= 1e-9 * scale, (nb, k)


def test_bins_that_hold_no_mode(N=64):
    """Bins below the fundamental mode: no modes, no values, and no launch
    without blocks."""
    import paper_1506_02729_gb300 as fkp
    sv = mockgen.survey_small(N=N, assign=2)
    gal, ran = mockgen.catalog(sv, 3)
    kf = 2 * math.pi / sv.L
    got = fkp.Plan(sv.geometry(), (0.0, 0.1 * kf, 5)).power(to_device(gal), to_device(ran))
    assert not got["nmodes"].any() and np.isnan(got["P0"]).all()


def test_schedule_does_not_depend_on_the_first_plans_bins(N=256):
    """Later plans of a grid reuse the schedule that the first one timed, so it
    is timed with every mode carried: a context whose first plan bins the
    lowest modes only (one k_x tile of 16) reads the y-pass time of one whose
    first plan bins to the corner (within a factor of 3; that plan's own y-pass
    takes a tenth of it)."""
    import paper_1506_02729_gb300 as fkp
    sv = mockgen.survey_small(N=N, assign=2)
    kf = 2 * math.pi / sv.L
    full = int(math.ceil(math.sqrt(3) * N / 2))
    ms = {}
    for i, nb in enumerate((1, full)):  # another budget, another context
        ms[nb] = fkp.Plan(sv.geometry(), (0.5 * kf, kf, nb), budget=(100 << 30) + i).schedule()["tuned_ms"]
    assert ms[1][1] > ms[full][1] / 3, ms
    assert ms[1][2] > ms[full][2] / 3, ms
