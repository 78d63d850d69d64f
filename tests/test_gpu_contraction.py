"""GPU: the tensor-core contraction at the edges of its tiling, against the
FP32 CUDA-core contraction of the same device shell fields."""
import math

import numpy as np
import pytest

import mockgen
from tests.helpers import to_device
from tests.test_gpu_bispectrum import B_TOL

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

B0, B2, B4, B4B = 16, 32, 64, 512


@pytest.mark.parametrize("N,S,want", [
    (64, 1, B0),                  # one triangle
    (64, 2, B0 | B2 | B4),        # a few pairs of one tile
    (64, 15, B0 | B2 | B4),       # 120 pairs: a tile not full
    (64, 16, B0 | B2 | B4),       # 136 pairs: the second tile begins
    (64, 20, B0 | B2 | B4B),      # zero-area pairs too, several tiles per warpgroup
    (128, 42, B0 | B2 | B4),      # 126 field rows: the widest B operand, several groups of tiles
    (200, 64, B0),                # the most shells
    (200, 64, B0 | B2 | B4B),     # the most rows and pairs
], ids=["one", "few", "tile-1", "tile+1", "split", "rows126", "shells64", "pairs"])
@pytest.mark.parametrize("mode", [1, 2], ids=["bf16x3", "bf16x6"])
def test_tiling_edges_match_fp32(N, S, want, mode):
    """Shells of width 1 about |n| = 1..S, so that the number of pairs S (S +
    1)/2 crosses the tiles of 128.  Both splits' B_l within the bound that the
    other contraction tests hold the accurate mode to (four times it for the
    hi/lo split, whose dropped terms are that much larger), and the same
    triangles.  N^3 is not always a multiple of the 32 points of a chunk times
    the slices, so ragged slice ends are among the cases."""
    import paper_1506_02729_gb300 as fkp
    sv = mockgen.survey_small(N=N, assign=3)
    gal, ran = mockgen.catalog(sv, 5)
    kf = 2 * math.pi / sv.L
    plan = fkp.Plan(sv.geometry(), (0.5 * kf, kf, 8), bshells=(1, 1, 1, S), want=1 | want)
    g, r = to_device(gal), to_device(ran)
    ref = plan.bispectrum(g, r, contraction=0)[1]
    got = plan.bispectrum(g, r, contraction=mode)[1]
    tol = B_TOL if mode == 2 else 4 * B_TOL
    m = ref["NT"] >= 100 if S > 2 else ref["NT"] > 0
    mono = np.abs(ref["T0"][m])
    for k, w in (("T0", B0), ("T2", B2), ("T4", B4), ("T22", B4B)):
        if want & w:
            # graded as B_l is: by the noise-free scale of all triangles of these shells
            d = np.maximum(np.maximum(np.abs(ref[k][m]), mono), np.median(mono))
            assert np.max(np.abs(got[k][m] - ref[k][m]) / d) < tol, k


@pytest.mark.parametrize("N,coarser", [(128, False), (160, True)])
def test_hi_lo_split_on_a_coarser_sum_grid(N, coarser):
    """The hi/lo split's dropped terms average over the points of the sum grid:
    where that is smaller than the plan's (160 -> 128) its sums are those of the
    3-way split, on the plan's own grid they are not."""
    import paper_1506_02729_gb300 as fkp
    sv = mockgen.survey_small(N=N, assign=3)
    gal, ran = mockgen.catalog(sv, 5)
    kf = 2 * math.pi / sv.L
    plan = fkp.Plan(sv.geometry(), (0.5 * kf, kf, 8), bshells=(3, 3, 3, 6), want=1 | B0 | B2 | B4)
    g, r = to_device(gal), to_device(ran)
    b3, b6 = (plan.bispectrum(g, r, contraction=c)[1] for c in (1, 2))
    for k in ("T0", "T2", "T4"):
        assert np.array_equal(b3[k], b6[k]) == coarser, k
