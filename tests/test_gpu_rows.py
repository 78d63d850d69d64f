"""GPU: the FFT passes walk only the rows and planes that hold objects.  Small
clouds of objects at chosen places of the box give the P_l of the FP64 oracle,
whatever rows they leave empty."""
import math

import numpy as np
import pytest

import mockgen
from oracle import power as op
from tests.helpers import P_TOL, p_errors, to_device

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

L = 960.0


def _cloud(boxes, n, seed):
    g = np.random.default_rng(seed)
    pos = np.concatenate([lo + (hi - lo) * g.random((n, 3)) for lo, hi in
                          ((np.array(a, float), np.array(b, float)) for a, b in boxes)])
    nb = np.full(len(pos), 1e-4)
    return {k: pos[:, i].astype(np.float32) for i, k in enumerate("xyz")} | {"nbar": nb.astype(np.float32)}


def _cell(*ijk, N):
    return [np.array(v, float) * (L / N) for v in ijk]


# boxes in cells: [lo, hi) per axis (x, y, z)
PLACES = {
    "one_tile": [((20, 20, 20), (28, 28, 28))],
    "tile_edges": [((15.4, 31.5, 31.5), (16.6, 32.6, 32.6))],       # taps reach into the next tiles and planes
    "two_planes_a_gap_between": [((10, 10, 6), (14, 14, 9)), ((30, 40, 50), (34, 44, 53))],
    "low_corner": [((2.6, 2.6, 2.6), (5, 5, 5))],
    "high_corner": [((51, 51, 51), (55, 55, 55))],
}


@pytest.mark.parametrize("place", sorted(PLACES))
@pytest.mark.parametrize("N,assign,interlace", [(64, 2, False), (60, 3, False), (64, 4, False), (64, 4, True)],
                         ids=["cic", "tsc_runtime", "pcs", "pcs_interlaced"])
def test_empty_rows(place, N, assign, interlace):
    import paper_1506_02729_gb300 as fkp
    boxes = [_cell(a, b, N=64) for a, b in PLACES[place]]
    gal, ran = _cloud(boxes, 200, 1), _cloud(boxes, 1500, 2)
    geom = dict(L=L, N=N, assign=assign, origin=(0.0, 0.0, 0.0), observer=(480.0, 480.0, 480.0), P_fkp=1e4,
                interlace=interlace)
    kf = 2 * math.pi / L
    bins = (0.5 * kf, kf, 24)
    ref = op.power(gal, ran, geom, bins)
    plan = fkp.Plan(geom, bins)
    g, r = to_device(gal), to_device(ran)
    got = plan.power(g, r)
    assert np.array_equal(got["nmodes"], ref["nmodes"])
    assert max(p_errors(got, ref).values()) < P_TOL, p_errors(got, ref)
    # galaxies and the cached randoms in different places: both occupy rows
    other = _cloud([_cell((34, 8, 40), (40, 12, 44), N=64)], 300, 3)
    ref = op.power(other, ran, geom, bins)
    plan.cache_randoms(r)
    got = plan.power(to_device(other), None)
    assert max(p_errors(got, ref).values()) < P_TOL, p_errors(got, ref)
    # the next mock on the same buffers: nothing of the last one's rows is left
    ref = op.power(gal, ran, geom, bins)
    got = plan.power(g, None)
    assert max(p_errors(got, ref).values()) < P_TOL, p_errors(got, ref)


@pytest.mark.parametrize("lo", [(0.0, 0.0, 0.0), (-3.0, 61.0, 30.0), (62.5, 30.0, -1.0)])
@pytest.mark.parametrize("N,assign", [(64, 3), (60, 4), (90, 2)])
def test_periodic_wrap(lo, N, assign):
    """Taps that wrap around the box reach the rows and planes of the far side."""
    import paper_1506_02729_gb300 as fkp
    box = [_cell(lo, tuple(v + 3.0 for v in lo), N=64)]
    gal, ran = _cloud(box, 200, 4), _cloud(box, 1500, 5)
    geom = dict(L=L, N=N, assign=assign, origin=(0.0, 0.0, 0.0), observer=(480.0, 480.0, 480.0), P_fkp=1e4,
                periodic=True)
    kf = 2 * math.pi / L
    plan = fkp.Plan(geom, (0.5 * kf, kf, 24))
    g, r = to_device(gal), to_device(ran)
    got = plan.power(g, r)
    # the same field handed in whole, where the passes take every row: the
    # same arithmetic on the same values, so the same bits
    F = torch.from_numpy(plan.grid(g, r).astype(np.float32) * np.float32(2.0 ** -40)).cuda()
    ref = plan.power_from_grid(F, got["I22"], got["N0"])
    for k in ("P0", "P2", "P4", "P4b", "nmodes"):
        assert np.array_equal(got[k], ref[k], equal_nan=True), k


def test_batch_of_mocks_in_different_places():
    """Each mock of a fused batch has its own rows: the batch equals single calls."""
    import paper_1506_02729_gb300 as fkp
    N = 64
    geom = dict(L=L, N=N, assign=3, origin=(0.0, 0.0, 0.0), observer=(480.0, 480.0, 480.0), P_fkp=1e4)
    kf = 2 * math.pi / L
    plan = fkp.Plan(geom, (0.5 * kf, kf, 24))
    ms = []
    for i, p in enumerate(sorted(PLACES)):
        boxes = [_cell(a, b, N=64) for a, b in PLACES[p]]
        ms.append((to_device(_cloud(boxes, 100, 10 + i)), to_device(_cloud(boxes, 900, 20 + i))))
    got = plan.power_batch([g for g, _ in ms], [r for _, r in ms])
    for (g, r), b in zip(ms, got):
        one = plan.power(g, r)
        for k in ("P0", "P2", "P4", "P4b"):
            assert np.array_equal(b[k], one[k], equal_nan=True), k


@pytest.mark.parametrize("assign", [2, 3, 4])
@pytest.mark.parametrize("N,periodic", [(64, False), (64, True), (60, True)])
def test_second_grid_of_a_pair_is_the_shifted_grid(N, periodic, assign):
    """The second grid of an interlaced pair, filled from the first grid's
    tiles, equals bit for bit the grid of a plan whose origin is half a cell
    further (integer sums of the same rounded taps), with objects on both sides
    of every tile face and, when periodic, around the box."""
    import paper_1506_02729_gb300 as fkp
    lo, hi = (0.0, 64.0) if periodic else (4.0, 59.0)
    box = [_cell((lo,) * 3, (hi,) * 3, N=64)]
    gal, ran = _cloud(box, 3000, 6), _cloud(box, 30000, 7)
    g, r = to_device(gal), to_device(ran)
    geom = dict(L=L, N=N, assign=assign, origin=(0.0, 0.0, 0.0), observer=(480.0, 480.0, 480.0), P_fkp=1e4,
                periodic=periodic)
    kf = 2 * math.pi / L
    pair = fkp.Plan(dict(geom, interlace=True), (0.5 * kf, kf, 8), bshells=(3, 3, 3, 4), want=1 | 16)
    half = 0.5 * L / N
    one = fkp.Plan(dict(geom, origin=(half,) * 3), (0.5 * kf, kf, 8), bshells=(3, 3, 3, 4), want=1 | 16)
    for a, b in zip(pair.grid(g, r, which=1, with_w=True), one.grid(g, r, with_w=True)):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("n", [1, 3, 4, 5, 4095, 8193])
@pytest.mark.parametrize("shift", [0, 1, 3])
def test_catalog_lengths_and_alignments(n, shift):
    """The count launch reads four objects at a time where all arrays start on
    16-byte boundaries: lengths around multiples of four and of a block's share,
    and views that start off those boundaries, give the grid and the scalars of
    an aligned copy (the scalars to the FP64 rounding of another order of sums:
    n terms, 1e-12)."""
    import paper_1506_02729_gb300 as fkp
    N = 64
    box = [_cell((8, 8, 8), (56, 56, 56), N=64)]
    geom = dict(L=L, N=N, assign=3, origin=(0.0, 0.0, 0.0), observer=(480.0, 480.0, 480.0), P_fkp=1e4)
    kf = 2 * math.pi / L
    plan = fkp.Plan(geom, (0.5 * kf, kf, 8))
    base = _cloud(box, n + shift, 8)
    base["w"] = np.linspace(0.5, 1.5, n + shift).astype(np.float32)
    ran = to_device(_cloud(box, 5000, 9))
    whole = to_device(base)
    view = {k: v[shift:] for k, v in whole.items()}
    copy = {k: v.clone() for k, v in view.items()}
    assert np.array_equal(plan.grid(view, ran), plan.grid(copy, ran))
    a, b = plan.power(view, ran), plan.power(copy, ran)
    for k in ("alpha", "I22", "N0", "S3", "W_g"):
        assert abs(a[k] / b[k] - 1) < 1e-12, k
    assert abs(a["W_g"] / float(copy["w"].double().sum()) - 1) < 1e-12


@pytest.mark.parametrize("assign", [2, 3, 4])
@pytest.mark.parametrize("interlace", [False, True], ids=["plain", "pair"])
def test_half_a_cell_outside_a_periodic_box(assign, interlace):
    """Objects within a few roundings of u = -1/2 and u = N - 1/2, where a
    rounding of u + 1/2 decides between the first cell and the last: every
    launch takes the same one, so all of their weight lies in the cells around
    the corner (three axes of up to four weights that each round to 2^-23 or
    better: 2e-6 of it) and no other cell is touched."""
    import paper_1506_02729_gb300 as fkp
    N, H = 64, 15.625
    edge = np.float32(-3 * H) + np.float32([-0.5 * H, (N - 0.5) * H])
    near = [edge]
    for to in (-1e9, 1e9):
        e = edge
        for _ in range(3):
            e = np.nextafter(e, np.float32(to), dtype=np.float32)
            near.append(e)
    near = np.concatenate(near)
    gen = np.random.default_rng(12)
    gal = {k: gen.choice(near, 3000) for k in "xyz"} | {"nbar": np.full(3000, 1e-4, np.float32)}
    ran = {k: np.full(100, (32 - 3) * H, np.float32) for k in "xyz"} | {"nbar": np.full(100, 1e-4, np.float32)}
    geom = dict(L=N * H, N=N, assign=assign, origin=(-3 * H,) * 3, observer=(0.0, 0.0, 0.0), P_fkp=1e4, periodic=True)
    kf = 2 * math.pi / (N * H)
    plan = fkp.Plan(dict(geom, interlace=interlace), (0.5 * kf, kf, 8))
    F = plan.grid(to_device(gal), to_device(ran), which=1 if interlace else 0)
    corner = np.ix_(*[[-3, -2, -1, 0, 1, 2]] * 3)
    middle = np.ix_(*[range(28, 37)] * 3)
    W = 3000 * 0.5  # w = 1/(1 + nbar P) = 1/2
    assert abs(F[corner].sum() * 2.0 ** -40 / W - 1) < 2e-6
    assert np.count_nonzero(F) == np.count_nonzero(F[corner]) + np.count_nonzero(F[middle])


# origins whose sums with far positions are ties of the FP32 spacing there (32,
# 64, 128, that is 2, 4, 8 cells), so that the two grids of a pair round apart
FAR = dict(L=1024.0, N=64, origin=(-48.0, -32.0, -64.0), observer=(480.0, 480.0, 480.0), P_fkp=1e4, periodic=True)
FAR_EXP = (28, 29, 30)


def _far(n, seed, axes, cells=(0, 64)):
    """n objects, on the given axes 2^28 to 2^31 away, elsewhere in the box, all with
    their first-grid cell in [cells) modulo the box; exact weights; and the
    largest distance between an object's two cells."""
    g = np.random.default_rng(seed)
    cat, apart = {}, 0
    for a, k in enumerate("xyz"):
        lo = np.float32(FAR["origin"][a])
        if a in axes:
            ulp = 2.0 ** (FAR_EXP[a] - 23)
            x = (2.0 ** FAR_EXP[a] + ulp * g.integers(1, 2 ** 21, 400 * n)).astype(np.float32)
            x *= g.choice(np.float32([-1, 1]), x.size)
        else:
            x = (lo + 1024 * g.random(400 * n)).astype(np.float32)
        c1 = np.floor((x - lo) * np.float32(1 / 16)).astype(np.int64)
        c2 = np.floor((x - (lo + np.float32(8))) * np.float32(1 / 16)).astype(np.int64)
        keep = np.nonzero((c1 % 64 >= cells[0]) & (c1 % 64 < cells[1]))[0][:n]
        assert len(keep) == n
        cat[k] = x[keep]
        apart = max(apart, int((c1 - c2)[keep].max()))
    cat["nbar"] = np.full(n, 1e-4, np.float32)
    cat["w"] = (g.integers(1, 1024, n) / 1024.0).astype(np.float32)
    return cat, apart


@pytest.mark.parametrize("assign", [2, 3, 4])
@pytest.mark.parametrize("axes", [(0,), (1,), (2,), (0, 1, 2)], ids=["x", "y", "z", "xyz"])
def test_pair_takes_positions_many_boxes_away(assign, axes):
    """A periodic box takes positions up to 1e8 cells away.  There the two FP32
    coordinates of an interlaced pair round apart, and an object's cell in the
    second grid may lie several below its cell in the first: the second grid is
    still, bit for bit, the grid of a plan whose origin is half a cell further."""
    import paper_1506_02729_gb300 as fkp
    (gal, da), (ran, dr) = _far(3000, 1, axes), _far(9000, 2, axes)
    assert max(da, dr) > 1
    geom = dict(FAR, assign=assign)
    kf = 2 * math.pi / 1024.0
    pair = fkp.Plan(dict(geom, interlace=True), (0.5 * kf, kf, 8), bshells=(3, 3, 3, 4), want=1 | 16)
    one = fkp.Plan(dict(geom, origin=tuple(o + 8.0 for o in FAR["origin"])), (0.5 * kf, kf, 8), bshells=(3, 3, 3, 4),
                   want=1 | 16)
    g, r = to_device(gal), to_device(ran)
    for a, b in zip(pair.grid(g, r, which=1, with_w=True), one.grid(g, r, with_w=True)):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("cached", [False, True], ids=["both", "cached_randoms"])
@pytest.mark.parametrize("far", ["galaxies", "randoms", "none"])
def test_rows_of_a_pair_with_positions_many_boxes_away(far, cached):
    """Such objects may reach rows of the second grid that no tile of the first
    grid announces: the spectra are those of the same survey with a weightless
    galaxy in every tile, which makes every row count."""
    import paper_1506_02729_gb300 as fkp
    gal = _far(500, 3, (0, 1, 2) if far == "galaxies" else (), cells=(16, 32))[0]
    ran = _far(2000, 4, (0, 1, 2) if far == "randoms" else (), cells=(16, 32))[0]
    t = np.stack(np.meshgrid(*[np.arange(8.5, 64, 16)] * 3), -1).reshape(-1, 3)
    fill = {k: np.concatenate([gal[k], (FAR["origin"][a] + 16 * t[:, a]).astype(np.float32)]) for a, k in enumerate("xyz")}
    fill["nbar"] = np.full(len(fill["x"]), 1e-4, np.float32)
    fill["w"] = np.concatenate([gal["w"], np.zeros(len(t), np.float32)])
    kf = 2 * math.pi / 1024.0
    plan = fkp.Plan(dict(FAR, assign=3, interlace=True), (0.5 * kf, kf, 24))
    g, f, r = to_device(gal), to_device(fill), to_device(ran)
    if cached:
        plan.cache_randoms(r)
        r = None
    got, ref = plan.power(g, r), plan.power(f, r)
    for k in ("P0", "P2", "P4", "P4b", "nmodes"):
        assert np.array_equal(got[k], ref[k], equal_nan=True), k


@pytest.mark.parametrize("n", [3, 4099, 50001])
def test_results_do_not_depend_on_where_the_arrays_lie(n):
    """Device arrays off 16-byte boundaries, aligned copies of them and host
    arrays give the same bits: every launch takes the objects in one order."""
    import paper_1506_02729_gb300 as fkp
    box = [_cell((8, 8, 8), (56, 56, 56), N=64)]
    geom = dict(L=L, N=64, assign=3, origin=(0.0, 0.0, 0.0), observer=(480.0, 480.0, 480.0), P_fkp=1e4)
    kf = 2 * math.pi / L
    plan = fkp.Plan(geom, (0.5 * kf, kf, 8))
    gal, ran = _cloud(box, n + 3, 8), _cloud(box, 10 * n + 3, 9)
    for c, seed in ((gal, 10), (ran, 11)):  # densities of no round FP32 value: the sums round
        c["nbar"] = (1e-4 * (0.5 + np.random.default_rng(seed).random(len(c["x"])))).astype(np.float32)
    want = None
    for shift in (0, 1, 2, 3):
        lead = {k: np.concatenate([v[:shift], v[3:]]) for k, v in gal.items()}
        rlead = {k: np.concatenate([v[:shift], v[3:]]) for k, v in ran.items()}
        g, r = ({k: v[shift:] for k, v in to_device(c).items()} for c in (lead, rlead))
        host = [{k: np.ascontiguousarray(v[shift:]) for k, v in c.items()} for c in (lead, rlead)]
        for cats in ((g, r), tuple({k: v.clone() for k, v in c.items()} for c in (g, r)), host):
            got = plan.power(*cats)
            want = want or got
            for k in ("alpha", "I22", "I33", "N0", "N0_fkp", "S3", "W_g", "W_r", "Lab", "P0", "P2", "P4", "P4b"):
                assert np.array_equal(got[k], want[k], equal_nan=True), (shift, k)
