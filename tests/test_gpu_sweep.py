"""Points and segments drawn row by row over a strip's sample lattice: layers
and requests at the edges of that path, byte-equal to the oracle in every mode,
strip height and column part -- points: leaves with 1 to 33 points, strip, part
and grid borders, samples at exactly R and R +- 1 units, rows on both sides of
the 32-bit radius, reaches wider than the 32-column window, crowded and sparse
leaves; segments: level, upright, almost level and slanted ones, zero lengths,
ends far outside the strip and the grid's whole width, leaves with few and
with many (piece, row) pairs."""
import numpy as np
import pytest

import oracle
import oracle_par
from geom import centre, ps
from workloads import gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2005_12489_gb300 import hv  # noqa: E402

STYLE_T = (230, 40, 20, 0, 30, 90, 200, 0)
MODES = [hv.HV_MODE_MASK, hv.HV_MODE_COVERAGE, hv.HV_MODE_RGBA]
HALF = 1 << 30


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    c = hv.hv_create(0)
    yield c
    hv.hv_destroy(c)


def _check(ctx, pts, reqs, radius=None, batches=(1, 3, 200), lines=False):
    pts = np.ascontiguousarray(pts, dtype=np.int32)
    reqs = np.array(reqs, dtype=np.uint32)
    off = np.arange(0, len(pts) + 1, 2, dtype=np.uint64)   # lines: a segment per vertex pair
    L = hv.hv_layer_load_linestrings(ctx, pts, off) if lines else hv.hv_layer_load_points(ctx, pts)
    hv.hv_layer_build_index(L, hv.HV_INDEX_RTREE | hv.HV_INDEX_LEARNED)
    s = hv.make_style(STYLE_T[:3], STYLE_T[4:7])
    try:
        for mode in MODES:
            ref = oracle_par.render(
                lambda r: oracle.render_lines(pts, off, r, mode, STYLE_T, R_units=radius) if lines
                else oracle.render_points(pts, r, mode, STYLE_T, R_units=radius), reqs)
            for index in (hv.HV_INDEX_RTREE, hv.HV_INDEX_LEARNED):
                for per in batches:      # column parts, 4-row strips, full strips (requests repeated)
                    rows = np.resize(np.arange(len(reqs)), max(per, len(reqs))) if per > len(reqs) else np.arange(len(reqs))
                    for k in range(0, len(rows), per):
                        part = rows[k:k + per]
                        d = torch.from_numpy(hv.make_requests(reqs[part]).view(np.uint8).copy()).cuda()
                        out = torch.full((len(part), hv.hv_tile_bytes(mode)), 0xAB, dtype=torch.uint8, device="cuda")
                        if radius is None:
                            hv.hv_render_tiles(L, d, len(part), mode, index, s, out, out.numel(), None)
                        else:
                            hv.hv_render_buffer(L, d, len(part), mode, index, radius, s, out, out.numel(), None)
                        assert np.array_equal(out.cpu().numpy(), ref[part]), (mode, index, per)
        assert hv.hv_layer_take_status(L) == 0
    finally:
        hv.hv_layer_free(L)


@pytest.mark.parametrize("z", [0, 1, 8, 9, 13, 19])
def test_samples_at_exactly_R(ctx, z):
    """Around samples of a tile's corners and strip borders: points at R and
    R +- 1 units along an axis and on a 3-4-5 slant."""
    t = (1 << z) // 2
    pts, reqs = [], []
    for r16 in (5, 16, 32, 240):
        R = r16 << (19 - z)
        reqs.append([z, t, t, r16])
        for i, j in ((0, 0), (255, 255), (63, 15), (64, 16), (130, 131)):
            cx, cy = centre(z, t, t, i, j)
            for o in (0, ps(z) // 4):
                for d in (-1, 0, 1):
                    pts += [(cx + o + R + d, cy + o), (cx + o, cy + o - R - d),
                            (cx + o + 4 * R // 5 + d, cy + o - 3 * R // 5)]
    pts = np.array([p for p in pts if all(-HALF <= v < HALF for v in p)] + [(0, 0), (-HALF, -HALF), (HALF - 1, HALF - 1)])
    _check(ctx, pts, reqs)


@pytest.mark.parametrize("n", [1, 31, 32, 33, 1025])
def test_leaf_remainders_and_grid_borders(ctx, n):
    rng = np.random.default_rng(n)
    edge = rng.choice([-HALF, HALF - 1, 0, -1], size=(n, 2))
    pts = np.where(rng.random((n, 2)) < 0.5, edge, rng.integers(-HALF, HALF, (n, 2)))
    _check(ctx, pts, [[0, 0, 0, 16], [0, 0, 0, 1024], [1, 0, 0, 40], [1, 1, 1, 1], [2, 3, 0, 512], [5, 31, 31, 32]])


def test_crowded_and_sparse_leaves(ctx):
    """Clusters far narrower than a pixel, duplicates, and lone points, at
    radii from a sixteenth of a pixel to 64 px."""
    rng = np.random.default_rng(9)
    c = rng.integers(-2 ** 20, 2 ** 20, (40, 2))
    crowd = (c[rng.integers(0, 40, 60_000)] + rng.integers(-300, 300, (60_000, 2)))
    pts = np.concatenate([crowd, np.repeat(c, 50, axis=0), rng.integers(-2 ** 22, 2 ** 22, (500, 2))])
    reqs = gen.density_tiles(pts.astype(np.int32), 6, 7, 16, [1, 16, 33, 130], seed=5)
    _check(ctx, pts, np.concatenate([reqs, [[9, 256, 256, 1024], [12, 2048, 2048, 700]]]))


@pytest.mark.parametrize("radius", [0, 1, 46340, 46341, 3_000_003, 1 << 29])
def test_ground_radii(ctx, radius):
    rng = np.random.default_rng(11)
    pts = rng.integers(-2 ** 24, 2 ** 24, (3000, 2))
    _check(ctx, pts, [[5, 16, 16, 1], [8, 128, 127, 1], [13, 4096, 4095, 1], [19, 262144, 262143, 1], [0, 0, 0, 1]],
           radius=radius, batches=(1, 150))


def _fan(rng, n, spread, size):
    """n segments (2n, 2): slopes from level to upright with near misses of
    both, lengths over three decades, some of length 0, swapped ends."""
    a = rng.integers(-spread, spread, (n, 2)).astype(np.float64)
    th = np.choose(rng.integers(0, 5, n), [np.zeros(n), np.full(n, np.pi / 2), rng.uniform(0, 2 * np.pi, n),
                                           10.0 ** rng.uniform(-7, -1, n), np.pi / 2 - 10.0 ** rng.uniform(-7, -1, n)])
    d = size * 10.0 ** rng.uniform(-3, 0, n) * (rng.random(n) > 0.05)
    b = a + np.stack([d * np.cos(th), d * np.sin(th)], 1)
    flip = (rng.random(n) < 0.5)[:, None]
    seg = np.stack([np.where(flip, b, a), np.where(flip, a, b)], 1)
    return np.clip(np.round(seg), -HALF, HALF - 1).astype(np.int32).reshape(-1, 2)


@pytest.mark.parametrize("spread, size", [(2 ** 12, 2 ** 11), (2 ** 18, 2 ** 20), (2 ** 24, 2 ** 29), (2 ** 29, 2 ** 30)])
def test_segments_of_every_slope(ctx, spread, size):
    rng = np.random.default_rng(spread)
    seg = _fan(rng, 1500, spread, size)
    zs = [z for z in (0, 3, 9, 13, 19) if (1 << (31 - z)) < 4096 * spread]
    _check(ctx, seg, [[z, (1 << z) // 2 - k, (1 << z) // 2 - (1 - k), r] for z in zs for k in (0, 1) if z
                      for r in (1, 8, 40)] + [[0, 0, 0, 16], [2, 1, 2, 1024]], lines=True, batches=(1, 120))


@pytest.mark.parametrize("radius", [0, 7, 100_003, 1 << 27])
def test_segments_at_ground_radii(ctx, radius):
    seg = _fan(np.random.default_rng(5), 400, 2 ** 22, 2 ** 23)
    _check(ctx, seg, [[7, 64, 63, 1], [11, 1024, 1024, 1], [16, 32768, 32767, 1]], radius=radius, lines=True,
           batches=(1, 150))


def _rings(rng):
    """Polygons for the fill: a comb of 401 vertices across many tiles, squares
    on sample positions and word borders, nested rings, slivers, one as wide
    as the grid, and overlapping stars."""
    P = []
    x = np.repeat(np.linspace(-3e6, 3e6, 200), 2)
    y = np.tile([-2e6, 2e6, 2e6, -2e6], 100) + rng.integers(-5, 5, 400)
    P.append([np.concatenate([np.stack([x, y], 1), [[0, 2.5e6]]])])
    for z, i, j, k in ((9, 0, 0, 32), (11, 31, 15, 33), (13, 224, 240, 32), (10, 255, 255, 3)):
        cx, cy = centre(z, (1 << z) // 2, (1 << z) // 2, i, j)
        d = k * ps(z)
        sq = np.array([[0, 0], [d, 0], [d, d], [0, d]])
        P.append([sq + (cx, cy), sq // 2 + (cx + d // 4, cy + d // 4)])
        P.append([sq + (cx + ps(z) // 4, cy - ps(z) // 4)])
    P.append([np.array([[-HALF, -5], [HALF - 1, 3], [HALF - 1, 90_000], [-HALF, 70_000]])])
    P.append([np.array([[-HALF, -HALF], [HALF - 1, -HALF], [0, -HALF // 2]])])
    for _ in range(60):
        c, m = rng.integers(-2 ** 22, 2 ** 22, 2), int(rng.integers(3, 90))
        a = np.sort(rng.uniform(0, 2 * np.pi, m))
        r = 2.0 ** rng.uniform(8, 22) * rng.uniform(0.3, 1, m)
        P.append([c + np.stack([r * np.cos(a), r * np.sin(a)], 1)])
    rings = [np.clip(np.floor(r), -HALF, HALF - 1).astype(np.int32) for p in P for r in p]
    ro = np.concatenate([[0], np.cumsum([len(r) for r in rings])]).astype(np.uint64)
    po = np.concatenate([[0], np.cumsum([len(p) for p in P])]).astype(np.uint64)
    return np.concatenate(rings), ro, po


@pytest.mark.parametrize("aa", [False, True])
def test_fill_of_every_width(ctx, aa):
    xy, ro, po = _rings(np.random.default_rng(8))
    L = hv.hv_layer_load_polygons(ctx, xy, ro, po)
    hv.hv_layer_build_index(L, hv.HV_INDEX_RTREE | hv.HV_INDEX_LEARNED)
    reqs = np.array([[0, 0, 0, 8], [1, 0, 1, 16], [8, 128, 127, 8]] +
                    [[z, (1 << z) // 2 - a, (1 << z) // 2 - b, 4] for z in (9, 11, 13, 16) for a in (0, 1) for b in (0, 1)],
                    dtype=np.uint32)
    s, fill = hv.make_style(STYLE_T[:3], STYLE_T[4:7]), hv.make_fill_style(aa=aa)
    try:
        for mode in MODES:
            ref = oracle_par.render(lambda r: oracle.render_polygons(xy, ro, po, r, mode, STYLE_T, aa=aa), reqs)
            for index in (hv.HV_INDEX_RTREE, hv.HV_INDEX_LEARNED):
                for per in (1, 3, 150):
                    rows = np.resize(np.arange(len(reqs)), max(per, len(reqs)))
                    for k in range(0, len(rows), per):
                        part = rows[k:k + per]
                        d = torch.from_numpy(hv.make_requests(reqs[part]).view(np.uint8).copy()).cuda()
                        out = torch.full((len(part), hv.hv_tile_bytes(mode)), 0xAB, dtype=torch.uint8, device="cuda")
                        hv.hv_render_tiles_styled(L, d, len(part), mode, index, s, fill, out, out.numel(), None)
                        assert np.array_equal(out.cpu().numpy(), ref[part]), (mode, index, per)
        assert hv.hv_layer_take_status(L) == 0
    finally:
        hv.hv_layer_free(L)
