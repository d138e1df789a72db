"""Buffers with ground radii far larger than a sample spacing, byte-equal to the
oracle: segments and polygon outlines whose distance from a sample of the tile
is within a few units of the radius, single tiles (column parts) and full
batches (16-row strips), MASK and COVERAGE."""
import numpy as np
import pytest

import oracle
from geom import centre, polys_to_arrays

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2005_12489_gb300 import hv  # noqa: E402

HALF = 1 << 30
STYLE_T = (230, 40, 20, 0, 30, 90, 200, 0)


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    c = hv.hv_create(0)
    yield c
    hv.hv_destroy(c)


def check(ctx, kind, xy, req, radius):
    """One layer (points; lines: a segment per vertex pair; polygons: a ring per
    three vertices), one tile, both modes, alone and 160 times in a batch."""
    xy = np.ascontiguousarray(xy, dtype=np.int32)
    reqs = np.array([req], dtype=np.uint32)
    if kind == "points":
        L = hv.hv_layer_load_points(ctx, xy)
        ref = lambda mode: oracle.render_points(xy, reqs, mode, STYLE_T, R_units=radius)  # noqa: E731
    elif kind == "lines":
        off = np.arange(0, len(xy) + 1, 2, dtype=np.uint64)
        L = hv.hv_layer_load_linestrings(ctx, xy, off)
        ref = lambda mode: oracle.render_lines(xy, off, reqs, mode, STYLE_T, R_units=radius)  # noqa: E731
    else:
        xy, ro, po = polys_to_arrays([[r] for r in xy.reshape(-1, 3, 2).tolist()])
        L = hv.hv_layer_load_polygons(ctx, xy, ro, po)
        ref = lambda mode: oracle.render_polygons(xy, ro, po, reqs, mode, STYLE_T, R_units=radius)  # noqa: E731
    try:
        hv.hv_layer_build_index(L)
        for mode in (hv.HV_MODE_MASK, hv.HV_MODE_COVERAGE):
            want = ref(mode)[0]
            for n in (1, 160):
                d = torch.from_numpy(hv.make_requests(np.repeat(reqs, n, 0)).view(np.uint8).copy()).cuda()
                out = torch.full((n, hv.hv_tile_bytes(mode)), 0xAB, dtype=torch.uint8, device="cuda")
                hv.hv_render_buffer(L, d, n, mode, hv.HV_INDEX_RTREE, radius, None, out, out.numel(), None)
                got = out.cpu().numpy()
                assert np.array_equal(got[0], want) and np.array_equal(got[-1], want), (kind, mode, n, req, radius, xy)
        assert hv.hv_layer_take_status(L) == 0
    finally:
        hv.hv_layer_free(L)


def grazes(rng, z, radius, n):
    """n segments (n, 2, 2) whose distance from a sample of tile (z, 2^(z-1),
    2^(z-1)) is the radius, give or take three units: any slope, level and
    upright ones and near misses of both, the contact inside or at an end."""
    out = []
    t = (1 << z) // 2
    while len(out) < n:
        p = np.array(centre(z, t, t, int(rng.integers(0, 256)), int(rng.integers(0, 256))), dtype=np.float64)
        th = rng.choice([0.0, np.pi / 2, rng.uniform(0, 2 * np.pi), 10.0 ** rng.uniform(-6, -1),
                         np.pi / 2 - 10.0 ** rng.uniform(-6, -1)])
        size = 2.0 ** rng.uniform(0, 29)
        along = rng.choice([rng.uniform(0, 1), rng.integers(0, 2)])
        turn = rng.uniform(-1.5, 1.5) if along in (0, 1) else 0.0
        nrm = np.array([-np.sin(th + turn), np.cos(th + turn)]) * rng.choice([-1, 1])
        a = p + nrm * (radius + rng.integers(-3, 4)) - np.array([np.cos(th), np.sin(th)]) * size * along
        b = a + np.array([np.cos(th), np.sin(th)]) * size
        if max(np.abs(a).max(), np.abs(b).max()) < HALF - 2:
            out.append(np.round([a, b]))
    return np.array(out)


def test_segment_at_a_radius_of_millions_of_spacings(ctx):
    xy = [(-291826, 13957715), (-250905, 13958577)]
    check(ctx, "lines", xy, (19, 262144, 262144, 1), 13_959_460)
    check(ctx, "polygons", xy + [(-270_000, 14_300_000)], (19, 262144, 262144, 1), 13_959_460)


@pytest.mark.parametrize("z", [13, 16, 19])
@pytest.mark.parametrize("radius", [100_003, 330_084, 3_000_017, 13_959_460, 1 << 27, (1 << 29) - 12_345, 1 << 29])
def test_grazing_segments(ctx, z, radius):
    rng = np.random.default_rng(z * 1000 + radius % 997)
    for k, seg in enumerate(grazes(rng, z, radius, 12)):
        t = (1 << z) // 2
        check(ctx, "lines", seg, (z, t, t, 1), radius)
        if k % 3 == 0:
            # a third vertex farther from the tile than the segment
            far = np.clip(np.round(seg.mean(0) * 1.5), -HALF, HALF - 1)
            check(ctx, "polygons", np.concatenate([seg, far[None]]), (z, t, t, 1), radius)


@pytest.mark.parametrize("kind", ["points", "lines", "polygons"])
@pytest.mark.parametrize("radius, f", [((1 << 24) + 1, 1 << 24), ((1 << 25) + 1, 1 << 25), ((1 << 28) + 15, 1 << 28)])
@pytest.mark.parametrize("offset", [4, 8])
def test_row_that_is_only_just_within_reach(ctx, kind, radius, f, offset):
    """An object left of the tile, f above its first super-sample or pixel row:
    the radius is no float, and the row is reached by the last few units of it."""
    y = offset - f
    xy = [(-3000, y), (-2000, y)] + ([(-2500, y - 100_000)] if kind == "polygons" else [])
    check(ctx, kind, xy, (19, 262144, 262144, 1), radius)


@pytest.mark.parametrize("kind", ["points", "lines", "polygons"])
def test_radius_beyond_the_tile(ctx, kind):
    """Every sample of the tiles lies within the radius of any record: all are
    covered, and a layer of many records takes about the time of one record (drawing
    each of its boxes took a dozen times as long)."""
    rng = np.random.default_rng(8)
    z, radius = 10, 1 << 28
    d = torch.from_numpy(hv.make_requests(np.repeat(np.array([[z, 512, 511, 1]]), 60, 0)).view(np.uint8).copy()).cuda()
    out = torch.zeros((60, 65536), dtype=torch.uint8, device="cuda")
    ms = []
    for n in (1, 50_000):
        xy = rng.integers(-2 ** 22, 2 ** 22, (3 * n, 2)).astype(np.int32)
        if kind == "points":
            L = hv.hv_layer_load_points(ctx, xy)
        elif kind == "lines":
            L = hv.hv_layer_load_linestrings(ctx, xy, np.arange(0, 3 * n + 1, 3, dtype=np.uint64))
        else:
            xy = np.repeat(xy[::3], 3, 0) + np.tile([[0, 0], [900, 0], [0, 900]], (n, 1)).astype(np.int32)
            L = hv.hv_layer_load_polygons(ctx, xy, np.arange(0, 3 * n + 1, 3, dtype=np.uint64), np.arange(n + 1, dtype=np.uint64))
        hv.hv_layer_build_index(L)
        best = 1e9
        for _ in range(20):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            out.zero_()
            a.record()
            hv.hv_render_buffer(L, d, 60, hv.HV_MODE_COVERAGE, hv.HV_INDEX_RTREE, radius, None, out, out.numel(),
                                torch.cuda.current_stream())
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
            assert bool(((out & 7) == 4).all())
        ms.append(best)
        assert hv.hv_layer_take_status(L) == 0
        hv.hv_layer_free(L)
    assert ms[1] < 4 * ms[0], ms
