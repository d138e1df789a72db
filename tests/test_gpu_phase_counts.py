"""Leaf visits in the phase profile: how many decided a sample, and how many met
no record in reach, where the strips of a tile make them countable by hand."""
import numpy as np
import pytest

from geom import at, centre, polys_to_arrays, ps

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2005_12489_gb300 import hv  # noqa: E402

Z, T = 12, 2048
REQ = np.array([[Z, T, T, 16]], dtype=np.uint32)     # radius 1 px
VISITS, EMPTY, DECIDED = (hv.PHASE_NAMES.index(k) for k in ("leaf_visits", "leaf_empty", "leaf_decided"))


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    c = hv.hv_create(0)
    yield c
    hv.hv_destroy(c)


def profile(L, mode=hv.HV_MODE_COVERAGE, req=REQ):
    hv.hv_layer_build_index(L)
    d = torch.from_numpy(hv.make_requests(req).view(np.uint8).copy()).cuda()
    out = torch.zeros((1, hv.hv_tile_bytes(mode)), dtype=torch.uint8, device="cuda")
    ph = torch.zeros(2 * hv.HV_PHASE_COUNT, dtype=torch.int64, device="cuda")
    hv.hv_render_tiles_phases(L, d, 1, mode, hv.HV_INDEX_RTREE, None, out, out.numel(), ph)
    torch.cuda.synchronize()
    hv.hv_layer_free(L)
    ph = ph.cpu().numpy().reshape(2, -1)
    return ph[:, [VISITS, EMPTY, DECIDED]].tolist(), out.cpu().numpy()[0].reshape(256, 256)


def strips_with(tile):
    return int(tile.reshape(64, -1).any(1).sum())


def test_points(ctx):
    # two points ten rows apart, in one leaf too wide to draw as a box: each strip between them visits it
    xy = np.array([at(Z, T, T, 10, 9), at(Z, T, T, 200, 30)], dtype=np.int32)
    (got, _), tile = profile(hv.hv_layer_load_points(ctx, xy))
    assert got[2] == strips_with(tile) and got[0] >= got[1] + got[2]
    assert got[0] >= 6                       # strips 2 .. 7 meet the leaf's box


def test_lines(ctx):
    xy = np.array([at(Z, T, T, 20, 18), at(Z, T, T, 90, 101)], dtype=np.int32)
    (got, _), tile = profile(hv.hv_layer_load_linestrings(ctx, xy, np.array([0, 2], dtype=np.uint64)))
    assert got[2] == strips_with(tile) > 20 and got[1] <= got[0] - got[2]
    # one segment left of the tile and one right of it: the leaf's box spans the tile, no record is in reach
    far = 20 * ps(Z)
    a, b = centre(Z, T, T, 0, 0), centre(Z, T, T, 255, 255)
    xy = np.array([(a[0] - far, a[1]), (a[0] - far, b[1]), (b[0] + far, a[1]), (b[0] + far, b[1])], dtype=np.int32)
    (got, _), tile = profile(hv.hv_layer_load_linestrings(ctx, xy, np.array([0, 2, 4], dtype=np.uint64)))
    assert got == [64, 64, 0] and not tile.any()


def test_polygons(ctx):
    ring = [at(Z, T, T, 40, 41), at(Z, T, T, 150, 41), at(Z, T, T, 150, 171), at(Z, T, T, 40, 171)]
    xy, ro, po = polys_to_arrays([[ring]])
    (fill, outline), tile = profile(hv.hv_layer_load_polygons(ctx, xy, ro, po))
    assert fill[2] == strips_with(tile & 8) and fill[0] == fill[1] + fill[2]
    assert outline[2] == strips_with(tile & 7) and outline[0] >= outline[1] + outline[2]


@pytest.mark.parametrize("lines", [False, True])
def test_wide_reach_around_a_crowd(ctx, lines):
    """20,000 records within a tenth of a sample spacing and a radius of 64 px: the
    samples beside the disc are in no record's reach, so that a strip that the disc's
    border crosses visits a few of the 625 leaves (all of them, when reach was
    bounded to a column or two only)."""
    rng = np.random.default_rng(4)
    a = rng.integers(-600, 600, (20_000, 2)) + (8192, 8192)      # on a super-sample of tile (8, 128, 128)
    a += 64 * ps(8)
    req = np.array([[8, 128, 128, 1024]], dtype=np.uint32)
    if lines:
        xy = np.stack([a, a + rng.integers(-50, 50, a.shape)], 1).reshape(-1, 2).astype(np.int32)
        L = hv.hv_layer_load_linestrings(ctx, xy, np.arange(0, len(xy) + 1, 2, dtype=np.uint64))
    else:
        L = hv.hv_layer_load_points(ctx, a.astype(np.int32))
    (got, _), tile = profile(L, req=req)
    assert 16 <= strips_with(tile) <= 40 and got[0] < 64 * 100, got
