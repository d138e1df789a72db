"""Segments and outlines across the whole grid, cut into small pieces, in the
tiles along its borders at zooms 0 to 2 and thin radii, byte-equal to the
oracle: between a strip's outermost lattice points and the opposite ends the
coordinates differ by exactly 2^31."""
import numpy as np
import pytest

import oracle
import oracle_par
from geom import polys_to_arrays

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2005_12489_gb300 import hv  # noqa: E402

HALF = 1 << 30


def _segments(z, mode):
    """Level and upright segments near the four borders, ending half a sample
    spacing (and a unit beside that) before the opposite border, both ways round."""
    h = 1 << (23 - z if mode == hv.HV_MODE_MASK else 22 - z)
    out = []
    for k, d in ((1, 0), (2, 0), (3, 1), (7, -1)):
        a, near, far = -HALF + k * h // 2, -HALF, HALF - h // 2 + d
        for s in (((a, near), (a, far)), ((a, far), (a, near))):
            out += [s, tuple((y, x) for x, y in s)]
            out += [tuple((min(-x, HALF - 1), min(-y, HALF - 1)) for x, y in s),
                    tuple((min(-y, HALF - 1), min(-x, HALF - 1)) for x, y in s)]
    return out


@pytest.mark.parametrize("z", [0, 1, 2])
@pytest.mark.parametrize("kind", ["lines", "polygons"])
def test_whole_grid_segments_at_the_borders(z, kind):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    rng = np.random.default_rng(z)
    last = (1 << z) - 1
    tiles = sorted({(x, y) for x in (0, last) for y in (0, last)})
    reqs = np.array([[z, x, y, r] for x, y in tiles for r in (1, 2, 3, 8)], dtype=np.uint32)
    ctx = hv.hv_create(0)
    try:
        for mode in (hv.HV_MODE_MASK, hv.HV_MODE_COVERAGE):
            # short ones around the grid's middle, so that the long ones are cut into pieces of 2^21 to 2^22 units
            c = rng.integers(-2 ** 20, 2 ** 20, (20_000, 2))
            short = np.stack([c, c + rng.integers(-500, 500, c.shape)], 1)
            seg = np.concatenate([np.array(_segments(z, mode)), short]).astype(np.int32)
            if kind == "lines":
                off = np.arange(0, 2 * len(seg) + 1, 2, dtype=np.uint64)
                xy = seg.reshape(-1, 2)
                L = hv.hv_layer_load_linestrings(ctx, xy, off)
                ref = oracle_par.render(lambda r: oracle.render_lines(xy, off, r, mode), reqs)
            else:
                xy, ro, po = polys_to_arrays([[s] for s in seg.tolist()])   # rings of two vertices
                L = hv.hv_layer_load_polygons(ctx, xy, ro, po)
                ref = oracle_par.render(lambda r: oracle.render_polygons(xy, ro, po, r, mode), reqs)
            hv.hv_layer_build_index(L)
            assert hv.hv_layer_info_get(L).piece_extent <= 1 << 22
            for n in (1, len(reqs), 160):
                rows = np.resize(np.arange(len(reqs)), max(n, len(reqs)))
                for k in range(0, len(rows), n):
                    part = rows[k:k + n]
                    d = torch.from_numpy(hv.make_requests(reqs[part]).view(np.uint8).copy()).cuda()
                    out = torch.full((len(part), hv.hv_tile_bytes(mode)), 0xAB, dtype=torch.uint8, device="cuda")
                    hv.hv_render_tiles(L, d, len(part), mode, hv.HV_INDEX_RTREE, None, out, out.numel(), None)
                    assert np.array_equal(out.cpu().numpy(), ref[part]), (mode, n)
            assert hv.hv_layer_take_status(L) == 0
            hv.hv_layer_free(L)
    finally:
        hv.hv_destroy(ctx)
