"""The same tiles in every strip height and column part that a batch size picks
for its layer kind (1: 8 column parts; 2: 4; 40 and 80: 8- or 4-row strips; 160:
16 rows), byte-equal to the oracle in every mode."""
import numpy as np
import pytest

import oracle
from workloads import gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2005_12489_gb300 import hv  # noqa: E402

STYLE_T = (230, 40, 20, 0, 30, 90, 200, 0)


def _layer(ctx, kind):
    if kind == "points":
        pts = gen.gmm_points(40_000, seed=21, k=6)
        return hv.hv_layer_load_points(ctx, pts), pts, lambda r, m: oracle.render_points(pts, r, m, STYLE_T)
    if kind == "lines":
        xy, off = gen.walk_lines(1_500, 9_000, seed=22, n_cities=6)
        return (hv.hv_layer_load_linestrings(ctx, xy, off), gen.segment_midpoints(xy, off, 500),
                lambda r, m: oracle.render_lines(xy, off, r, m, STYLE_T))
    xy, ro, po = gen.star_polygons(1_500, seed=23, k=6, rho_median=2e-3)
    return (hv.hv_layer_load_polygons(ctx, xy, ro, po), gen.polygon_centres(xy, ro, po),
            lambda r, m: oracle.render_polygons(xy, ro, po, r, m, STYLE_T))


@pytest.mark.parametrize("kind", ["points", "lines", "polygons"])
def test_batch_sizes_render_the_same_tiles(kind):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    ctx = hv.hv_create(0)
    L, anchors, reference = _layer(ctx, kind)
    try:
        hv.hv_layer_build_index(L)
        reqs = np.concatenate([[[0, 0, 0, 16]], gen.density_tiles(anchors, 7, 4, 13, 24, seed=24)])
        for mode in (hv.HV_MODE_MASK, hv.HV_MODE_COVERAGE, hv.HV_MODE_RGBA):
            ref = reference(reqs, mode)
            for n in (1, 2, 40, 80, 160):
                rows = np.arange(len(reqs)) if n <= len(reqs) else np.resize(np.arange(len(reqs)), n)
                for k in range(0, len(rows), n):
                    got = hv.render(L, reqs[rows[k:k + n]], mode, hv.make_style(STYLE_T[:3], STYLE_T[4:7]))
                    assert np.array_equal(got, ref[rows[k:k + n]]), (mode, n, k)
    finally:
        hv.hv_layer_free(L)
        hv.hv_destroy(ctx)
