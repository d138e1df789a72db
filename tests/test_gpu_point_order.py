"""Point layers sorted by their keys alone: the sorted keys are those of the
level-by-level Hilbert definition, and tiles rendered from the points read back
off the keys equal the oracle's, at layer sizes around a leaf, a sort block and
with all points alike."""
import numpy as np
import pytest

import oracle
from workloads import gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2005_12489_gb300 import hv  # noqa: E402

HALF = 1 << 30


def _keys(pts):
    x, y = (pts.astype(np.int64) + HALF).T.copy()
    d = np.zeros(len(x), dtype=np.uint64)
    for i in range(30, -1, -1):
        rx, ry = (x >> i) & 1, (y >> i) & 1
        d = (d << np.uint64(2)) | ((3 * rx) ^ ry).astype(np.uint64)
        flip = (ry == 0) & (rx == 1)
        x, y = np.where(flip, ~x, x), np.where(flip, ~y, y)
        x, y = np.where(ry == 0, y, x), np.where(ry == 0, x, y)
    return d


@pytest.mark.parametrize("n", [1, 31, 32, 33, 1025, 4097, 100_003])
@pytest.mark.parametrize("alike", [False, True])
def test_points_sorted_by_key(n, alike):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    pts = np.ascontiguousarray(gen.gmm_points(max(n, 16), seed=n, k=4)[:n], dtype=np.int32)
    if alike:
        pts[:] = pts[0]
    else:
        edge = np.array([[-HALF, -HALF], [HALF - 1, HALF - 1], [-HALF, HALF - 1], [HALF - 1, -HALF], [0, 0], [-1, -1]])
        pts[:min(n, 6)] = edge[:min(n, 6)]
    ctx = hv.hv_create(0)
    L = hv.hv_layer_load_points(ctx, pts)
    try:
        hv.hv_layer_build_index(L)
        got = torch.empty(n, dtype=torch.int64, device="cuda")
        hv.hv_layer_keys(L, 0, got, n)
        assert np.array_equal(got.cpu().numpy().astype(np.uint64), np.sort(_keys(pts)))
        reqs = np.concatenate([[[0, 0, 0, 1024], [3, 0, 0, 64]], gen.density_tiles(pts, 6, 2, 14, 32, seed=n)])
        out = hv.render(L, reqs, hv.HV_MODE_COVERAGE)
        assert np.array_equal(out, oracle.render_points(pts, reqs, hv.HV_MODE_COVERAGE, (0,) * 8))
    finally:
        hv.hv_layer_free(L)
        hv.hv_destroy(ctx)
