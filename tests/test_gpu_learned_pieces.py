"""The learned index's error pass over pieces of every length: bounds that hold
for every key, and a time that follows the number of keys, not of pieces."""
import numpy as np
import pytest

from workloads import gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2005_12489_gb300 import hv  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    c = hv.hv_create(0)
    yield c
    hv.hv_destroy(c)


def build(ctx, pts, segments, mlp):
    L = hv.hv_layer_load_points(ctx, pts)
    opts = hv.hv_build_opts()
    opts.learned_segments = segments
    opts.max_error = 1 << 30
    opts.learned_steps = 20
    if not mlp:
        opts.learned_hidden = hv.HV_LEARNED_NO_MLP
    hv.hv_layer_build_index(L, hv.HV_INDEX_RTREE | hv.HV_INDEX_LEARNED, opts)
    return L


@pytest.mark.parametrize("mlp", [False, True])
@pytest.mark.parametrize("n, segments", [(1023, 1), (1024, 1), (1025, 1), (40_000, 7), (300_001, 100), (2_000_000, 1),
                                         (5_001, 5_001), (5_001, 2_501), (5_001, 1_700), (5_001, 150)])
def test_no_key_outside_its_bound(ctx, n, segments, mlp):
    pts = gen.gmm_points(n, seed=n, k=8)
    pts[n // 2:n // 2 + n // 8] = pts[0]          # a run of equal keys across parts and pieces
    L = build(ctx, pts, segments, mlp)
    try:
        keys = torch.empty(n, dtype=torch.int64, device="cuda")
        hv.hv_layer_keys(L, 0, keys, n)
        pos = torch.empty(n, dtype=torch.int64, device="cuda")
        assert hv.hv_learned_lookup(L, 0, keys, n, pos) == 0      # full searches taken
        k = keys.cpu().numpy()
        assert np.array_equal(pos.cpu().numpy(), np.searchsorted(k, k))
    finally:
        hv.hv_layer_free(L)


def test_few_long_pieces_cost_no_more_than_many(ctx):
    """10 M keys in 10 pieces against 20 thousand: the error pass alone (no
    network) took some hundred times as long with a warp per piece."""
    pts = gen.gmm_points(10_000_000, seed=6, k=64)
    ms = {}
    for segments in (0, 8, 0, 8):
        L = build(ctx, pts, segments, False)
        ms.setdefault(segments, []).append(hv.hv_layer_info_get(L).train_ms)
        hv.hv_layer_free(L)
    assert min(ms[8]) < 10 * min(ms[0]), ms
