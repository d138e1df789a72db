"""A point layer whose sort fails part of the way (an error code from a fake of
the library's sort, after one of its eight passes) keeps its points: the next
build of its index succeeds and renders the oracle's tiles."""
import glob
import os
import shutil
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = r"""
#include <cub/device/device_radix_sort.cuh>
namespace cub {
struct FailingRadixSort {
    // every other sort, from the first on, stops after its lowest eight bits
    template <class K, class N>
    static cudaError_t SortKeys(void* temp, size_t& bytes, DoubleBuffer<K>& keys, N n, int bit0, int bit1) {
        static int calls = 0;
        if (temp == nullptr || calls++ % 2 == 1) return DeviceRadixSort::SortKeys(temp, bytes, keys, n, bit0, bit1);
        DeviceRadixSort::SortKeys(temp, bytes, keys, n, bit0, bit0 + 8);
        return cudaErrorMemoryAllocation;
    }
    template <class... A>
    static cudaError_t SortPairs(A&&... a) { return DeviceRadixSort::SortPairs((A&&)a...); }
};
}  // namespace cub
#define DeviceRadixSort FailingRadixSort
"""

PROGRAM = r"""
import sys
import numpy as np
sys.path.insert(0, sys.argv[2])
from paper_2005_12489_gb300 import hv
hv.LIB_PATH = sys.argv[1]
import oracle
from workloads import gen
for n in (5, 70_001):
    pts = gen.gmm_points(max(n, 16), seed=n, k=4)[:n]
    reqs = np.concatenate([[[0, 0, 0, 1024]], gen.density_tiles(pts, 6, 2, 12, 32, seed=n)])
    want = oracle.render_points(pts, reqs, hv.HV_MODE_COVERAGE)
    ctx = hv.hv_create(0)
    held = hv.hv_ctx_device_bytes(ctx)
    L = hv.hv_layer_load_points(ctx, pts)
    loaded = hv.hv_ctx_device_bytes(ctx)
    try:
        hv.hv_layer_build_index(L)
    except hv.HVError as e:
        assert e.status == hv.HV_ECUDA, e
    else:
        raise AssertionError("the planted failure did not show")
    assert hv.hv_ctx_device_bytes(ctx) == loaded
    hv.hv_layer_build_index(L, hv.HV_INDEX_RTREE | hv.HV_INDEX_LEARNED)
    for index in (hv.HV_INDEX_RTREE, hv.HV_INDEX_LEARNED):
        assert np.array_equal(hv.render(L, reqs, hv.HV_MODE_COVERAGE, index_kind=index), want)
    hv.hv_layer_free(L)
    assert hv.hv_ctx_device_bytes(ctx) <= held + (1 << 24)   # (the context's own scratch)
    hv.hv_destroy(ctx)
print("kept")
"""


def test_points_survive_a_failed_sort(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    pkg = os.path.join(ROOT, "paper_2005_12489_gb300")
    fake, obj, lib = tmp_path / "fake.h", tmp_path / "hv_build.o", tmp_path / "libhivision.so"
    fake.write_text(FAKE)
    arch = ["-gencode", "arch=compute_103a,code=sm_103a"]
    subprocess.run([nvcc, *arch, "-O2", "-std=c++17", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr", "-include",
                    str(fake), "-I", os.path.join(ROOT, "include"), "-c", os.path.join(pkg, "csrc", "hv_build.cu"), "-o",
                    str(obj)], check=True)
    others = [o for o in glob.glob(os.path.join(pkg, "_build", "*.o")) if os.path.basename(o) != "hv_build.o"]
    subprocess.run([nvcc, *arch, "-shared", "-o", str(lib), str(obj), *others, "-lcudart_static", "-lrt", "-ldl",
                    "-lpthread"], check=True)
    prog = tmp_path / "prog.py"
    prog.write_text(PROGRAM)
    r = subprocess.run([sys.executable, str(prog), str(lib), ROOT], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout == "kept\n", r.stderr[-2000:]
