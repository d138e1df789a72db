"""The Hilbert index of hv_device.cuh (states of all levels by prefix
composition) and its inverse, compiled for the host, against the level by
level definition: every point of the coarse grids, the grid's corners and
borders, and random points of every magnitude."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cstdio>
#include <random>
#include "hv_device.cuh"
static uint64_t by_levels(int32_t gx, int32_t gy) {
    uint32_t x = (uint32_t)(gx + hv::kGridHalf), y = (uint32_t)(gy + hv::kGridHalf);
    uint64_t d = 0;
    for (int i = 30; i >= 0; i--) {
        const uint32_t rx = (x >> i) & 1u, ry = (y >> i) & 1u;
        d = 4 * d + ((3u * rx) ^ ry);
        if (ry == 0) {
            if (rx == 1) x = ~x, y = ~y;
            const uint32_t t = x;
            x = y;
            y = t;
        }
    }
    return d;
}
static long bad = 0;
static void check(int32_t x, int32_t y) {
    const uint64_t k = by_levels(x, y);
    const int2 p = hv::hilbert_point(k);
    bad += hv::hilbert_key(x, y) != k || p.x != x || p.y != y;
}
int main() {
    const int32_t half = hv::kGridHalf, edge[8] = {-half, -half + 1, -1, 0, 1, half / 2, half - 2, half - 1};
    for (int a = 0; a < 8; a++)
        for (int b = 0; b < 8; b++) check(edge[a], edge[b]);
    for (int32_t x = 0; x < 64; x++)
        for (int32_t y = 0; y < 64; y++) check((x << 25) - half, (y << 25) - half), check(x - half, y - half), check(x - 32, y - 32);
    std::mt19937_64 rng(7);
    for (int i = 0; i < 2000000; i++) {
        const uint64_t v = rng();
        int32_t x = (int32_t)((uint32_t)(v & 0x7fffffff) >> (i % 31)) - half, y = (int32_t)((uint32_t)((v >> 32) & 0x7fffffff) >> (i % 29)) - half;
        check(i & 1 ? -1 - x : x, i & 4 ? -1 - y : y);
    }
    printf("bad %ld\n", bad);
}
"""


def test_hilbert_index_equals_its_level_by_level_definition(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "hilbert.cu", tmp_path / "hilbert"
    src.write_text(SOURCE)
    subprocess.run([nvcc, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                    os.path.join(ROOT, "paper_2005_12489_gb300", "csrc"), "-o", str(exe), str(src)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout == "bad 0\n"
