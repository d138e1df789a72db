"""The arithmetic of the render kernel's strip sweep (hv_sweep.cuh up to the
traversal, and the predicates of hv_device.cuh) compiled for the host, so that
tests run the code itself and not a copy.  The device's approximate root,
reciprocal root and reciprocal are replaced by the correctly rounded ones with a
random relative error of at most 2^-22; warp-wide functions are declared only.
Integers wrap as on the device."""
import ctypes
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2005_12489_gb300", "csrc")

SHIM = r"""
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <random>
using std::max; using std::min;
#define __device__
#define __host__
#define __forceinline__ inline
#define __noinline__ inline
struct int2 { int x, y; };
struct int4 { int x, y, z, w; };
struct float4 { float x, y, z, w; };
inline int2 make_int2(int x, int y) { return {x, y}; }
inline int4 make_int4(int x, int y, int z, int w) { return {x, y, z, w}; }
inline float4 make_float4(float x, float y, float z, float w) { return {x, y, z, w}; }
static int64_t g_tests = 0;   // exact tests of samples, and sides taken
template <class T> T __ldg(const T* p) { return *p; }
inline float __int_as_float(int v) { float f; memcpy(&f, &v, 4); return f; }
inline float __uint_as_float(uint32_t v) { float f; memcpy(&f, &v, 4); return f; }
inline uint32_t __float_as_uint(float v) { uint32_t u; memcpy(&u, &v, 4); return u; }
inline int to_int(double v) { return v != v ? 0 : v >= 2147483647.0 ? 2147483647 : v <= -2147483648.0 ? (-2147483647 - 1) : (int)v; }
inline int __float2int_ru(float v) { return to_int(std::ceil((double)v)); }
inline int __float2int_rd(float v) { return to_int(std::floor((double)v)); }
inline float __fdividef(float a, float b) { return a / b; }
inline int __ffs(uint32_t v) { return v ? __builtin_ctz(v) + 1 : 0; }
inline int __clz(uint32_t v) { return v ? __builtin_clz(v) : 32; }
inline int __popc(uint32_t v) { return __builtin_popcount(v); }
inline uint64_t __umul64hi(uint64_t a, uint64_t b) { return (uint64_t)(((unsigned __int128)a * b) >> 64); }
inline uint32_t atomicOr(uint32_t* p, uint32_t v) { const uint32_t o = *p; *p |= v; return o; }
inline uint32_t atomicXor(uint32_t* p, uint32_t v) { const uint32_t o = *p; *p ^= v; return o; }
uint32_t __ballot_sync(uint32_t, bool); bool __any_sync(uint32_t, bool); void __syncwarp();
uint32_t __reduce_or_sync(uint32_t, uint32_t);
template <class T> T __shfl_sync(uint32_t, T, int); template <class T> T __shfl_up_sync(uint32_t, T, int);
static std::mt19937_64 g_err(1);
inline float off(double v) { return (float)(v * (1.0 + ((int)(g_err() % 3) - 1) * 0x1p-22)); }
inline float host_sqrt(float x) { return off(std::sqrt((double)x)); }
inline float host_rsqrt(float x) { return off(1.0 / std::sqrt((double)x)); }
inline float host_rcp(float x) { return off(1.0 / (double)x); }
constexpr uint32_t kFull = ~0u;
constexpr int HV_LAYER_POINTS = 0, HV_LAYER_LINES = 1, HV_LAYER_POLYGONS = 2, kPolyFill = 3;
constexpr int kWarps = 8, kThreads = 256, kStripRows = 16, kTile = 256, kMaxLevels = 16;
constexpr uint32_t kLogNode = 0, kLogLeaf = 1, kLogPolyNode = 2, kLogPolyLeaf = 3, kLogPoly = 4;
struct Front {};
struct Params { const int4* poly_edges; const uint64_t* poly_edge_off; uint64_t n_poly, n_edges; };
struct Src { const void* obj; const uint32_t* ids; uint64_t n; };
void log_read(const Params&, uint32_t, uint64_t, int); void check_failed(const Params&, uint32_t, uint64_t);
"""


def source():
    """The host form of the two files."""
    dev = open(os.path.join(CSRC, "hv_device.cuh")).read()
    sweep = open(os.path.join(CSRC, "hv_sweep.cuh")).read()
    dev = dev[dev.index("constexpr int32_t kGridHalf"):dev.rindex("}  // namespace hv")].replace(
        "constexpr uint32_t kFull = 0xffffffffu;", "")
    sweep = sweep[sweep.index("constexpr int kBitStride"):sweep.index("// ---- traversal")]
    sweep = re.sub(r'asm\("shl\.b32[^;]*;[^;]*;', "r = (uint32_t)n > 31u ? 0u : v << n;", sweep)
    sweep = re.sub(r'asm\("(sqrt|rsqrt|rcp)\.[^;]*;[^;]*;', r"r = host_\1(x);", sweep)
    assert "asm(" not in sweep
    return SHIM + re.sub(r"((?:bool segment_within|int side_of_nearest)\([^)]*\) \{)", r"\1 g_tests++;", dev + sweep)


def library(tmp_path, entries):
    """Compile the host form and `entries` (C++ with extern "C" functions) and load it."""
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    src, so = tmp_path / "sweep_host.cpp", tmp_path / "sweep_host.so"
    src.write_text(source() + entries)
    subprocess.run([cxx, "-O2", "-std=c++17", "-fwrapv", "-ffp-contract=off", "-w", "-fPIC", "-shared", "-o", str(so),
                    str(src)], check=True)
    return ctypes.CDLL(str(so))
