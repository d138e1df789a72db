// Device-side grid arithmetic and exact predicates (HiVision Sec. 3.2).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace hv {

constexpr unsigned kFull = 0xffffffffu;
constexpr int32_t kGridHalf = 1 << 30;
constexpr int32_t kEmptyLo = 0x7fffffff;          // min-corner of an empty box
constexpr int32_t kEmptyHi = (int32_t)0x80000000; // max-corner of an empty box

// Interleave with zeros: bit i moves to bit 2 i (and back).
__host__ __device__ inline uint64_t spread_bits(uint32_t v) {
    uint64_t x = v;
    x = (x | (x << 16)) & 0x0000ffff0000ffffull;
    x = (x | (x << 8)) & 0x00ff00ff00ff00ffull;
    x = (x | (x << 4)) & 0x0f0f0f0f0f0f0f0full;
    x = (x | (x << 2)) & 0x3333333333333333ull;
    return (x | (x << 1)) & 0x5555555555555555ull;
}
__host__ __device__ inline uint32_t squeeze_bits(uint64_t x) {
    x &= 0x5555555555555555ull;
    x = (x | (x >> 1)) & 0x3333333333333333ull;
    x = (x | (x >> 2)) & 0x0f0f0f0f0f0f0f0full;
    x = (x | (x >> 4)) & 0x00ff00ff00ff00ffull;
    x = (x | (x >> 8)) & 0x0000ffff0000ffffull;
    return (uint32_t)(x | (x >> 16));
}

// Hilbert curve index of (x, y) on a 2^31 grid (x, y shifted to [0, 2^31)),
// the quadrant-rotation curve; 62-bit result.
//
// Read top down, level i sees the bits (X, Y) of x and y, exchanged if s and
// complemented if c: rx = X ^ s (X ^ Y) ^ c, ry likewise; its digit is (3 rx) ^
// ry, and a digit with ry = 0 flips s, and c too if rx = 1.  Over GF(2) the
// step from one level's (s, c) to the next's is affine: with X = Y it is s ^ c ^
// !Y, c; else c ^ !Y, s ^ !Y.  So the states of all levels at once are a prefix
// composition of the levels' maps (s' = a s ^ b c ^ e, c' = d s ^ g c ^ f), a bit
// per level and word, in five doubling steps: about 150 instructions where the
// loop over 31 levels takes 370.
__host__ __device__ inline uint64_t hilbert_key(int32_t gx, int32_t gy) {
    // level 30 in bit 31
    const uint32_t X = (uint32_t)(gx + kGridHalf) << 1, Y = (uint32_t)(gy + kGridHalf) << 1;
    const uint32_t q = X ^ Y, n = ~Y;
    // the map of the level above (the top one's is the identity)
    uint32_t a = (~q >> 1) | 0x80000000u, b = ~0u >> 1, e = n >> 1;
    uint32_t d = q >> 1, g = (~q >> 1) | 0x80000000u, f = (n & q) >> 1;
#pragma unroll
    for (int k = 1; k < 32; k <<= 1) {
        const uint32_t top = ~(~0u >> k);
        const uint32_t a2 = (a >> k) | top, b2 = b >> k, e2 = e >> k;
        const uint32_t d2 = d >> k, g2 = (g >> k) | top, f2 = f >> k;
        const uint32_t na = (a & a2) ^ (b & d2), nb = (a & b2) ^ (b & g2), ne = (a & e2) ^ (b & f2) ^ e;
        const uint32_t nd = (d & a2) ^ (g & d2), ng = (d & b2) ^ (g & g2), nf = (d & e2) ^ (g & f2) ^ f;
        a = na, b = nb, e = ne, d = nd, g = ng, f = nf;
    }
    // from s = c = 0 above the top level the state is (e, f)
    const uint32_t flip = (q & e) ^ f, rx = X ^ flip, ry = Y ^ flip;
    return (spread_bits(rx >> 1) << 1) | spread_bits((rx ^ ry) >> 1);
}

// The grid point of a Hilbert index.  The digits give every level's flips of s
// and c directly, so the states are two prefix XORs.
__host__ __device__ inline int2 hilbert_point(uint64_t key) {
    const uint32_t rx = squeeze_bits(key >> 1), ry = rx ^ squeeze_bits(key);
    uint32_t s = ~ry & 0x7fffffffu, c = s & rx;
    s >>= 1;
    c >>= 1;
#pragma unroll
    for (int k = 1; k < 32; k <<= 1) {
        s ^= s >> k;
        c ^= c >> k;
    }
    const uint32_t u = rx ^ c, v = ry ^ c, w = (u ^ v) & s;
    int2 p;
    p.x = (int32_t)(u ^ w) - kGridHalf;
    p.y = (int32_t)(v ^ w) - kGridHalf;
    return p;
}

// Centre of a box, rounded down, computed without overflow.
__host__ __device__ inline int32_t mid32(int32_t a, int32_t b) {
    return (int32_t)(((int64_t)a + (int64_t)b) >> 1);
}

// Unsigned 64 x 64 -> 128-bit product compare: a*a <= b*c.
__device__ __forceinline__ bool sq_le_prod(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t lo1 = a * a, hi1 = __umul64hi(a, a);
    uint64_t lo2 = b * c, hi2 = __umul64hi(b, c);
    return hi1 < hi2 || (hi1 == hi2 && lo1 <= lo2);
}

// Distance from s to the closed segment [a, b] is <= R.  With d = b - a,
// w = s - a, t = w.d and L = d.d the nearest point is a when t <= 0, b when
// t >= L, and otherwise the squared distance is (w x d)^2 / L, compared as
// (w x d)^2 <= R^2 L in 128 bits (|w x d| < 2^63, R^2 L < 2^121).
__device__ __forceinline__ bool segment_within(int32_t ax, int32_t ay, int32_t bx, int32_t by,
                                               int32_t sx, int32_t sy, int64_t R2) {
    int64_t dx = (int64_t)bx - ax, dy = (int64_t)by - ay;
    int64_t wx = (int64_t)sx - ax, wy = (int64_t)sy - ay;
    int64_t t = wx * dx + wy * dy;
    if (t <= 0) return wx * wx + wy * wy <= R2;
    int64_t L = dx * dx + dy * dy;
    if (t >= L) {
        int64_t ex = (int64_t)sx - bx, ey = (int64_t)sy - by;
        return ex * ex + ey * ey <= R2;
    }
    int64_t cr = wx * dy - wy * dx;
    uint64_t c = (uint64_t)(cr < 0 ? -cr : cr);
    return sq_le_prod(c, (uint64_t)R2, (uint64_t)L);
}

__device__ __forceinline__ bool box_hit(int4 b, int32_t x0, int32_t y0, int32_t x1, int32_t y1) {
    return b.x <= x1 && b.z >= x0 && b.y <= y1 && b.w >= y0;
}

}  // namespace hv
