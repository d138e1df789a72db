// Strip sweep: Algorithm 1 (SIBV) and Algorithm 2 (SIBF) over a strip, object
// by object.
//
// The samples of a strip form one lattice: the four super-samples of a pixel
// sit at a quarter of the pixel size from its centre, so together they are a
// square grid of spacing ps / 2 (MASK mode: the pixel centres, spacing ps).
// The strip keeps one bit per sample in shared memory.  An object within
// distance R of a sample is, per sample row, within one interval of columns
// (the set of points within R of a point, or of a segment, is convex), so an
// object is drawn by one exact interval per row it reaches, ORed into the
// bits.  Each leaf of the index is read once per strip, instead of once per
// 8 x 4 pixel block that it reaches, and only while a sample that it can reach
// is still open; inner nodes and frontier entries are pruned by the same test.
//
// Bound: instruction issue for points and outlines (71% and 68% of the slots busy);
// segments and fill (53%, 50%), with few leaves per strip, wait at barriers and for
// their reads.  DRAM 5 to 11% of the measured copy rate.  Drawn by strips, 600
// tiles of 100M clustered points at 2 px take 2.4 M warp instructions per tile
// where the 8 x 4 block traversal took 5.7 M: 4,000 tiles 23.5 -> 11 ms; 341 tiles of
// 100,000 points at zoom 0-4, 1 px, MASK 414 -> 72 us; 36 single tiles of 10M
// points 1,340 -> 776 us in all.  Segments: 4,000 tiles of 50M segments at 1 px
// 19.7 -> 5.5 ms; the outlines of 1,000 tiles of 2M polygons 12 -> 8.5 ms (dense
// low-zoom tiles: 390 leaves of short edges per strip, 22 pieces and 71 (piece, row)
// pairs each).
//
// The fill draws polygon by polygon: one pass over a polygon's edges gives every
// crossing of the strip's rows, and a parity scan per row the filled samples.
// 1,000 tiles of 2M polygons: the fill launch 3.5 -> 1.3 ms, both 12.4 -> 10.0
// ms; 33 tiles with anti-aliased pattern fill 525 -> 360 us.
//
// Included by hv_render.cu (one translation unit with the cull).
#pragma once

constexpr int kBitStride = 17;   // words per sample row: 512 columns and a pad word (row-parallel reads then hit 32 banks)
constexpr int kSampleRows = 2 * kStripRows;
static_assert(kSampleRows <= 32, "one lane per sample row");

template <int kKind>
struct SweepSmem : Front {
    // polygon outlines: the fill launch's results, and the composed ones for the encode
    uint8_t res[kKind == HV_LAYER_POLYGONS ? kStripRows * kTile : 16];
    // polygon fill: per warp, the crossings of one polygon's edges, a bit per column and row
    uint32_t cross[kKind == kPolyFill ? kWarps : 1][kKind == kPolyFill ? kSampleRows * kBitStride : 1];
    uint32_t bits[kSampleRows * kBitStride];
    int32_t reach[64];
    uint32_t stk_node[kWarps][kMaxLevels + 1];
    uint32_t stk_mask[kWarps][kMaxLevels + 1];
    // per warp, what the (piece, row) or (edge, row) pairs of 32 objects share
    float4 pair_obj[kWarps][kKind == HV_LAYER_POINTS ? 1 : (kKind == kPolyFill ? 32 : 64)];
    int pair_row[kWarps][kKind == HV_LAYER_POINTS ? 1 : 32];
    int next_entry;
};

// Pairs (object, row) of a warp, numbered through over the objects that have
// rows: `start` is the lane's first pair.  The objects lie in shared memory in order,
// those without rows left out, so that a pair's object is the number of starts up to it: in
// each round of 32 pairs one OR over the lanes marks the starts in it and the
// bits up to the lane's own are counted.  (A binary search over the starts with
// shuffles, and the object's fields by shuffles as well, took 15 shuffles a round
// and held the fields in registers, spilling 96 bytes in the outline launch
// against 52: 4,000 tiles of 50M segments 5.84 ms against 5.57, 1,000 tiles of
// 2M polygons 10.38 ms against 9.96.)
struct PairRounds {
    int start, before;
    bool some;
    __device__ PairRounds(int start_, int count) : start(start_), before(0), some(count > 0) {}
    // the object of pair base + lane, base = 0, 32, ..
    __device__ __forceinline__ int object(int base, int lane) {
        const int at = start - base;
        const uint32_t marks = __reduce_or_sync(kFull, some && (uint32_t)at < 32u ? 1u << at : 0u);
        const int k = before + __popc(marks & ((2u << lane) - 1u)) - 1;
        before += __popc(marks);
        return k;
    }
};

// Inclusive prefix sum over the lanes.
__device__ __forceinline__ int lane_sums(int v, int lane) {
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int u = __shfl_up_sync(kFull, v, d);
        if (lane >= d) v += u;
    }
    return v;
}

// The CTA's samples: (i, j) lies at (xc + (i - hw) h, yc + (j - hh) h), h = 2^s.
// Objects are taken relative to (xc, yc), the strip's middle, so that every
// difference that matters fits 32 bits: an object that reaches a sample lies
// within 2^30 + 2^22 of the middle along each axis (zoom 0: inside the grid;
// zoom >= 1: half the strip plus R is at most 2^30), and farther coordinates
// are clamped to that, which leaves them out of reach.
struct Lattice {
    int s, hw, hh;      // log2 of the spacing; half the columns and rows
    int32_t xc, yc;
    int32_t R;
    int64_t R2;
    int rs;             // R >> rs <= 63
    bool narrow;        // R <= kNarrow: squares fit 32 bits
};

constexpr int32_t kNarrow = 46340;   // floor(sqrt(2^31))
constexpr int kTableReach = 16;      // spacings
constexpr int32_t kRelMax = (1 << 30) + (1 << 22);

__device__ __forceinline__ int32_t rel32(int32_t v, int32_t c) { return max(min(v - c, kRelMax), -kRelMax); }

__device__ __forceinline__ float sqrt_approx(float x) {
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// floor(sqrt(B)), 0 <= B < 2^31.  The approximate root is off by less than
// 2^-22 of itself (conversion 2^-24, root 2^-23): scaled up by 2^-21 it is at
// least sqrt(B) and less than sqrt(B) + 0.05, so its integer part is the root
// or one above it.
__device__ __forceinline__ uint32_t isqrt_narrow(uint32_t B) {
    uint32_t w = (uint32_t)(sqrt_approx((float)B) * (1.f + 0x1p-21f));
    if (w * w > B) w--;
    return w;
}

// floor(sqrt(B)), 0 <= B <= 2^58: one Newton step from the single-precision
// root (off by at most 2^-21 of itself, so the step leaves an error below
// one unit), then the exact neighbour.
__device__ __forceinline__ uint32_t isqrt_wide(uint64_t B) {
    const float f = sqrt_approx((float)B);
    const int32_t w0 = (int32_t)f;
    const int64_t r = (int64_t)B - (int64_t)w0 * w0;
    int32_t w = w0 + (int32_t)floorf(__fdividef((float)r, 2.f * fmaxf(f, 1.f)));
    w = max(w, 0);
    if ((uint64_t)w * (uint64_t)w > B) w--;
    else if ((uint64_t)(w + 1) * (uint64_t)(w + 1) <= B) w++;
    return (uint32_t)w;
}

// A half-width of the columns that are within R of a row at distance f <= R,
// for a box [x0, x1]: floor(sqrt(R^2 - f^2)), or with a wide R any value that
// gives the same columns floor((x0 + w) / h) and ceil((x1 - w) / h).  Then
// (R - f)(R + f) in single precision keeps its relative error (three roundings
// and the root's: under 2^-21 of w) whatever cancels, so w lies within
// wl..wh; nearly always both give the same columns, and the exact root is
// taken only where they do not (a few in 10^4 at 2 px; 64-bit squares for
// every row made the zoom levels with R > 46340 the slowest).
template <bool kNarrowR>
__device__ __forceinline__ int32_t half_width(const Lattice& g, int32_t f, int32_t x0, int32_t x1) {
    if (kNarrowR) return (int32_t)isqrt_narrow((uint32_t)g.R2 - (uint32_t)(f * f));
    const float w = sqrt_approx((float)(g.R - f) * (float)(g.R + f));
    const int32_t wl = max((int32_t)(w * (1.f - 0x1p-20f)) - 1, 0), wh = (int32_t)(w * (1.f + 0x1p-20f)) + 1;
    if (((x0 + wl) >> g.s) != ((x0 + wh) >> g.s) || ((wl - x1) >> g.s) != ((wh - x1) >> g.s))
        return (int32_t)isqrt_wide((uint64_t)(g.R2 - (int64_t)f * f));
    return wl;
}

// Columns of sample row `row` (bits of its words): set [lo, hi], 0 <= lo <= hi.
// Bits that are set already are left alone (a plain read first: most words
// that meet dense data are full, and the reads of one word are a broadcast
// where the atomics would queue).  True if a bit of them was not set: this and the
// functions that draw objects report it to the phase profile, which counts the leaf
// visits that decided a sample; elsewhere nothing reads it.
__device__ __forceinline__ bool set_bits(uint32_t* word, uint32_t m) {
    return (m & ~*(volatile uint32_t*)word) && (m & ~atomicOr(word, m));
}
__device__ __forceinline__ bool set_columns(uint32_t* row, int lo, int hi) {
    const int k0 = lo >> 5, k1 = hi >> 5;
    uint32_t m = ~0u << (lo & 31);
    const uint32_t last = ~0u >> (31 - (hi & 31));
    bool fresh = false;
    for (int k = k0; k < k1; k++) {
        fresh |= set_bits(row + k, m);
        m = ~0u;
    }
    m &= last;
    return set_bits(row + k1, m) | fresh;
}

// Set the samples that lie within R of every point of the lane's box
// [x0, x1] x [y0, y1] (relative coordinates): exactly the covered samples of
// a point (x0 = x1, y0 = y1), and samples certainly covered when the box holds
// at least one point.  In row y the farthest row distance is f = max(|y - y0|,
// |y - y1|), and with w = floor(sqrt(R^2 - f^2)) the columns are [x1 - w, x0 + w].
// Only the rows of `open` (a bit per sample row) are drawn.
template <bool kNarrowR>
__device__ __forceinline__ bool splat(uint32_t* bits, const Lattice& g, int32_t x0, int32_t y0, int32_t x1,
                                      int32_t y1, uint32_t open) {
    const int r0 = max(g.hh - ((g.R - y1) >> g.s), 0);
    const int r1 = min(((y0 + g.R) >> g.s) + g.hh, 2 * g.hh - 1);
    if (r0 > r1) return false;
    open &= (~0u << r0) & (~0u >> (31 - r1));
    bool fresh = false;
    while (open) {
        const int r = __ffs(open) - 1;
        open &= open - 1;
        const int32_t y = (r - g.hh) << g.s;
        const int32_t f = max(abs(y - y0), abs(y - y1));
        const int32_t w = half_width<kNarrowR>(g, f, x0, x1);
        const int lo = max(g.hw - ((w - x1) >> g.s), 0), hi = min(((x0 + w) >> g.s) + g.hw, 2 * g.hw - 1);
        if (lo <= hi) fresh |= set_columns(bits + r * kBitStride, lo, hi);
    }
    return fresh;
}

// The half-widths of reach by row distance, for the tests that only need an
// upper bound: reach[k] >= floor(sqrt(R^2 - f^2)) for every f with f >> rs = k,
// where rs makes R >> rs at most 63.  (Single precision, rounded up, the
// factors formed as integers: a radius above 2^24 need not be a float, and
// its rounding could cancel all of R - f.  A table read in place of a root per
// row.)
__device__ __forceinline__ void fill_reach(int32_t* reach, const Lattice& g, int tid) {
    if (tid <= (g.R >> g.rs)) {
        const int32_t f = tid << g.rs;
        reach[tid] = min((int32_t)(sqrt_approx((float)(g.R - f) * (float)(g.R + f)) * (1.f + 0x1p-19f)) + 1, g.R);
    }
}

// An upper bound of the half-width at row distance f <= R.  The table's is off by up
// to about R f / 64 w: with R of many spacings that is columns, in which samples
// outside every object's reach stay open and keep boxes from being pruned.  There
// (kFine) a root is taken, good to 2^-19.  300 tiles of 200,000 crowded points at
// 64 px 9.56 -> 0.35 ms, of 50,000 polygons' outlines 28.1 -> 1.87 ms; as a branch taken
// for each row instead of an instantiation 4,000 tiles of 100M points at 2 px lose 7%.
// From kTableReach = 16 spacings on, where the table is off by a quarter of a column (616
// calls with radii of 12 to 64 px: 221 ms in all, 272 from 32 spacings on, 456 from 64).
template <bool kFine>
__device__ __forceinline__ int32_t reach_width(const int32_t* reach, const Lattice& g, int32_t f) {
    if (!kFine) return reach[f >> g.rs];
    return min((int32_t)(sqrt_approx((float)(g.R - f) * (float)(g.R + f)) * (1.f + 0x1p-19f)) + 1, g.R);
}

// Is a sample of columns lo..hi of the row open?
__device__ __forceinline__ bool columns_open(const uint32_t* row, int lo, int hi) {
    const int k1 = hi >> 5;
    uint32_t m = ~0u << (lo & 31);
    for (int k = lo >> 5; k < k1; k++) {
        if (m & ~*(volatile const uint32_t*)(row + k)) return true;
        m = ~0u;
    }
    return (m & (~0u >> (31 - (hi & 31))) & ~*(volatile const uint32_t*)(row + k1)) != 0u;
}

// Is a sample of the row within [x0 - w, x1 + w] open?
__device__ __forceinline__ bool row_open(const uint32_t* row, const Lattice& g, int32_t x0, int32_t x1, int32_t w) {
    const int lo = max(g.hw - ((w - x0) >> g.s), 0), hi = min(((x1 + w) >> g.s) + g.hw, 2 * g.hw - 1);
    return lo <= hi && columns_open(row, lo, hi);
}

// Sample rows (one lane each) with an open sample that an object inside the
// box could cover: within R of the box (rounded up).  Zero: nothing below the
// box matters.
template <bool kFine>
__device__ __forceinline__ uint32_t open_rows(const uint32_t* bits, const int32_t* reach, const Lattice& g, int32_t x0,
                                              int32_t y0, int32_t x1, int32_t y1, int lane) {
    const int32_t y = (lane - g.hh) << g.s;
    const int32_t f = max(max(y0 - y, y - y1), 0);
    const bool open = lane < 2 * g.hh && f <= g.R && row_open(bits + lane * kBitStride, g, x0, x1, reach_width<kFine>(reach, g, f));
    return __ballot_sync(kFull, open);
}

// open_rows for the lane's own box: is any sample in reach open (in one of
// the given rows)?  One pass for the 32 children of a node; those that pass
// take open_rows again when their turn comes, after their siblings.
template <bool kFine>
__device__ __forceinline__ bool box_open(const uint32_t* bits, const int32_t* reach, const Lattice& g, int32_t x0,
                                         int32_t y0, int32_t x1, int32_t y1, uint32_t rows) {
    const int r0 = max(g.hh - ((g.R - y0) >> g.s), 0), r1 = min(((y1 + g.R) >> g.s) + g.hh, 2 * g.hh - 1);
    if (r0 > r1) return false;
    rows &= (~0u << r0) & (~0u >> (31 - r1));
    while (rows) {
        const int r = __ffs(rows) - 1;
        rows &= rows - 1;
        const int32_t y = (r - g.hh) << g.s;
        if (row_open(bits + r * kBitStride, g, x0, x1, reach_width<kFine>(reach, g, max(max(y0 - y, y - y1), 0)))) return true;
    }
    return false;
}

// Shifts that give 0 for amounts of 32 (the C operator leaves those undefined).
__device__ __forceinline__ uint32_t shl32(uint32_t v, int n) {
    uint32_t r;
    asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(n));
    return r;
}

// The same samples as splat for 32 boxes whose reach together is at most 32
// columns wide, from column c0 on: per open row each lane forms its box's
// columns as one word and the warp's OR is the row's new coverage, kept by the
// lane of that number and merged into the bits once.  A row costs about half
// of one in splat (no clipping, one atomic for 32 boxes, no queue of
// atomics on the same word where the boxes crowd), but every lane takes part
// in every row.
template <bool kNarrowR>
__device__ __forceinline__ bool splat_window(uint32_t* bits, const Lattice& g, int32_t x0, int32_t y0, int32_t x1,
                                             int32_t y1, int c0, bool active, uint32_t rows, int lane) {
    bool fresh = false;
    const int32_t origin = (c0 - g.hw) * (1 << g.s);
    x0 -= origin;
    x1 -= origin;
    uint32_t acc = 0u;
    while (rows) {
        const int r = __ffs(rows) - 1;
        rows &= rows - 1;
        const int32_t y = (r - g.hh) << g.s;
        const int32_t f = max(abs(y - y0), abs(y - y1));
        uint32_t m = 0u;
        if (active && f <= g.R) {
            const int32_t w = half_width<kNarrowR>(g, f, x0, x1);
            // columns ceil((x1 - w) / h) .. floor((x0 + w) / h), within 0 .. 31; an
            // empty interval ends one before its start, or earlier (a box too wide)
            const int lo = -((w - x1) >> g.s), end = ((x0 + w) >> g.s) + 1;
            if (lo < end) m = shl32(1u, end) - shl32(1u, lo);
        }
        m = __reduce_or_sync(kFull, m);
        if (lane == r) acc = m;
    }
    if (acc) {
        const int k = c0 >> 5, sh = c0 & 31, words = g.hw >> 4;
        uint32_t* row = bits + lane * kBitStride;
        const uint32_t a = acc << sh, b = sh ? acc >> (32 - sh) : 0u;
        if (k >= 0 && k < words) fresh |= set_bits(row + k, a);
        if (k + 1 >= 0 && k + 1 < words) fresh |= set_bits(row + k + 1, b);
    }
    return fresh;
}

// A box of points is worth drawing when it is no wider than about R (the
// samples that a larger one certainly covers are few or none).
__device__ __forceinline__ bool small_box(const Lattice& g, int32_t x0, int32_t y0, int32_t x1, int32_t y1) {
    const uint32_t most = (uint32_t)g.R + (uint32_t)(g.R >> 2);
    return (uint32_t)(x1 - x0) <= most && (uint32_t)(y1 - y0) <= most;
}

// Is every sample of the strip within R of every point of the box (relative
// coordinates)?  In single precision and with its rounding to spare: a box that only just
// covers the strip is drawn like any other.
__device__ __forceinline__ bool covers_strip(const Lattice& g, int32_t x0, int32_t y0, int32_t x1, int32_t y1) {
    const float h = (float)(1 << g.s), hw = (float)g.hw * h, hh = (float)g.hh * h, R = (float)g.R * (1.f - 0x1p-20f);
    const float dx = fmaxf((float)x1 + hw, hw - (float)x0), dy = fmaxf((float)y1 + hh, hh - (float)y0);
    return fmaf(dx, dx, dy * dy) <= R * R;
}

// ---- segments ---------------------------------------------------------------

// A piece of a segment as its row intervals see it, in sample spacings relative
// to the lattice point (col, row) in the middle of the part of the piece's
// box that lies in the strip's reach: the unit direction m (my >= 0), the
// line's signed offset c0 = m x a and the positions ta <= tb of the segment's
// ends along m.  |E| bounds the rounding of everything below as a distance from
// the segment; negative: the contact points are not to be relied on, and every sample
// that may be within R of the line is decided exactly (-infinite: nor is the line).
struct PieceRow {
    float mx, my, c0, ta, tb, E;
    uint32_t at;      // col + 1024 | (row + 1024) << 16
    uint32_t span;    // columns within Chebyshev distance R of the box: first | last << 16
};

__device__ __forceinline__ float rsqrt_approx(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ uint32_t magnitude(int32_t v) { return v < 0 ? 0u - (uint32_t)v : (uint32_t)v; }

// The line's offset and the nearer end's position along it (from either end
// the offset is the same; the far end lies |d| beyond the near one).  Inside
// the reach every coordinate is at most M = the visible box's size + R / h + 3;
// a near end within 4 M is taken in single precision, one farther away from
// exact int64 products rounded once, and ends beyond 8 M are cut off there,
// where they no longer matter.  Root and quotient are good to 2^-22, so the
// interval ends that draw_row finds are off by fewer than 16 roundings of
// 2^-22 M; E = 2^-17 M.  The contact point's position t = (..) / my is the one
// step that a small my magnifies; its error acts squared over 2 R, and
// pieces too level for that to stay below E (but not exactly level ones, whose
// contact points are the ends) are left to the exact test; so are most lines that
// pass the strip at a distance (a long piece's box is wide), all with R = 0.
__device__ __forceinline__ PieceRow piece_row(const Lattice& g, int4 o, int32_t x0, int32_t y0, int32_t x1, int32_t y1,
                                              int clo, int chi) {
    PieceRow q;
    const int ex0 = max(x0 >> g.s, -g.hw - 1), ex1 = min(x1 >> g.s, g.hw);
    const int ey0 = max(y0 >> g.s, -g.hh - 1), ey1 = min(y1 >> g.s, g.hh);
    // (a box beyond one side of the strip: the middle of what is left, near it)
    const int mc = max(min((ex0 + ex1) >> 1, g.hw), -g.hw - 1), mr = max(min((ey0 + ey1) >> 1, g.hh), -g.hh - 1);
    q.at = (uint32_t)(mc + g.hw + 1024) | ((uint32_t)(mr + g.hh + 1024) << 16);
    q.span = (uint32_t)clo | ((uint32_t)chi << 16);
    const float scale = __int_as_float((127 - g.s) << 23);   // 1 / h
    const float rho = (float)g.R * scale;
    const float Y = (float)max(ey1 - ey0, 0) + rho + 3.f;
    const float M = fmaxf((float)max(ex1 - ex0, 0) + rho + 3.f, Y);
    q.E = 0x1p-17f * M;
    if (o.w < o.y || (o.w == o.y && o.z < o.x)) o = make_int4(o.z, o.w, o.x, o.y);
    // relative to the middle, wrapping: a value that wraps is still beyond 2^29,
    // by its magnitude as an unsigned number (a difference of 2^31 has none as an int)
    const uint32_t ox = (uint32_t)g.xc + (uint32_t)(mc << g.s), oy = (uint32_t)g.yc + (uint32_t)(mr << g.s);
    const int32_t ax = (int32_t)((uint32_t)o.x - ox), ay = (int32_t)((uint32_t)o.y - oy);
    const int32_t bx = (int32_t)((uint32_t)o.z - ox), by = (int32_t)((uint32_t)o.w - oy);
    const int32_t dx = o.z - o.x, dy = o.w - o.y;
    const float fx = (float)dx * scale, fy = (float)dy * scale;
    const float L2 = fmaf(fx, fx, fy * fy);
    const float inv = L2 > 0.f ? rsqrt_approx(L2) : 0.f, D = L2 * inv;
    q.mx = L2 > 0.f ? fx * inv : 1.f;
    q.my = fy * inv;
    const uint32_t fa = max(magnitude(ax), magnitude(ay)), fb = max(magnitude(bx), magnitude(by));
    bool from_a = fa <= fb;
    float near_t;
    const uint32_t fn = min(fa, fb);
    if (fn < (1u << 29) && (float)fn * scale <= 4.f * M) {
        const float nx = (float)(from_a ? ax : bx) * scale, ny = (float)(from_a ? ay : by) * scale;
        q.c0 = q.mx * ny - q.my * nx;
        near_t = fmaf(q.mx, nx, q.my * ny);
    } else {
        const int64_t wx = (int64_t)g.xc + ((int64_t)mc << g.s), wy = (int64_t)g.yc + ((int64_t)mr << g.s);
        const int64_t pa = max(llabs(o.x - wx), llabs(o.y - wy)), pb = max(llabs(o.z - wx), llabs(o.w - wy));
        from_a = pa <= pb;
        const int64_t nx = (from_a ? o.x : o.z) - wx, ny = (from_a ? o.y : o.w) - wy;
        // |d| < 2^31 and |n| <= 1.5 * 2^30 keep the sums below 2^63 (beyond: exact tests)
        const float k = inv * scale;
        q.c0 = (float)(dx * ny - dy * nx) * scale * k;
        near_t = (float)(dx * nx + dy * ny) * scale * k;
        if (min(pa, pb) > 3ll << 29) q.E = -__int_as_float(0x7f800000);
    }
    q.ta = from_a ? near_t : near_t - D;
    q.tb = from_a ? near_t + D : near_t;
    q.ta = fmaxf(fminf(q.ta, 8.f * M), -8.f * M);
    q.tb = fmaxf(fminf(q.tb, 8.f * M), -8.f * M);
    const float G = Y + fabsf(q.c0) + rho;
    if (q.my > 0.f && q.my * q.my * rho * M * 0x1p25f < 4.f * G * G) q.E = -fabsf(q.E);
    return q;
}

// Exact test of one sample (column i of row r), unless it is set already.
__device__ __forceinline__ bool test_sample(uint32_t* bits, const Lattice& g, const int4* seg, int i, int r) {
    uint32_t* word = bits + r * kBitStride + (i >> 5);
    if ((*(volatile uint32_t*)word >> (i & 31)) & 1u) return false;
    const int4 o = __ldg(seg);
    if (!segment_within(o.x, o.y, o.z, o.w, g.xc + (i - g.hw) * (1 << g.s), g.yc + (r - g.hh) * (1 << g.s), g.R2))
        return false;
    return !((atomicOr(word, 1u << (i & 31)) >> (i & 31)) & 1u);
}

// The capsule of radius r around a segment meets a row in one interval.  Its
// left end belongs to the disc around the contact point t = (y - c0 mx - r mx)
// / my, cut off at the segment's ends (the leftmost point in the row of that
// disc if it reaches the row; if it does not, neither does the capsule), and
// the right end likewise with + r mx.
//
// draw_row_slow: the rows that graze the capsule, where an end moves by much
// more than a rounding for one.  Columns inside the interval of radius R - E are
// covered, columns outside that of R + E are not, and those between take the exact
// test.  And pieces with a negative E: the columns within R + |E| of the line,
// (mx y - c0 -+ (R + |E|)) / my, take the exact test.  (With all columns of the piece's
// box tested 60 tiles of 2,000 grid-wide segments took 7.9 ms at R = 0, now 0.06 ms.)
// (Without kProf the result is false.)
template <bool kProf>
__device__ __noinline__ bool draw_row_slow(uint32_t* bits, const Lattice& g, const PieceRow q, const int4* seg, int r) {
    const int col = (int)(q.at & 0xffffu) - 1024, row = (int)(q.at >> 16) - 1024;
    const int clo = (int)(q.span & 0xffffu) - col, chi = (int)(q.span >> 16) - col;
    const float rho = (float)g.R * __int_as_float((127 - g.s) << 23);
    const float inv = rcp_approx(q.my);
    bool fresh = false;
    if (q.my == 0.f) {
        // a level segment (or a point): the row's distance is a whole number, which decides
        // the row at once (tested, a long one that grazes the row leaves 512 columns to
        // one lane: 60 us in a tile that took 46 without)
        const int4 o = __ldg(seg);
        const int32_t f = abs(rel32(o.y, g.yc) - (r - g.hh) * (1 << g.s));
        if (f > g.R) return false;
        const int32_t w = (int32_t)isqrt_wide((uint64_t)(g.R2 - (int64_t)f * f));
        const int c0 = max(g.hw - ((w - rel32(min(o.x, o.z), g.xc)) >> g.s), clo + col);
        const int c1 = min(((rel32(max(o.x, o.z), g.xc) + w) >> g.s) + g.hw, chi + col);
        return c0 <= c1 && set_columns(bits + r * kBitStride, c0, c1) && kProf;
    }
    if (q.E < 0.f) {
        // (beyond 4 M = 2^19 |E| there are no samples; 0 / 0 leaves a side open, and
        // the quotients are good to 2^-21 of themselves)
        const float w = rho - q.E, A = fmaf(q.mx, (float)(r - row), -q.c0), lim = -q.E * 0x1p19f;
        const float v0 = fminf(fmaxf((A - w) * inv, -lim), lim), v1 = fmaxf(fminf((A + w) * inv, lim), -lim);
        const int c0 = __float2int_ru(fmaxf(fmaf(fabsf(v0), -0x1p-20f, v0), (float)clo));
        const int c1 = __float2int_rd(fminf(fmaf(fabsf(v1), 0x1p-20f, v1), (float)chi));
        for (int c = c0; c <= c1; c++) fresh |= test_sample(bits, g, seg, c + col, r);
        return kProf && fresh;
    }
    const float ym = (float)(r - row) - q.c0 * q.mx, xm = q.c0 * q.my;
    int lo[2], hi[2];
    bool met[2];
#pragma unroll
    for (int k = 0; k < 2; k++) {
        const float rad = k ? rho - q.E : rho + q.E, r2 = rad * rad, rm = rad * q.mx;
        const float tl = fminf(fmaxf((ym - rm) * inv, q.ta), q.tb), tr = fminf(fmaxf((ym + rm) * inv, q.ta), q.tb);
        const float dl = fmaf(-tl, q.my, ym), dr = fmaf(-tr, q.my, ym);
        // (a graze: the half-chord's square is rounding alone, widened outside)
        const float wide = k ? 0.f : rad * q.E;
        const float al = fmaf(-dl, dl, r2) + wide, ar = fmaf(-dr, dr, r2) + wide;
        lo[k] = max(__float2int_ru(fmaf(tl, q.mx, -xm) - sqrt_approx(fmaxf(al, 0.f))), clo);
        hi[k] = min(__float2int_rd(fmaf(tr, q.mx, -xm) + sqrt_approx(fmaxf(ar, 0.f))), chi);
        met[k] = k ? rad > 0.f && fminf(al, ar) >= 0.f : fmaxf(al, ar) >= 0.f;
    }
    if (!met[0] || lo[0] > hi[0]) return false;
    lo[1] = max(lo[1], lo[0]);
    hi[1] = min(hi[1], hi[0]);
    if (met[1] && lo[1] <= hi[1])
        fresh = set_columns(bits + r * kBitStride, lo[1] + col, hi[1] + col);
    else
        lo[1] = hi[0] + 1, hi[1] = hi[0];
    for (int c = lo[0]; c <= hi[0]; c++) {
        if (c == lo[1]) c = hi[1] + 1;
        if (c <= hi[0]) fresh |= test_sample(bits, g, seg, c + col, r);
    }
    return kProf && fresh;
}

// Set the samples of row r within R of the segment.  Where both discs meet the
// row well inside (half-chords w with w^2 >= 8 R E), a distance error of E
// moves an end by E R / w, and by at most an eighth more for the curvature:
// a column nearer to the end than e = 1.25 E R / w takes the exact test, every
// other column is decided by its side of the end.  One column at most is that
// near only while e < 1/2, that is w^2 > 6.25 (R E)^2, which the first condition
// implies for R up to about 200 spacings (every radius in pixels); rows of larger
// ground radii where e may reach 1/2 go to draw_row_slow, which tests them all.
template <bool kProf = false>
__device__ __forceinline__ bool draw_row(uint32_t* bits, const Lattice& g, const PieceRow& q, const int4* seg, int r) {
    const int col = (int)(q.at & 0xffffu) - 1024, row = (int)(q.at >> 16) - 1024;
    const float rho = (float)g.R * __int_as_float((127 - g.s) << 23);
    const float ym = (float)(r - row) - q.c0 * q.mx, xm = q.c0 * q.my, inv = rcp_approx(q.my);
    const float r2 = rho * rho, rm = rho * q.mx, rE = rho * q.E;
    const float tl = fminf(fmaxf((ym - rm) * inv, q.ta), q.tb), tr = fminf(fmaxf((ym + rm) * inv, q.ta), q.tb);
    const float dl = fmaf(-tl, q.my, ym), dr = fmaf(-tr, q.my, ym);
    const float al = fmaf(-dl, dl, r2), ar = fmaf(-dr, dr, r2);
    if (!(fminf(al, ar) >= rE * fmaxf(8.f, 6.5f * rE)) || !(q.E > 0.f && q.E < rho)) {
        // beyond R + E of the row both half-chords are imaginary
        if (q.E > 0.f && fmaxf(al, ar) < -8.f * rE - 2.f * q.E * q.E) return false;
        return draw_row_slow<kProf>(bits, g, q, seg, r);
    }
    const float wl = sqrt_approx(al), wr = sqrt_approx(ar);
    const float xl = fmaf(tl, q.mx, -xm) - wl, xr = fmaf(tr, q.mx, -xm) + wr;
    const float el = 1.25f * rE * rcp_approx(wl), er = 1.25f * rE * rcp_approx(wr);
    const float nl = rintf(xl), nr = rintf(xr);
    const bool vl = fabsf(xl - nl) <= el, vr = fabsf(xr - nr) <= er;
    const int il = (int)nl, ir = (int)nr;
    const int clo = (int)(q.span & 0xffffu) - col, chi = (int)(q.span >> 16) - col;
    // a doubtful column is left out of the interval and tested
    const int lo = max(il + (vl || nl < xl ? 1 : 0), clo), hi = min(ir - (vr || nr > xr ? 1 : 0), chi);
    bool fresh = false;
    if (lo <= hi) fresh = set_columns(bits + r * kBitStride, lo + col, hi + col);
    if (vl && il >= clo && il <= chi) fresh |= test_sample(bits, g, seg, il + col, r);
    if (vr && ir >= clo && ir <= chi) fresh |= test_sample(bits, g, seg, ir + col, r);
    return fresh;
}

// What a leaf visit came to, per lane, for the phase profile.
struct Visit {
    bool reached = false;   // an object that an open sample is in reach of
    bool decided = false;   // a sample decided
};

// A segment leaf: 32 pieces, each with a run of open rows that it reaches.
// The (piece, row) pairs are numbered through by a prefix sum over the lanes
// and the lanes take them in turn, so a leaf costs ceil(pairs / 32) rounds
// whatever the pieces' heights.
template <bool kProf>
__device__ __forceinline__ Visit draw_segments(const Params& p, const Src& src, uint32_t* bits, float4* pair_obj,
                                               int* pair_row, const int32_t* reach, const Lattice& g, uint32_t leaf,
                                               uint32_t rows, int lane) {
    Visit v;
    const uint64_t i = (uint64_t)leaf * 32 + lane;
    int4 o = make_int4(0, 0, 0, 0), pb = make_int4(kEmptyLo, kEmptyLo, kEmptyHi, kEmptyHi);
    const int4* rec = (const int4*)src.obj + 2 * i;
    if (i < src.n) {
        o = __ldg(rec);
        pb = __ldg(rec + 1);
    }
    const int32_t x0 = rel32(pb.x, g.xc), y0 = rel32(pb.y, g.yc), x1 = rel32(pb.z, g.xc), y1 = rel32(pb.w, g.yc);
    const int r0 = max(g.hh - ((g.R - y0) >> g.s), 0), r1 = min(((y1 + g.R) >> g.s) + g.hh, 2 * g.hh - 1);
    const int clo = max(g.hw - ((g.R - x0) >> g.s), 0), chi = min(((x1 + g.R) >> g.s) + g.hw, 2 * g.hw - 1);
    uint32_t mine = 0u;
    if (i < src.n && r0 <= r1 && clo <= chi) mine = rows & (~0u << r0) & (~0u >> (31 - r1));
    if (kProf) v.reached = mine != 0u && box_open<true>(bits, reach, g, x0, y0, x1, y1, mine);
    const uint32_t some = __ballot_sync(kFull, mine != 0u);
    if (some == 0u) return v;
    // from the first to the last open row
    const int first = __ffs(mine) - 1, count = mine ? 32 - __clz(mine) - first : 0;
    const int sum = lane_sums(count, lane), total = __shfl_sync(kFull, sum, 31), start = sum - count;
    if (count) {
        const PieceRow q = piece_row(g, o, x0, y0, x1, y1, clo, chi);
        const int k = __popc(some & ((1u << lane) - 1u));
        pair_obj[2 * k] = make_float4(q.mx, q.my, q.c0, q.E);
        pair_obj[2 * k + 1] = make_float4(q.ta, q.tb, __uint_as_float(q.at), __uint_as_float(q.span));
        pair_row[k] = (first - start) * 32 + lane;   // a pair's row less its number, and the piece
    }
    __syncwarp();
    PairRounds rounds(start, count);
    for (int base = 0; base < total; base += 32) {
        const int k = rounds.object(base, lane), j = base + lane;
        if (j < total) {
            const float4 a = pair_obj[2 * k], b = pair_obj[2 * k + 1];
            const int at = pair_row[k];
            PieceRow q;
            q.mx = a.x, q.my = a.y, q.c0 = a.z, q.E = a.w;
            q.ta = b.x, q.tb = b.y, q.at = __float_as_uint(b.z), q.span = __float_as_uint(b.w);
            v.decided |= draw_row<kProf>(bits, g, q, (const int4*)src.obj + 2 * ((uint64_t)leaf * 32 + (at & 31)), (at >> 5) + j);
        }
        __syncwarp();
    }
    return v;
}

// ---- polygon fill ---------------------------------------------------------------

// End of the columns that an edge crosses strictly to the right in the row at
// height y (Algorithm 2's ray test): column c is crossed when (c - hw) h ey < N
// with N = ex (y - ly) + lx ey, so the columns are those before ceil(N / (h ey))
// + hw, cut off to lo..hi.  The quotient is estimated in single precision (cut off to
// the strip, a hundredth of a column or less away, then truncated towards zero), raised
// by the exact remainder's quotient, and settled by the sign of what remains.
// |N| <= 2^62: it is ey times the crossing's coordinate.
__device__ __forceinline__ int crossing_end(const Lattice& g, int32_t lx, int32_t ly, int32_t ex, int32_t ey, int32_t y,
                                            int lo, int hi) {
    const int64_t N = (int64_t)ex * ((int64_t)y - ly) + (int64_t)lx * ey;
    const float inv = rcp_approx((float)ey) * __int_as_float((127 - g.s) << 23);   // 1 / (h ey)
    lo -= g.hw;
    hi -= g.hw;
    int t = (int)fmaxf(fminf((float)N * inv, (float)hi), (float)lo);
    int64_t d = N - (int64_t)(t * (1 << g.s)) * ey;
    t = (int)fmaxf(fminf((float)t + ceilf((float)d * inv), (float)hi), (float)lo);
    d = N - (int64_t)(t * (1 << g.s)) * ey;
    if (d > 0) t++;
    else if (d <= -((int64_t)ey << g.s)) t--;
    return max(min(t, hi), lo) + g.hw;
}

// One polygon (box columns clo..chi, open rows `rows`): every edge toggles, per
// row that it straddles, all columns before its crossing; kept as one bit per
// crossing, a column's parity is the XOR of the bits after it, formed once
// for the whole row.  Edges are taken 32 at a time, their (edge, row) pairs
// shared over the lanes as for segments; then a lane per row turns the bits
// into filled samples and clears them.
__device__ __forceinline__ bool fill_polygon(const Params& p, uint32_t* bits, uint32_t* cross, int4* pair_obj,
                                             int* pair_row, const Lattice& g, uint64_t e0, uint64_t e1, int clo, int chi, uint32_t rows, int lane) {
    const int rf = __ffs(rows) - 1, rl = 31 - __clz(rows);
    for (uint64_t base = e0; base < e1; base += 32) {
        int4 e = make_int4(0, 0, 0, 0);   // a level edge straddles no row
        if (base + lane < e1) e = __ldg(p.poly_edges + base + lane);
        if (e.y > e.w) e = make_int4(e.z, e.w, e.x, e.y);
        const int32_t lx = e.x - g.xc, ly = e.y - g.yc, hy = e.w - g.yc, ex = e.z - e.x, ey = e.w - e.y;
        // rows with ly <= y < hy
        const int r0 = max(g.hh - ((-ly) >> g.s), rf), r1 = min(g.hh - ((-hy) >> g.s) - 1, rl);
        const int count = max(r1 - r0 + 1, 0);
        const uint32_t some = __ballot_sync(kFull, count > 0);
        if (some == 0u) continue;
        const int sum = lane_sums(count, lane), total = __shfl_sync(kFull, sum, 31), start = sum - count;
        if (count) {
            const int k = __popc(some & ((1u << lane) - 1u));
            pair_obj[k] = make_int4(lx, ly, ex, ey);
            pair_row[k] = r0 - start;
        }
        __syncwarp();
        PairRounds rounds(start, count);
        for (int first = 0; first < total; first += 32) {
            const int k = rounds.object(first, lane), j = first + lane;
            if (j < total) {
                const int4 o = pair_obj[k];
                const int r = pair_row[k] + j;
                const int t = crossing_end(g, o.x, o.y, o.z, o.w, (r - g.hh) * (1 << g.s), clo, chi + 1);
                if (t > clo) atomicXor(cross + r * kBitStride + (t >> 5), 1u << (t & 31));
            }
        }
        __syncwarp();
    }
    __syncwarp();
    bool fresh = false;
    if (lane >= rf && lane <= rl) {
        uint32_t carry = 0u;
        uint32_t* c = cross + lane * kBitStride;
        uint32_t* row = bits + lane * kBitStride;
        const int k0 = clo >> 5;
        for (int k = (chi + 1) >> 5; k >= k0; k--) {
            const uint32_t d = c[k];
            uint32_t s = d;   // bit b: XOR of the word's bits from b on
            s ^= s >> 1;
            s ^= s >> 2;
            s ^= s >> 4;
            s ^= s >> 8;
            s ^= s >> 16;
            uint32_t f = s ^ d ^ carry;
            carry ^= 0u - (s & 1u);
            if (d) c[k] = 0u;
            if (k == k0) f &= ~0u << (clo & 31);
            if (k < g.hw >> 4) fresh |= set_bits(row + k, f);
        }
    }
    __syncwarp();
    return fresh;
}

// A leaf of the polygon-box tree: the polygons whose box holds an open sample.
__device__ __forceinline__ Visit fill_polygons(const Params& p, const Src& src, uint32_t* bits, uint32_t* cross,
                                               int4* pair_obj, int* pair_row, const int32_t* reach, const Lattice& g,
                                               uint32_t leaf, uint32_t rows, int lane) {
    Visit v;
    const uint64_t i = (uint64_t)leaf * 32 + lane;
    int4 b = make_int4(kEmptyLo, kEmptyLo, kEmptyHi, kEmptyHi);
    uint32_t id = 0;
    if (i < src.n) {
        b = __ldg((const int4*)src.obj + i);
        id = __ldg(src.ids + i);
    }
    const int32_t x0 = rel32(b.x, g.xc), y0 = rel32(b.y, g.yc), x1 = rel32(b.z, g.xc), y1 = rel32(b.w, g.yc);
    uint32_t m = __ballot_sync(kFull, b.x <= b.z && i < src.n && box_open<false>(bits, reach, g, x0, y0, x1, y1, rows));
    v.reached = m != 0u;
    while (m) {
        const int k = __ffs(m) - 1;
        m &= m - 1;
        const int32_t kx0 = __shfl_sync(kFull, x0, k), kx1 = __shfl_sync(kFull, x1, k);
        const uint32_t open = open_rows<false>(bits, reach, g, kx0, __shfl_sync(kFull, y0, k), kx1, __shfl_sync(kFull, y1, k), lane);
        if (open == 0) continue;
        const uint32_t pid = __shfl_sync(kFull, id, k);
        log_read(p, kLogPoly, pid, lane);
        if (pid >= p.n_poly) {
            if (lane == 0) check_failed(p, 5, pid);
            continue;
        }
        const uint64_t e0 = __ldg(p.poly_edge_off + pid), e1 = __ldg(p.poly_edge_off + pid + 1);
        if (e0 > e1 || e1 > p.n_edges) {
            if (lane == 0) check_failed(p, 6, ((uint64_t)pid << 24) | (e1 & 0xffffff));
            continue;
        }
        const int clo = max(g.hw - ((-kx0) >> g.s), 0), chi = min((kx1 >> g.s) + g.hw, 2 * g.hw - 1);
        v.decided |= fill_polygon(p, bits, cross, pair_obj, pair_row, g, e0, e1, clo, chi, open, lane);
    }
    return v;
}

// ---- traversal ----------------------------------------------------------------

// One frontier entry (its box [bx0, bx1] in x, rows: its open rows): a
// depth-first descent of its subtree down to the points of its leaves.  Per
// step the lanes hold 32 boxes -- the children of an inner node, or the points
// of a leaf -- and draw them: a point's covered samples, or those that a small
// child box certainly covers.  The stack keeps the children still to visit of
// the current level-1 node in registers, of the levels above in shared
// memory; a child is taken only if a sample that it can reach is open then,
// and below it only the rows with such a sample matter.  (One drawing site and
// one reach test for leaves and nodes keep the loop small for the instruction
// cache.)
template <int kKind, bool kNarrowR, bool kFine, bool kProf>
__device__ __forceinline__ void sweep_entry(const Params& p, SweepSmem<kKind>& sm, const Src& src, const Lattice& g,
                                             int level, uint32_t id, uint32_t rows, int32_t bx0, int32_t bx1,
                                             int lane, int warp) {
    if (level < 0 || level > kMaxLevels || id >= src.lvl_n[level]) {
        if (lane == 0) check_failed(p, 2, ((uint64_t)level << 40) | id);
        return;
    }
    uint32_t* stk_node = sm.stk_node[warp];
    uint32_t* stk_mask = sm.stk_mask[warp];
    // rows that a point reaches; the window form pays up to about twice that
    const int reach_rows = 2 * (2 * (g.R >> g.s) + 1);
    int lvl = level;
    uint32_t node = id;
    uint32_t mask1 = 0u, node1 = 0u;              // the current level-1 node and its children to take
    int32_t cx0 = 0, cy0 = 0, cx1 = 0, cy1 = 0;   // its child boxes
    long long t0 = 0;
    while (true) {
        int32_t x0 = 0, y0 = 0, x1 = 0, y1 = 0;
        bool draw = false;
        Visit visit;
        if (lvl == 0 && kKind != HV_LAYER_POINTS) {
            log_read(p, kKind == kPolyFill ? kLogPolyLeaf : kLogLeaf, node, lane);
            t0 = tick<kProf>();
            if constexpr (kKind == kPolyFill)
                visit = fill_polygons(p, src, sm.bits, sm.cross[warp], (int4*)sm.pair_obj[warp], sm.pair_row[warp], sm.reach, g, node, rows, lane);
            else
                visit = draw_segments<kProf>(p, src, sm.bits, sm.pair_obj[warp], sm.pair_row[warp], sm.reach, g, node, rows, lane);
        } else if (lvl == 0) {
            log_read(p, kLogLeaf, node, lane);
            t0 = tick<kProf>();
            const uint64_t i = (uint64_t)node * 32 + lane;
            int2 o = make_int2(0, 0);
            draw = i < src.n;
            if (draw) o = __ldg((const int2*)src.obj + i);
            x0 = x1 = rel32(o.x, g.xc);
            y0 = y1 = rel32(o.y, g.yc);
            if (kProf) visit.reached = draw && box_open<kFine>(sm.bits, sm.reach, g, x0, y0, x1, y1, rows);
        } else {
            const int32_t* base = src.lvl[lvl] + (uint64_t)node * 128;
            if (p.log != nullptr)
                log_read(p, kKind == kPolyFill ? kLogPolyNode : kLogNode, (uint64_t)(base - src.nodes) >> 7, lane);
            const int32_t ax0 = __ldg(base + lane), ay0 = __ldg(base + 32 + lane);
            const int32_t ax1 = __ldg(base + 64 + lane), ay1 = __ldg(base + 96 + lane);
            x0 = rel32(ax0, g.xc), y0 = rel32(ay0, g.yc), x1 = rel32(ax1, g.xc), y1 = rel32(ay1, g.yc);
            draw = ax0 <= ax1;   // not a padding box
        }
        const bool valid = draw;
        if constexpr (kKind == HV_LAYER_POINTS) {
            draw = draw && small_box(g, x0, y0, x1, y1);
            const int c0 = g.hw - ((g.R - bx0) >> g.s);
            if (((bx1 + g.R) >> g.s) + g.hw - c0 < 32 && __popc(rows) <= reach_rows) {
                if (__any_sync(kFull, draw))
                    visit.decided = splat_window<kNarrowR>(sm.bits, g, x0, y0, x1, y1, c0, draw, rows, lane);
            } else if (draw) {
                visit.decided = splat<kNarrowR>(sm.bits, g, x0, y0, x1, y1, rows);
            }
        }
        __syncwarp();
        if (lvl == 0) {
            prof_since<kProf>(sm, kPLeaf, t0, lane);
            prof_add<kProf>(sm, kPLeafVisits, 1, lane);
            if constexpr (kProf) {
                const bool decided = __any_sync(kFull, visit.decided), reached = __any_sync(kFull, visit.reached);
                prof_add<kProf>(sm, decided ? kPLeafDecided : kPLeafEmpty, decided || !reached, lane);
            }
            if (level == 0) return;
            lvl = 1;
        } else {
            prof_add<kProf>(sm, kPNodeVisits, 1, lane);
            const uint32_t m = __ballot_sync(kFull, valid && box_open<kFine>(sm.bits, sm.reach, g, x0, y0, x1, y1, rows));
            if (lvl == 1) {
                mask1 = m;
                node1 = node;
                cx0 = x0, cy0 = y0, cx1 = x1, cy1 = y1;
            } else {
                stk_node[lvl] = node;
                stk_mask[lvl] = m;
                __syncwarp();
            }
        }
        // the next child to take
        while (true) {
            int32_t by0, by1;
            int c;
            if (lvl == 1) {
                if (mask1 == 0) {
                    if (level == 1) return;
                    lvl = 2;
                    continue;
                }
                c = __ffs(mask1) - 1;
                mask1 &= mask1 - 1;
                node = node1 * 32u + (uint32_t)c;
                bx0 = __shfl_sync(kFull, cx0, c), by0 = __shfl_sync(kFull, cy0, c);
                bx1 = __shfl_sync(kFull, cx1, c), by1 = __shfl_sync(kFull, cy1, c);
            } else {
                const uint32_t m = stk_mask[lvl], up = stk_node[lvl];
                __syncwarp();
                if (m == 0) {
                    if (lvl == level) return;
                    lvl++;
                    continue;
                }
                c = __ffs(m) - 1;
                stk_mask[lvl] = m & (m - 1);
                __syncwarp();
                const int32_t* nb = src.lvl[lvl] + (uint64_t)up * 128 + c;
                bx0 = rel32(__ldg(nb), g.xc), by0 = rel32(__ldg(nb + 32), g.yc);
                bx1 = rel32(__ldg(nb + 64), g.xc), by1 = rel32(__ldg(nb + 96), g.yc);
                node = up * 32u + (uint32_t)c;
            }
            rows = open_rows<kFine>(sm.bits, sm.reach, g, bx0, by0, bx1, by1, lane);
            if (rows == 0) continue;
            if (node >= src.lvl_n[lvl - 1]) {
                if (lane == 0) check_failed(p, 3, ((uint64_t)(lvl - 1) << 40) | node);
                continue;
            }
            lvl--;
            break;
        }
    }
}

// Every frontier entry of the strip, taken by the warps in turn, and the side
// tree (objects longer than the learned index's halo) as one more entry.
template <int kKind, bool kNarrowR, bool kFine, bool kProf>
__device__ void sweep_pass(const Params& p, SweepSmem<kKind>& sm, const Src& src, const Src& side, const TreeArg& st,
                           bool side_hit, const Lattice& g, int tid) {
    const int lane = tid & 31, warp = tid >> 5;
    const int f_count = sm.f_count, f_level = sm.f_level, fb = sm.f_buf;
    uint32_t* bits = sm.bits;
    const long long t_active = tick<kProf>();
    if constexpr (kKind == HV_LAYER_POINTS) {
        // What the frontier's boxes certainly cover, a box per thread: where the
        // points are dense most leaves of the frontier are then covered unread
        // (36 single tiles of 10M points 1,030 -> 933 us in all; 4,000 tiles of
        // 100M points, with frontiers of nodes, 11.05 -> 11.01 ms).
        bool whole = false;
        for (int e = tid; e < f_count; e += kThreads) {
            const int4 b = sm.fbox[fb][e];
            const int32_t x0 = rel32(b.x, g.xc), y0 = rel32(b.y, g.yc), x1 = rel32(b.z, g.xc), y1 = rel32(b.w, g.yc);
            // (a radius larger than the tile: nothing else is needed)
            if (kFine && covers_strip(g, x0, y0, x1, y1)) {
                whole = true;
                break;
            }
            if (small_box(g, x0, y0, x1, y1)) splat<kNarrowR>(bits, g, x0, y0, x1, y1, ~0u);
        }
        if (!kFine) {
            __syncthreads();
        } else if (__syncthreads_or(whole)) {
            for (int k = tid; k < kSampleRows * kBitStride; k += kThreads) bits[k] = ~0u;
            return;
        }
    }
    const int n_entries = f_count + (side_hit ? 1 : 0);
    while (true) {
        int e = 0;
        if (lane == 0) e = atomicAdd(&sm.next_entry, 1);
        e = __shfl_sync(kFull, e, 0);
        if (e >= n_entries) break;
        prof_add<kProf>(sm, kPFrontierEntries, 1, lane);
        const bool from_side = e >= f_count;
        const int4 b = from_side ? st.root_box : sm.fbox[fb][e];
        const int32_t x0 = rel32(b.x, g.xc), x1 = rel32(b.z, g.xc);
        const uint32_t rows = open_rows<kFine>(bits, sm.reach, g, x0, rel32(b.y, g.yc), x1, rel32(b.w, g.yc), lane);
        if (rows == 0) continue;
        const long long t0 = tick<kProf>();
        sweep_entry<kKind, kNarrowR, kFine, kProf>(p, sm, from_side ? side : src, g, from_side ? st.top : f_level,
                                            from_side ? 0u : sm.fid[fb][e], rows, x0, x1, lane, warp);
        prof_since<kProf>(sm, kPDescend, t0, lane);
    }
    prof_since<kProf>(sm, kPBlocksWarp, t_active, lane);
}

// Is one of the frontier's boxes within R of every sample by its farthest corner?  An
// object lies in it, so the strip is covered: where the radius is larger than the tile
// nothing else is read (60 tiles of 200,000 crowded points at R = 2^29: 641 -> 102 us).
// (Points make the same test where they draw the frontier's boxes.  A
// call, and there a part of the loop: other forms cost 4,000 tiles of 100M points at 2 px,
// which never take it, 1 to 3% in registers.)
__device__ __noinline__ bool strip_covered(uint32_t* bits, const int4* box, int n, Lattice g, int tid) {
    bool whole = false;
    for (int e = tid; e < n; e += kThreads) {
        const int4 b = box[e];
        whole |= covers_strip(g, rel32(b.x, g.xc), rel32(b.y, g.yc), rel32(b.z, g.xc), rel32(b.w, g.yc));
    }
    if (!__syncthreads_or(whole)) return false;
    for (int k = tid; k < kSampleRows * kBitStride; k += kThreads) bits[k] = ~0u;
    return true;
}

// Covered samples of 16 / 4 pixels from column c of pixel row j, as counts.
__device__ __forceinline__ uint32_t pixel_count(uint32_t top, uint32_t bottom, int q) {
    return (uint32_t)(__popc((top >> (2 * q)) & 3u) + __popc((bottom >> (2 * q)) & 3u));
}

// CTAs per SM.  Points: six, 11.0 ms for 4,000 tiles of 100M points against 11.4
// with five and 12.6 with four (40 registers with a small spill; the dependent
// steps of a row leave issue slots that more warps fill); in column parts, where
// a grid is resident at four per SM, five: one tile 17.2 against 18.0 us.
// Segments, outlines and fill: four; with five for segments and outlines 1,000
// polygon tiles 10.3 against 9.7 ms, 33 styled ones 361 against 341 us, 4,000
// line tiles 5.55 ms with either.
template <int kKind, bool kSplit>
struct SweepTraits {
    static constexpr int kPerSM = kKind == HV_LAYER_POINTS ? (kSplit ? 5 : 6) : 4;
};

template <int kKind, bool kProf, bool kSplit>
__global__ void __launch_bounds__(kThreads, SweepTraits<kKind, kSplit>::kPerSM) k_sweep(const Params p) {
    __shared__ SweepSmem<kKind> sm;
    const int tid = threadIdx.x;
    const long long t_start = tick<kProf>();
    if constexpr (kProf) {
        if (tid < kPN) sm.prof[tid] = 0;
    }
    const int rows = p.rows;
    const int parts = kSplit ? p.parts : 1, cols = kTile / parts;
    const uint32_t tile = blockIdx.x / (p.strips * parts);
    const int sp = (int)(blockIdx.x % (p.strips * parts));
    const int strip = sp / parts, col0 = (sp % parts) * cols;
    const uint32_t n = p.n_dev ? min(*p.n_dev, p.n) : p.n;
    if (tile >= n) return;
    const hv_tile_req q = p.reqs[tile];
    const bool ok = q.z <= 19 && q.x < (1u << q.z) && q.y < (1u << q.z) && (p.R_units >= 0 || (q.r16 >= 1 && q.r16 <= 1024));
    for (int k = tid; k < kSampleRows * kBitStride; k += kThreads) sm.bits[k] = 0u;
    if constexpr (kKind == kPolyFill)
        for (int k = tid; k < kWarps * kSampleRows * kBitStride; k += kThreads) sm.cross[0][k] = 0u;
    uint8_t* const out = p.out + (uint64_t)tile * p.tile_bytes;
    const bool mask_mode = p.mode == HV_MODE_MASK;
    // the samples are the pixel centres (else the super-samples)
    const bool centres = mask_mode || (kKind == kPolyFill && !p.fill_aa);
    if constexpr (kKind == HV_LAYER_POLYGONS) {
        decode_fill(p, out, sm.res, strip, col0, cols, tid, p.fill_aa && !mask_mode);
        __syncthreads();
        // a MASK pixel whose centre is already filled is decided (unless a
        // pattern may leave it transparent)
        if (mask_mode && p.pat_w == 0) {
            const int wpr = cols / 32, wsh = __ffs(wpr) - 1;
            if (tid < rows * wpr) {
                const int jl = tid >> wsh, w = tid & (wpr - 1);
                uint32_t word = 0u;
                for (int b = 0; b < 32; b++)
                    if (sm.res[jl * kTile + col0 + 32 * w + b] >> kResFillShift) word |= 1u << b;
                sm.bits[jl * kBitStride + w] = word;
            }
        }
    }
    if (!ok && tid == 0 && sp == 0) atomicOr(p.status, 1u);
    if (tid == 0) sm.next_entry = 0;
    __syncthreads();
    if (tid == 0) prof_since<kProf>(sm, kPPrologue, t_start, 0);
    if (ok) {
        const int z = q.z, L = 23 - z;
        const int32_t ps = 1 << L;
        const int32_t X0 = (int32_t)(-(int64_t)kGridHalf + (int64_t)q.x * ((int64_t)1 << (31 - z)));
        const int32_t Y0 = (int32_t)(-(int64_t)kGridHalf + (int64_t)q.y * ((int64_t)1 << (31 - z)));
        Lattice g;
        g.s = centres ? L : L - 1;
        g.hw = centres ? cols / 2 : cols;
        g.hh = centres ? rows / 2 : rows;
        g.R = kKind == kPolyFill ? 0 : (p.R_units >= 0 ? p.R_units : (int32_t)q.r16 << (19 - z));
        g.R2 = (int64_t)g.R * g.R;
        g.rs = max(32 - __clz(g.R) - 6, 0);
        g.narrow = g.R <= kNarrow;
        const int32_t half = 1 << g.s >> 1;   // the first sample lies half a spacing inside the strip
        g.xc = X0 + (col0 + cols / 2) * ps + half;
        g.yc = Y0 + (strip * rows + rows / 2) * ps + half;
        // the strip's samples, widened by R (fits 32 bits: inside the grid, plus at most 2^29)
        const int32_t bx0 = g.xc - (g.hw << g.s) - g.R, bx1 = g.xc + ((g.hw - 1) << g.s) + g.R;
        const int32_t by0 = g.yc - (g.hh << g.s) - g.R, by1 = g.yc + ((g.hh - 1) << g.s) + g.R;
        const bool learned = p.use_learned != 0;
        const TreeArg& tree = kKind == kPolyFill ? p.mtree : p.tree;
        const TreeArg& stree = kKind == kPolyFill ? p.mside : p.side;
        const long long t_cull = tick<kProf>();
        set_levels(sm, 0, tree, tid);
        set_levels(sm, 1, stree, tid);
        fill_reach(sm.reach, g, tid);
        __syncthreads();
        if (!learned)
            cull(p, tree, kKind == kPolyFill, sm, bx0, by0, bx1, by1, tid);
        else
            learned_cull(p, tree, kKind == kPolyFill ? p.mlm : p.lm, kKind == kPolyFill ? p.mhalo : p.halo, sm, bx0, by0,
                         bx1, by1, tid);
        if (tid == 0) prof_since<kProf>(sm, kPCull, t_cull, 0);
        const int4 sb = stree.root_box;
        const bool side_hit = stree.top > 0 && sb.x <= bx1 && sb.z >= bx0 && sb.y <= by1 && sb.w >= by0;
        if (sm.f_count > 0 || side_hit) {
            const long long t_pass = tick<kProf>();
            if (tid == 0) prof_add<kProf>(sm, kPBlocks, (unsigned long long)(rows / kBH) * (cols / kBW), 0);
            Src src{p.obj, nullptr, tree.n_obj, tree.nodes, sm.lvl_base[0], sm.lvl_n[0]};
            Src side{p.side_obj, p.side_ids, stree.n_obj, stree.nodes, sm.lvl_base[1], sm.lvl_n[1]};
            if constexpr (kKind == kPolyFill) {
                src.obj = p.mbr_obj;
                src.ids = p.mbr_ids;
                side.obj = p.mside_obj;
                side.ids = p.mside_ids;
            }
            // (segments draw the same way at every radius)
            if (kKind != kPolyFill && (g.R >> g.s) > kTableReach) {
                if (kKind == HV_LAYER_POINTS || !strip_covered(sm.bits, sm.fbox[sm.f_buf], sm.f_count, g, tid))
                    sweep_pass<kKind, false, true, kProf>(p, sm, src, side, stree, side_hit, g, tid);
            } else if (kKind != HV_LAYER_POINTS || g.narrow)
                sweep_pass<kKind, true, false, kProf>(p, sm, src, side, stree, side_hit, g, tid);
            else
                sweep_pass<kKind, false, false, kProf>(p, sm, src, side, stree, side_hit, g, tid);
            __syncthreads();
            if (tid == 0) prof_since<kProf>(sm, kPBlocksCta, t_pass, 0);
        }
    }
    // ---- encode the strip (Sec. 4.1 Render Tiles) ----
    const long long t_enc = tick<kProf>();
    if constexpr (kKind == kPolyFill) {
        // the fill results for the outline launch, per pixel row at the start
        // of the row's part of the CTA's own output (see decode_fill)
        if (centres) {
            const int wpr = cols / 32, wsh = __ffs(wpr) - 1;
            if (tid < rows * wpr) {
                const int jl = tid >> wsh, w = tid & (wpr - 1);
                ((uint32_t*)(out + px_offset(p.mode, strip * rows + jl, col0)))[w] = sm.bits[jl * kBitStride + w];
            }
        } else {
            // a byte per pixel: its super-samples inside, 4 pixels per word
            const int wpr = cols / 4, wsh = __ffs(wpr) - 1;
            for (int k = tid; k < rows * wpr; k += kThreads) {
                const int jl = k >> wsh, w = k & (wpr - 1), sh = 8 * (w & 3);
                const uint32_t a = sm.bits[2 * jl * kBitStride + (w >> 2)] >> sh, b = sm.bits[(2 * jl + 1) * kBitStride + (w >> 2)] >> sh;
                uint32_t v = 0u;
#pragma unroll
                for (int c = 0; c < 4; c++) v |= pixel_count(a, b, c) << (8 * c);
                ((uint32_t*)(out + px_offset(p.mode, strip * rows + jl, col0)))[w] = v;
            }
        }
    } else if constexpr (kKind == HV_LAYER_POLYGONS) {
        // the covered samples join the fill results, a byte per pixel
        for (int k = tid; k < rows * cols; k += kThreads) {
            const int jl = k / cols, c = k % cols;
            uint32_t v;
            if (mask_mode)
                v = (sm.bits[jl * kBitStride + (c >> 5)] >> (c & 31)) & 1u ? kResCentre : 0u;
            else
                v = ((sm.bits[2 * jl * kBitStride + (c >> 4)] >> (2 * (c & 15))) & 3u) |
                    (((sm.bits[(2 * jl + 1) * kBitStride + (c >> 4)] >> (2 * (c & 15))) & 3u) << 2);
            sm.res[jl * kTile + col0 + c] |= (uint8_t)v;
        }
        __syncthreads();
        encode_polygons(p, sm.res, out, strip, col0, cols, tile, tid);
    } else if (mask_mode) {
        // the sample bits are the output: word w of row j = pixels 32w .. 32w+31
        const int wpr = cols / 32, wsh = __ffs(wpr) - 1;
        if (tid < rows * wpr) {
            const int jl = tid >> wsh, w = tid & (wpr - 1);
            *(uint32_t*)(out + px_offset(p.mode, strip * rows + jl, col0 + 32 * w)) = sm.bits[jl * kBitStride + w];
        }
    } else if (p.mode == HV_MODE_COVERAGE) {
        // 16 pixels (one sample word of two rows, one uint4) per thread and step
        const int upr = cols / 16, ush = __ffs(upr) - 1;
        for (int u = tid; u < rows * upr; u += kThreads) {
            const int jl = u >> ush, w = u & (upr - 1);
            const uint32_t a = sm.bits[2 * jl * kBitStride + w], b = sm.bits[(2 * jl + 1) * kBitStride + w];
            uint32_t w4[4];
#pragma unroll
            for (int k = 0; k < 4; k++) {
                uint32_t v = 0;
#pragma unroll
                for (int c = 0; c < 4; c++) v |= pixel_count(a, b, 4 * k + c) << (8 * c);
                w4[k] = v;
            }
            *(uint4*)(out + px_offset(p.mode, strip * rows + jl, col0 + 16 * w)) = make_uint4(w4[0], w4[1], w4[2], w4[3]);
        }
    } else {
        // 4 pixels (a byte of two sample rows, one uint4) per thread and step
        const int upr = cols / 4, ush = __ffs(upr) - 1;
        const uint32_t rgb = (uint32_t)p.line.x | ((uint32_t)p.line.y << 8) | ((uint32_t)p.line.z << 16);
        for (int u = tid; u < rows * upr; u += kThreads) {
            const int jl = u >> ush, c4 = u & (upr - 1);
            const int sh = 8 * (c4 & 3);
            const uint32_t a = sm.bits[2 * jl * kBitStride + (c4 >> 2)] >> sh, b = sm.bits[(2 * jl + 1) * kBitStride + (c4 >> 2)] >> sh;
            uint32_t w[4];
#pragma unroll
            for (int c = 0; c < 4; c++) {
                const uint32_t v = pixel_count(a, b, c);
                w[c] = v ? rgb | (((255u * v + 2u) >> 2) << 24) : 0u;
            }
            *(uint4*)(out + px_offset(p.mode, strip * rows + jl, col0 + 4 * c4)) = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
    if constexpr (kProf) {
        __syncthreads();
        if (tid == 0) {
            const unsigned long long now = (unsigned long long)clock64();
            sm.prof[kPEncode] += now - (unsigned long long)t_enc;
            sm.prof[kPTotal] += now - (unsigned long long)t_start;
            sm.prof[kPCtas] = 1;
            // CTA-wide phases hold every warp of the CTA
            const int cta_phases[6] = {kPTotal, kPPrologue, kPCull, kPBin, kPBlocksCta, kPEncode};
            for (int k = 0; k < 6; k++) sm.prof[cta_phases[k]] *= kWarps;
        }
        __syncthreads();
        if (tid < kPN && sm.prof[tid]) atomicAdd(p.phases + tid, sm.prof[tid]);
    }
}
