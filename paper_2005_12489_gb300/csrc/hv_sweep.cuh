// Coverage sweep: Algorithm 1 (SIBV) over a strip, object by object.
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
// Bound: instruction issue (72% of the slots busy; DRAM a few percent).  Drawn
// by strips, 600 tiles of 100M clustered points at 2 px take 2.4 M warp
// instructions per tile where the 8 x 4 block traversal took 5.7 M: 4,000
// tiles 23.5 -> 11.8 ms; 341 tiles of 100,000 points at zoom 0-4, 1 px, MASK
// 414 -> 73 us; one tile of 10M points 35 -> 29 us.
//
// Included by hv_render.cu (one translation unit with the block kernels).
#pragma once

constexpr int kBitStride = 17;   // words per sample row: 512 columns and a pad word (row-parallel reads then hit 32 banks)
constexpr int kSweepPerSM = 6;   // CTAs per SM (40 registers); measured against 4 and 5 at k_sweep
constexpr int kSampleRows = 2 * kStripRows;
static_assert(kSampleRows <= 32, "one lane per sample row");

struct SweepSmem : Front {
    uint32_t bits[kSampleRows * kBitStride];
    int32_t reach[64];
    uint32_t stk_node[kWarps][kMaxLevels + 1];
    uint32_t stk_mask[kWarps][kMaxLevels + 1];
    int next_entry;
};

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
// where the atomics would queue).
__device__ __forceinline__ void set_columns(uint32_t* row, int lo, int hi) {
    const int k0 = lo >> 5, k1 = hi >> 5;
    uint32_t m = ~0u << (lo & 31);
    const uint32_t last = ~0u >> (31 - (hi & 31));
    for (int k = k0; k < k1; k++) {
        if (m & ~*(volatile uint32_t*)(row + k)) atomicOr(row + k, m);
        m = ~0u;
    }
    m &= last;
    if (m & ~*(volatile uint32_t*)(row + k1)) atomicOr(row + k1, m);
}

// Set the samples that lie within R of every point of the lane's box
// [x0, x1] x [y0, y1] (relative coordinates): exactly the covered samples of
// a point (x0 = x1, y0 = y1), and samples certainly covered when the box holds
// at least one point.  In row y the farthest row distance is f = max(|y - y0|,
// |y - y1|), and with w = floor(sqrt(R^2 - f^2)) the columns are [x1 - w, x0 + w].
// Only the rows of `open` (a bit per sample row) are drawn.
template <bool kNarrowR>
__device__ __forceinline__ void splat(uint32_t* bits, const Lattice& g, int32_t x0, int32_t y0, int32_t x1,
                                      int32_t y1, uint32_t open) {
    const int r0 = max(g.hh - ((g.R - y1) >> g.s), 0);
    const int r1 = min(((y0 + g.R) >> g.s) + g.hh, 2 * g.hh - 1);
    if (r0 > r1) return;
    open &= (~0u << r0) & (~0u >> (31 - r1));
    while (open) {
        const int r = __ffs(open) - 1;
        open &= open - 1;
        const int32_t y = (r - g.hh) << g.s;
        const int32_t f = max(abs(y - y0), abs(y - y1));
        const int32_t w = half_width<kNarrowR>(g, f, x0, x1);
        const int lo = max(g.hw - ((w - x1) >> g.s), 0), hi = min(((x0 + w) >> g.s) + g.hw, 2 * g.hw - 1);
        if (lo <= hi) set_columns(bits + r * kBitStride, lo, hi);
    }
}

// The half-widths of reach by row distance, for the tests that only need an
// upper bound: reach[k] >= floor(sqrt(R^2 - f^2)) for every f with f >> rs = k,
// where rs makes R >> rs at most 63.  (Single precision, rounded up; a
// table read in place of a root per row.)
__device__ __forceinline__ void fill_reach(int32_t* reach, const Lattice& g, int tid) {
    if (tid <= (g.R >> g.rs)) {
        const float fR = (float)g.R, f = (float)(tid << g.rs);
        reach[tid] = min((int32_t)(sqrt_approx(fmaxf((fR - f) * (fR + f), 0.f)) * (1.f + 0x1p-19f)) + 1, g.R);
    }
}

// Is a sample of the row within [x0 - w, x1 + w] open?
__device__ __forceinline__ bool row_open(const uint32_t* row, const Lattice& g, int32_t x0, int32_t x1, int32_t w) {
    const int lo = max(g.hw - ((w - x0) >> g.s), 0), hi = min(((x1 + w) >> g.s) + g.hw, 2 * g.hw - 1);
    if (lo > hi) return false;
    const int k1 = hi >> 5;
    uint32_t m = ~0u << (lo & 31);
    for (int k = lo >> 5; k < k1; k++) {
        if (m & ~*(volatile const uint32_t*)(row + k)) return true;
        m = ~0u;
    }
    return (m & (~0u >> (31 - (hi & 31))) & ~*(volatile const uint32_t*)(row + k1)) != 0u;
}

// Sample rows (one lane each) with an open sample that an object inside the
// box could cover: within R of the box (rounded up).  Zero: nothing below the
// box matters.
__device__ __forceinline__ uint32_t open_rows(const uint32_t* bits, const int32_t* reach, const Lattice& g, int32_t x0,
                                              int32_t y0, int32_t x1, int32_t y1, int lane) {
    const int32_t y = (lane - g.hh) << g.s;
    const int32_t f = max(max(y0 - y, y - y1), 0);
    const bool open = lane < 2 * g.hh && f <= g.R && row_open(bits + lane * kBitStride, g, x0, x1, reach[f >> g.rs]);
    return __ballot_sync(kFull, open);
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
__device__ __forceinline__ void splat_window(uint32_t* bits, const Lattice& g, int32_t x0, int32_t y0, int32_t x1,
                                             int32_t y1, int c0, bool active, uint32_t rows, int lane) {
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
        if (k >= 0 && k < words && (a & ~*(volatile uint32_t*)(row + k))) atomicOr(row + k, a);
        if (k + 1 >= 0 && k + 1 < words && (b & ~*(volatile uint32_t*)(row + k + 1))) atomicOr(row + k + 1, b);
    }
}

// open_rows for the lane's own box: is any sample in reach open (in one of
// the given rows)?  One pass for the 32 children of a node; those that pass
// take open_rows again when their turn comes, after their siblings.
__device__ __forceinline__ bool box_open(const uint32_t* bits, const int32_t* reach, const Lattice& g, int32_t x0,
                                         int32_t y0, int32_t x1, int32_t y1, uint32_t rows) {
    const int r0 = max(g.hh - ((g.R - y0) >> g.s), 0), r1 = min(((y1 + g.R) >> g.s) + g.hh, 2 * g.hh - 1);
    if (r0 > r1) return false;
    rows &= (~0u << r0) & (~0u >> (31 - r1));
    while (rows) {
        const int r = __ffs(rows) - 1;
        rows &= rows - 1;
        const int32_t y = (r - g.hh) << g.s;
        if (row_open(bits + r * kBitStride, g, x0, x1, reach[max(max(y0 - y, y - y1), 0) >> g.rs])) return true;
    }
    return false;
}

// A box of points is worth drawing when it is no wider than about R (the
// samples that a larger one certainly covers are few or none).
__device__ __forceinline__ bool small_box(const Lattice& g, int32_t x0, int32_t y0, int32_t x1, int32_t y1) {
    const uint32_t most = (uint32_t)g.R + (uint32_t)(g.R >> 2);
    return (uint32_t)(x1 - x0) <= most && (uint32_t)(y1 - y0) <= most;
}

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
template <bool kNarrowR, bool kProf>
__device__ __forceinline__ void sweep_points(const Params& p, SweepSmem& sm, const Src& src, const Lattice& g,
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
        int32_t x0, y0, x1, y1;
        bool draw;
        if (lvl == 0) {
            log_read(p, kLogLeaf, node, lane);
            t0 = tick<kProf>();
            const uint64_t i = (uint64_t)node * 32 + lane;
            int2 o = make_int2(0, 0);
            draw = i < src.n;
            if (draw) o = __ldg((const int2*)src.obj + i);
            x0 = x1 = rel32(o.x, g.xc);
            y0 = y1 = rel32(o.y, g.yc);
        } else {
            const int32_t* base = src.lvl[lvl] + (uint64_t)node * 128;
            if (p.log != nullptr) log_read(p, kLogNode, (uint64_t)(base - src.nodes) >> 7, lane);
            const int32_t ax0 = __ldg(base + lane), ay0 = __ldg(base + 32 + lane);
            const int32_t ax1 = __ldg(base + 64 + lane), ay1 = __ldg(base + 96 + lane);
            x0 = rel32(ax0, g.xc), y0 = rel32(ay0, g.yc), x1 = rel32(ax1, g.xc), y1 = rel32(ay1, g.yc);
            draw = ax0 <= ax1;   // not a padding box
        }
        const bool valid = draw;
        draw = draw && small_box(g, x0, y0, x1, y1);
        const int c0 = g.hw - ((g.R - bx0) >> g.s);
        if (((bx1 + g.R) >> g.s) + g.hw - c0 < 32 && __popc(rows) <= reach_rows) {
            if (__any_sync(kFull, draw)) splat_window<kNarrowR>(sm.bits, g, x0, y0, x1, y1, c0, draw, rows, lane);
        } else if (draw) {
            splat<kNarrowR>(sm.bits, g, x0, y0, x1, y1, rows);
        }
        __syncwarp();
        if (lvl == 0) {
            prof_since<kProf>(sm, kPLeaf, t0, lane);
            prof_add<kProf>(sm, kPLeafVisits, 1, lane);
            if (level == 0) return;
            lvl = 1;
        } else {
            prof_add<kProf>(sm, kPNodeVisits, 1, lane);
            const uint32_t m = __ballot_sync(kFull, valid && box_open(sm.bits, sm.reach, g, x0, y0, x1, y1, rows));
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
            rows = open_rows(sm.bits, sm.reach, g, bx0, by0, bx1, by1, lane);
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
template <bool kNarrowR, bool kProf>
__device__ void sweep_pass(const Params& p, SweepSmem& sm, const Src& src, const Src& side, const TreeArg& st,
                           bool side_hit, const Lattice& g, int tid) {
    const int lane = tid & 31, warp = tid >> 5;
    const int f_count = sm.f_count, f_level = sm.f_level, fb = sm.f_buf;
    uint32_t* bits = sm.bits;
    const long long t_active = tick<kProf>();
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
        const uint32_t rows = open_rows(bits, sm.reach, g, x0, rel32(b.y, g.yc), x1, rel32(b.w, g.yc), lane);
        if (rows == 0) continue;
        const long long t0 = tick<kProf>();
        sweep_points<kNarrowR, kProf>(p, sm, from_side ? side : src, g, from_side ? st.top : f_level,
                                      from_side ? 0u : sm.fid[fb][e], rows, x0, x1, lane, warp);
        prof_since<kProf>(sm, kPDescend, t0, lane);
    }
    prof_since<kProf>(sm, kPBlocksWarp, t_active, lane);
}

// Covered samples of 16 / 4 pixels from column c of pixel row j, as counts.
__device__ __forceinline__ uint32_t pixel_count(uint32_t top, uint32_t bottom, int q) {
    return (uint32_t)(__popc((top >> (2 * q)) & 3u) + __popc((bottom >> (2 * q)) & 3u));
}

// Six CTAs per SM: 11.5 ms for 4,000 tiles of 100M points against 11.9 with
// five and 12.6 with four (40 registers with a small spill; the dependent steps
// of a row leave issue slots that more warps fill).
template <int kKind, bool kProf, bool kSplit>
__global__ void __launch_bounds__(kThreads, kSweepPerSM) k_sweep(const Params p) {
    __shared__ SweepSmem sm;
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
    if (!ok && tid == 0 && sp == 0) atomicOr(p.status, 1u);
    if (tid == 0) sm.next_entry = 0;
    __syncthreads();
    if (tid == 0) prof_since<kProf>(sm, kPPrologue, t_start, 0);
    const bool mask_mode = p.mode == HV_MODE_MASK;
    if (ok) {
        const int z = q.z, L = 23 - z;
        const int32_t ps = 1 << L;
        const int32_t X0 = (int32_t)(-(int64_t)kGridHalf + (int64_t)q.x * ((int64_t)1 << (31 - z)));
        const int32_t Y0 = (int32_t)(-(int64_t)kGridHalf + (int64_t)q.y * ((int64_t)1 << (31 - z)));
        Lattice g;
        g.s = mask_mode ? L : L - 1;
        g.hw = mask_mode ? cols / 2 : cols;
        g.hh = mask_mode ? rows / 2 : rows;
        g.R = p.R_units >= 0 ? p.R_units : (int32_t)q.r16 << (19 - z);
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
        const long long t_cull = tick<kProf>();
        set_levels(sm, 0, p.tree, tid);
        set_levels(sm, 1, p.side, tid);
        fill_reach(sm.reach, g, tid);
        __syncthreads();
        if (!learned)
            cull(p, p.tree, false, sm, bx0, by0, bx1, by1, tid);
        else
            learned_cull(p, p.tree, p.lm, p.halo, sm, bx0, by0, bx1, by1, tid);
        if (tid == 0) prof_since<kProf>(sm, kPCull, t_cull, 0);
        const int4 sb = p.side.root_box;
        const bool side_hit = p.side.top > 0 && sb.x <= bx1 && sb.z >= bx0 && sb.y <= by1 && sb.w >= by0;
        if (sm.f_count > 0 || side_hit) {
            const long long t_pass = tick<kProf>();
            if (tid == 0) prof_add<kProf>(sm, kPBlocks, (unsigned long long)(rows / kBH) * (cols / kBW), 0);
            Src src{p.obj, nullptr, p.tree.n_obj, p.tree.nodes, sm.lvl_base[0], sm.lvl_n[0], nullptr, nullptr};
            Src side{p.side_obj, p.side_ids, p.side.n_obj, p.side.nodes, sm.lvl_base[1], sm.lvl_n[1], nullptr, nullptr};
            if (g.narrow)
                sweep_pass<true, kProf>(p, sm, src, side, p.side, side_hit, g, tid);
            else
                sweep_pass<false, kProf>(p, sm, src, side, p.side, side_hit, g, tid);
            __syncthreads();
            if (tid == 0) prof_since<kProf>(sm, kPBlocksCta, t_pass, 0);
        }
    }
    // ---- encode the strip (Sec. 4.1 Render Tiles) ----
    const long long t_enc = tick<kProf>();
    uint8_t* out = p.out + (uint64_t)tile * p.tile_bytes;
    if (mask_mode) {
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
