// Tile rendering: tile cull, warp-cooperative traversal with early exit,
// exact predicates and the output encode, fused in one kernel (one
// instantiation per layer kind).
//
//   HiVision Algorithm 1 (SIBV): a pixel's value is the number of its four
//   super-samples within distance R of some object (points, segments,
//   polygon edges); MASK mode decides the pixel centre only.
//   HiVision Algorithm 2 (SIBF): a pixel centre is filled when, for some
//   polygon whose box contains it, that polygon's edges cross the ray from
//   the centre an odd number of times.
//
// Work decomposition.  One CTA (8 warps) renders a strip of 256 x rows pixels
// of one tile (rows = 16 for large batches, 8 or 4 for small ones; batches
// too small to fill the GPU even then split each 4-row strip into 2, 4 or 8
// column parts, one CTA each).  The CTA first culls the R-tree (or, with the
// learned index, the subtrees of the key ranges the model finds) against the
// strip's box expanded by R, breadth first, into a frontier of at most kFCap
// nodes in shared memory (the deepest level that fits).  Its warps then take
// the frontier's subtrees in turn and draw their objects into a bit per sample
// of the strip (hv_sweep.cuh); the epilogue encodes the bits (MASK bits,
// COVERAGE bytes or RGBA) with coalesced 16-byte stores.
#include "hv_device.cuh"
#include "hv_internal.h"
#include "hv_learned.cuh"

namespace hv {

namespace {

constexpr int kWarps = 8;
constexpr int kThreads = kWarps * 32;
constexpr int kStripRows = 16;   // the largest strip; a launch picks 4, 8 or 16 rows
constexpr int kBW = 8, kBH = 4;   // the pixel blocks that the phase profile counts
constexpr int kFCap = 512;
constexpr int kCullCells = 64;     // learned cull: at most this many Hilbert cells per strip
constexpr int kCullSub = kThreads / kCullCells;   // threads per cell
static_assert(kCullSub >= 2 && kCullSub <= 32 && (kCullSub & (kCullSub - 1)) == 0, "cell threads within a warp");
constexpr int kMaxPattern = 16;    // fill patterns: at most 16 x 16 texels

// result bits per pixel: bits 0-3 the outline's super-samples, bit 4 the
// centre, bits 5-7 the fill field (0: not filled; centre fill: 1; the
// anti-aliased fill: the number of super-samples inside, 0..4)
constexpr uint32_t kResCentre = 16u, kResFill = 32u;
constexpr int kResFillShift = 5;

struct TreeArg {
    const int32_t* nodes;
    uint64_t level_off[kMaxLevels + 1];
    uint64_t level_n[kMaxLevels + 1];
    int top;
    uint64_t n_obj;
    int4 root_box;
};

struct Params {
    const hv_tile_req* reqs;
    uint32_t n;
    int rows;                   // pixel rows per CTA strip: 4, 8 or 16
    int strips;                 // strips per tile (256 / rows)
    int parts;                  // CTAs per strip: 1, or 2 / 4 / 8 (128 / 64 / 32 columns each) for batches too small to fill the GPU
    const uint32_t* n_dev;      // if set, the batch size is min(*n_dev, n) (graph launches)
    int mode;
    uchar4 line;
    uchar4 fill;
    uint8_t* out;
    uint32_t tile_bytes;
    TreeArg tree;               // points, segments or polygon edges
    const void* obj;
    TreeArg mtree;              // polygon boxes (polygon layers)
    const int4* mbr_obj;
    const uint32_t* mbr_ids;
    const int4* poly_edges;
    const uint64_t* poly_edge_off;
    uint32_t* status;                 // bit 0: invalid request; bit 1: internal check failed
    unsigned long long* fault;        // first failed check: code << 56 | value
    uint64_t n_poly, n_edges;
    // learned candidate lookup (use_learned): models over the sorted keys of
    // the objects and of the polygon boxes, their halos and side trees
    int use_learned;
    int32_t R_units;            // >= 0: the radius of every tile (buffer analysis), else from r16
    // polygon fill style: anti-aliased fill, and a pattern of pat_w x pat_h
    // RGBA texels (0: none) laid over the global pixel grid
    int fill_aa;
    int pat_w, pat_h;
    const uchar4* pattern;      // device memory, pat_w * pat_h texels
    LModel lm, mlm;
    int32_t halo, mhalo;
    TreeArg side, mside;
    const void* side_obj;
    const uint32_t* side_ids;
    const int4* mside_obj;
    const uint32_t* mside_ids;
    // instrumentation (NULL in normal use): every node, leaf and polygon read
    // is appended as (tile << 38 | kind << 35 | id)
    unsigned long long* log;
    unsigned long long log_cap;
    unsigned long long* log_n;
    // phase profile (instrumented instantiation only): HV_PHASE_* counters
    unsigned long long* phases;
};

// Phase profile.  The instrumented instantiation (kProf) times the phases of
// every CTA with clock64() and adds them up over the launch, in warp-cycles:
// CTA-wide phases (one thread times them, every warp takes part) count their
// cycles times the warps of the CTA; block work counts each warp's own
// cycles.  The indices are the HV_PHASE_* values of the C header.
enum {
    kPTotal = 0, kPPrologue, kPCull, kPBin, kPBlocksCta, kPBlocksWarp, kPLeaf, kPDescend, kPEncode,
    kPCtas, kPBlocks, kPLeafVisits, kPNodeVisits, kPFrontierEntries, kPLeafEmpty, kPLeafDecided, kPN = 16
};

template <bool kProf>
__device__ __forceinline__ long long tick() {
    if constexpr (kProf) return clock64();
    return 0;
}

// kinds of logged reads
constexpr uint32_t kLogNode = 0, kLogLeaf = 1, kLogPolyNode = 2, kLogPolyLeaf = 3, kLogPoly = 4;

__device__ __forceinline__ void log_read(const Params& p, uint32_t kind, uint64_t id, int lane) {
    if (p.log != nullptr && lane == 0) {
        unsigned long long k = atomicAdd(p.log_n, 1ull);
        if (k < p.log_cap)
            p.log[k] = ((unsigned long long)(blockIdx.x / (p.strips * p.parts)) << 38) |
                       ((unsigned long long)kind << 35) | id;
    }
}

// Bounds checks on every index the traversal follows: a failure records the
// first offending value and the access is skipped (the tile is then wrong,
// never the memory).
__device__ __noinline__ void check_failed(const Params& p, uint32_t code, uint64_t v) {
    atomicCAS(p.fault, 0ull, ((unsigned long long)code << 56) | (v & ((1ull << 56) - 1)));
    atomicOr(p.status, 2u);
}

// The frontier is built in two buffers that the cull alternates; the sweep
// reads the final one (f_buf).
struct Front {
    int4 fbox[2][kFCap];
    uint32_t fid[2][kFCap];
    const int32_t* lvl_base[2][kMaxLevels + 1];   // [0]: tree being traversed, [1]: its side tree
    uint32_t lvl_n[2][kMaxLevels + 1];            // nodes per level
    int f_count, f_level, f_buf, next_count;
    int lvl_count[kMaxLevels + 1];
    unsigned long long prof[kPN];   // phase profile of the CTA (kProf only)
};

// Add the cycles since t0 (or a count) to a phase counter of the CTA (one
// lane per warp).
template <bool kProf>
__device__ __forceinline__ void prof_add(Front& sm, int k, unsigned long long v, int lane) {
    if constexpr (kProf) {
        if (lane == 0) atomicAdd(&sm.prof[k], v);
    }
}
template <bool kProf>
__device__ __forceinline__ void prof_since(Front& sm, int k, long long t0, int lane) {
    if constexpr (kProf) prof_add<kProf>(sm, k, (unsigned long long)(clock64() - t0), lane);
}

// Where a traversal reads its objects: a tree's sorted objects (with polygon
// ids for polygon boxes) and the per-level node bases in shared memory.
struct Src {
    const void* obj;
    const uint32_t* ids;
    uint64_t n;
    const int32_t* nodes;        // node array (for the read log)
    const int32_t* const* lvl;   // lvl[l] = first node of level l
    const uint32_t* lvl_n;       // lvl_n[l] = nodes of level l
};

// Level bases of a tree into shared memory slot `slot` (0: the tree being
// traversed, 1: its side tree).
__device__ __forceinline__ void set_levels(Front& sm, int slot, const TreeArg& t, int tid) {
#pragma unroll
    for (int l = 0; l <= kMaxLevels; l++)
        if (tid == l) {
            sm.lvl_base[slot][l] = (l >= 1 && l <= t.top) ? t.nodes + t.level_off[l] * 128 : nullptr;
            // level 0 counts leaves
            sm.lvl_n[slot][l] = l == 0 ? (uint32_t)((t.n_obj + 31) / 32) : (l <= t.top ? (uint32_t)t.level_n[l] : 0u);
        }
}

// Refine the shared frontier breadth first: replace every entry by its
// children that meet the box, one level at a time, while the next level fits
// (the deepest level that fits is kept).  One barrier per level: every level
// counts its entries in a counter of its own, and the loop's state is kept
// by every thread alike.
__device__ void refine(const Params& p, const TreeArg& t, bool fill, Front& sm, int32_t x0, int32_t y0,
                       int32_t x1, int32_t y1, int tid) {
    const int lane = tid & 31, warp = tid >> 5;
    int cur = sm.f_buf, lvl = sm.f_level, cnt = sm.f_count;
    if (tid <= kMaxLevels) sm.lvl_count[tid] = 0;
    __syncthreads();
    while (lvl >= 1 && cnt > 0) {
        const int32_t* base = sm.lvl_base[0][lvl];
        // two entries per step: their boxes are loaded together
        for (int e = warp; e < cnt; e += 2 * kWarps) {
            const int32_t* nd[2];
            uint32_t node[2];
            int4 b[2];
#pragma unroll
            for (int k = 0; k < 2; k++) {
                const int ek = e + k * kWarps;
                nd[k] = nullptr;
                node[k] = 0;
                if (ek < cnt) {
                    node[k] = sm.fid[cur][ek];
                    if (node[k] < sm.lvl_n[0][lvl])
                        nd[k] = base + (uint64_t)node[k] * 128;
                    else if (lane == 0)
                        check_failed(p, 8, ((uint64_t)lvl << 40) | node[k]);
                }
                b[k] = make_int4(kEmptyLo, kEmptyLo, kEmptyHi, kEmptyHi);
                if (nd[k])
                    b[k] = make_int4(__ldg(nd[k] + lane), __ldg(nd[k] + 32 + lane), __ldg(nd[k] + 64 + lane),
                                     __ldg(nd[k] + 96 + lane));
            }
#pragma unroll
            for (int k = 0; k < 2; k++) {
                if (p.log != nullptr && nd[k])
                    log_read(p, fill ? kLogPolyNode : kLogNode, (uint64_t)(nd[k] - t.nodes) >> 7, lane);
                const bool hit = box_hit(b[k], x0, y0, x1, y1);
                const uint32_t m = __ballot_sync(kFull, hit);
                if (m == 0) continue;
                int pos = 0;
                if (lane == 0) pos = atomicAdd(&sm.lvl_count[lvl], __popc(m));
                pos = __shfl_sync(kFull, pos, 0);
                if (hit) {
                    const int slot = pos + __popc(m & ((1u << lane) - 1u));
                    if (slot < kFCap) {
                        sm.fid[cur ^ 1][slot] = node[k] * 32u + (uint32_t)lane;
                        sm.fbox[cur ^ 1][slot] = b[k];
                    }
                }
            }
        }
        __syncthreads();
        const int nc = sm.lvl_count[lvl];
        if (nc > kFCap) break;  // keep the current (coarser) frontier
        cur ^= 1;
        cnt = nc;
        lvl--;
    }
    if (tid == 0) {
        sm.f_buf = cur;
        sm.f_count = cnt;
        sm.f_level = lvl;
    }
    __syncthreads();
}

// Breadth-first cull of a tree against a box into the shared frontier.  It
// starts at the lowest level with at most kFCap / 32 nodes, all of them: their
// children fit the frontier whatever the box, so the boxes of these nodes
// themselves are never needed, and the levels above cost no round.
__device__ void cull(const Params& p, const TreeArg& t, bool fill, Front& sm, int32_t x0, int32_t y0,
                     int32_t x1, int32_t y1, int tid) {
    constexpr uint32_t kSeeds = kFCap / 32;
    static_assert(kSeeds <= kThreads, "one thread per seed");
    int l0 = t.top;
    while (l0 > 1 && t.level_n[l0 - 1] <= kSeeds) l0--;
    const bool meets = t.top > 0 && t.root_box.x <= x1 && t.root_box.z >= x0 && t.root_box.y <= y1 && t.root_box.w >= y0;
    const int seeds = meets ? (int)t.level_n[l0] : 0;
    if (tid < seeds) sm.fid[0][tid] = (uint32_t)tid;
    if (tid == 0) {
        sm.f_buf = 0;
        sm.f_level = l0;
        sm.f_count = seeds;
    }
    __syncthreads();
    refine(p, t, fill, sm, x0, y0, x1, y1, tid);
}

// Learned cull (replaces the breadth-first R-tree cull): cover the strip's
// box, widened by the halo of object extents, with at most kCullCells aligned
// Hilbert cells (a cell's keys are a contiguous run of the sorted order), find each cell's position range through the learned model,
// and turn the ranges into R-tree subtrees at the finest level whose entries
// fit the frontier.  Every object whose centre lies in the box is under one of
// the entries; the sweep then proceeds exactly as after the R-tree cull.
__device__ void learned_cull(const Params& p, const TreeArg& t, const LModel& m, int32_t halo, Front& sm,
                             int32_t bx0, int32_t by0, int32_t bx1, int32_t by1, int tid) {
    __shared__ unsigned long long cnt[kMaxLevels + 1];
    const int64_t lo_g = -(int64_t)kGridHalf, hi_g = (int64_t)kGridHalf - 1;
    const int64_t x0 = max((int64_t)bx0 - halo, lo_g), x1 = min((int64_t)bx1 + halo, hi_g);
    const int64_t y0 = max((int64_t)by0 - halo, lo_g), y1 = min((int64_t)by1 + halo, hi_g);
    // neighbouring cells share subtrees: a hash set in the (idle) second
    // frontier buffer keeps each entry once
    uint32_t* seen = (uint32_t*)sm.fbox[1];
    constexpr int kSeen = 1024;
    for (int i = tid; i < kSeen; i += kThreads) seen[i] = 0u;
    if (tid <= kMaxLevels) cnt[tid] = 0;
    if (tid == 0) {
        sm.f_buf = 0;
        sm.f_count = 0;
        sm.f_level = 0;
        sm.next_count = 0;
    }
    __syncthreads();
    if (t.top == 0 || m.n == 0 || x0 > x1 || y0 > y1) return;
    int k = 0;
    while (k < 31) {
        int64_t nx = ((x1 + kGridHalf) >> k) - ((x0 + kGridHalf) >> k) + 1;
        int64_t ny = ((y1 + kGridHalf) >> k) - ((y0 + kGridHalf) >> k) + 1;
        if (nx * ny <= kCullCells) break;
        k++;
    }
    const int64_t gx0 = (x0 + kGridHalf) >> k, gy0 = (y0 + kGridHalf) >> k;
    const int nx = (int)(((x1 + kGridHalf) >> k) - gx0 + 1), ny = (int)(((y1 + kGridHalf) >> k) - gy0 + 1);
    // kCullSub neighbouring threads (one warp) per cell: its two lookups run
    // at once on two of them, and they share its entries below
    const int cell = tid / kCullSub, sub = tid % kCullSub, lane = tid & 31;
    uint64_t pos = 0;
    if (cell < nx * ny && sub < 2) {
        int64_t cx = ((gx0 + cell % nx) << k) - kGridHalf, cy = ((gy0 + cell / nx) << k) - kGridHalf;
        uint64_t span = (k >= 31) ? (1ull << 62) : (1ull << (2 * k));
        uint64_t klo = (k >= 31) ? 0ull : (hilbert_key((int32_t)cx, (int32_t)cy) & ~(span - 1));
        bool fb;
        pos = learn_lower_bound(m, sub == 0 ? klo : klo + span, &fb);
    }
    const uint64_t plo = __shfl_sync(kFull, pos, lane & ~(kCullSub - 1));
    const uint64_t phi = __shfl_sync(kFull, pos, (lane & ~(kCullSub - 1)) + 1);
    uint64_t a = 1, b = 0;   // leaf range of this thread's cell (empty)
    if (cell < nx * ny && phi > plo) {
        a = plo >> 5;
        b = (phi - 1) >> 5;
    }
    // entries per level: the leaves [a, b] span (b >> 5l) - (a >> 5l) + 1 subtrees of level l
    for (int l = 0; l < t.top; l++)
        if (sub == 0 && a <= b) atomicAdd(&cnt[l], (unsigned long long)((b >> (5 * l)) - (a >> (5 * l)) + 1));
    __syncthreads();
    int lvl = t.top;   // no level fits: fall back to the root alone
    for (int l = 0; l < t.top; l++)
        if (cnt[l] <= (unsigned long long)kFCap) { lvl = l; break; }
    if (lvl == t.top) {
        if (tid == 0) {
            sm.fid[0][0] = 0;
            sm.fbox[0][0] = t.root_box;
            sm.f_count = 1;
            sm.f_level = t.top;
        }
        __syncthreads();
        refine(p, t, false, sm, bx0, by0, bx1, by1, tid);
        return;
    }
    if (a <= b) {
        uint64_t e0 = a >> (5 * lvl), e1 = b >> (5 * lvl);
        const int32_t* par = sm.lvl_base[0][lvl + 1];
        const bool inside = (e1 >> 5) < sm.lvl_n[0][lvl + 1];
        if (!inside) check_failed(p, 9, ((uint64_t)lvl << 40) | (e1 & ((1ull << 40) - 1)));
        for (uint64_t e = e0 + sub; inside && e <= e1; e += kCullSub) {
            const int32_t* nd = par + (e >> 5) * 128;
            int c = (int)(e & 31);
            int4 bb = make_int4(__ldg(nd + c), __ldg(nd + 32 + c), __ldg(nd + 64 + c), __ldg(nd + 96 + c));
            if (bb.x <= bx1 && bb.z >= bx0 && bb.y <= by1 && bb.w >= by0) {
                // at most kFCap distinct entries, so the set never fills
                uint32_t key = (uint32_t)e + 1u, h = (key * 2654435761u) & (kSeen - 1), prev;
                while ((prev = atomicCAS(&seen[h], 0u, key)) != 0u && prev != key) h = (h + 1) & (kSeen - 1);
                if (prev == key) continue;
                int slot = atomicAdd(&sm.next_count, 1);
                if (slot < kFCap) {
                    sm.fid[0][slot] = (uint32_t)e;
                    sm.fbox[0][slot] = bb;
                }
            }
        }
    }
    __syncthreads();
    if (tid == 0) {
        sm.f_count = min(sm.next_count, kFCap);
        sm.f_level = lvl;
    }
    __syncthreads();
    refine(p, t, false, sm, bx0, by0, bx1, by1, tid);
}

// Kernel parts: one per layer kind, and polygon layers in two launches --
// first the fill (kPolyFill: Algorithm 2), which leaves the strip's fill bits
// as a bit mask (MASK layout, 32 bytes per pixel row) at the start of the
// strip's own part of the output, then the outline (the HV_LAYER_POLYGONS
// part: Algorithm 1 over the edges), which reads those bits back, decides
// the samples and encodes the composed strip over them.  Each CTA reads and
// writes only its own strip's part of the output, so the bits never meet
// another CTA's writes.
constexpr int kPolyFill = 3;

// The pattern texel of global pixel (gx, gy).
__device__ __forceinline__ uchar4 fill_texel(const Params& p, uint32_t gx, uint32_t gy) {
    return p.pattern[(gy % (uint32_t)p.pat_h) * (uint32_t)p.pat_w + gx % (uint32_t)p.pat_w];
}

// Byte offset, in a tile's output, of pixel (c, j) (column c a multiple of 32).
__device__ __forceinline__ uint64_t px_offset(int mode, int j, int c) {
    if (mode == HV_MODE_MASK) return (uint64_t)j * (kTile / 8) + (uint64_t)(c >> 3);
    return ((uint64_t)j * kTile + (uint64_t)c) * (mode == HV_MODE_COVERAGE ? 1u : 4u);
}

// The fill launch of a polygon layer hands the outline launch its results in
// the CTA's own part of the output (which the outline overwrites): per pixel
// row of the CTA, at the start of that row's part (cols pixels, at least
// cols / 8 bytes in every mode), a bit per pixel (centre fill), or with the
// anti-aliased fill a byte per pixel holding the number of super-samples
// inside.  This reads them back into the strip's shared results.
__device__ void decode_fill(const Params& p, const uint8_t* tile_out, uint8_t* res, int strip, int col0, int cols,
                            int tid, bool aa_bytes) {
    const int rows = p.rows;
    if (aa_bytes) {
        const int wpr = cols / 4, wsh = __ffs(wpr) - 1;   // words per row, as a shift
        for (int k = tid; k < rows * wpr; k += kThreads) {
            const int jl = k >> wsh, w = k & (wpr - 1);
            const uint32_t v = ((const uint32_t*)(tile_out + px_offset(p.mode, strip * rows + jl, col0)))[w];
            ((uint32_t*)(res + jl * kTile + col0))[w] = (v & 0x07070707u) << kResFillShift;
        }
        return;
    }
    const int wpr = cols / 32, wsh = __ffs(wpr) - 1;
    for (int k = tid; k < rows * wpr; k += kThreads) {
        const int jl = k >> wsh, w = k & (wpr - 1);
        const uint32_t word = ((const uint32_t*)(tile_out + px_offset(p.mode, strip * rows + jl, col0)))[w];
        uint32_t* r4 = (uint32_t*)(res + jl * kTile + col0 + 32 * w);
#pragma unroll
        for (int q = 0; q < 8; q++) {
            const uint32_t b = word >> (4 * q);
            r4[q] = ((b & 1u) ? kResFill : 0u) | ((b & 2u) ? kResFill << 8 : 0u) | ((b & 4u) ? kResFill << 16 : 0u) |
                    ((b & 8u) ? kResFill << 24 : 0u);
        }
    }
}

// The outline launch of a polygon layer encodes the strip composed over the
// fill results: per pixel v outline samples, the fill field (centre, or the
// anti-aliased count), a pattern texel by the global pixel coordinate.
__device__ void encode_polygons(const Params& p, const uint8_t* res, uint8_t* out, int strip, int col0, int cols,
                                uint32_t tile, int tid) {
    const int rows = p.rows;
    const hv_tile_req q = p.reqs[tile];
    const uint32_t gx0 = q.x * (uint32_t)kTile, gy0 = q.y * (uint32_t)kTile + (uint32_t)(strip * rows);
    if (p.mode == HV_MODE_MASK) {
        const int wpr = cols / 32, wsh = __ffs(wpr) - 1;
        if (tid < rows * wpr) {
            const int jl = tid >> wsh, c = col0 + 32 * (tid & (wpr - 1));
            uint32_t word = 0;
            for (int b = 0; b < 32; b++) {
                const uint32_t f = res[jl * kTile + c + b];
                bool filled = (f >> kResFillShift) != 0;
                if (filled && p.pat_w) filled = fill_texel(p, gx0 + c + b, gy0 + jl).w != 0;
                if ((f & kResCentre) || filled) word |= 1u << b;
            }
            *(uint32_t*)(out + px_offset(p.mode, strip * rows + jl, c)) = word;
        }
    } else if (p.mode == HV_MODE_COVERAGE) {
        // 16 pixels (one uint4) per thread and step
        const int upr = cols / 16, ush = __ffs(upr) - 1;
        for (int u = tid; u < rows * upr; u += kThreads) {
            const int jl = u >> ush, c = col0 + 16 * (u & (upr - 1));
            const uint8_t* r = res + jl * kTile + c;
            uint32_t w4[4];
            for (int k = 0; k < 4; k++) {
                uint32_t v = 0;
                for (int b = 0; b < 4; b++) {
                    const uint32_t f = r[4 * k + b];
                    uint32_t fill = f >> kResFillShift;
                    if (fill && p.pat_w && fill_texel(p, gx0 + c + 4 * k + b, gy0 + jl).w == 0) fill = 0;
                    // anti-aliased: the fill count in bits 4-6; else bit 3 for a filled centre
                    const uint32_t cv = __popc(f & 15u) | (p.fill_aa ? fill << 4 : (fill ? 8u : 0u));
                    v |= cv << (8 * b);
                }
                w4[k] = v;
            }
            *(uint4*)(out + px_offset(p.mode, strip * rows + jl, c)) = make_uint4(w4[0], w4[1], w4[2], w4[3]);
        }
    } else {
        // 4 pixels (one uint4) per thread and step
        const int upr = cols / 4, ush = __ffs(upr) - 1;
        for (int u = tid; u < rows * upr; u += kThreads) {
            const int jl = u >> ush, c = col0 + 4 * (u & (upr - 1));
            uint32_t w[4];
            for (int b = 0; b < 4; b++) {
                uint32_t f = res[jl * kTile + c + b];
                uint32_t v = __popc(f & 15u);
                uint32_t a = (255u * v + 2u) >> 2;
                // fill count: 0..4 anti-aliased, else 4 for a filled centre
                uint32_t fc = f >> kResFillShift;
                if (!p.fill_aa && fc) fc = 4;
                uchar4 fill = p.fill;
                if (fc && p.pat_w) {
                    fill = fill_texel(p, gx0 + c + b, gy0 + jl);
                    if (fill.w == 0) fc = 0;   // a transparent texel: not filled
                }
                uint32_t rgba = 0;
                if (fc == 4) {
                    uint32_t r = (p.line.x * a + fill.x * (255u - a) + 127u) / 255u;
                    uint32_t g = (p.line.y * a + fill.y * (255u - a) + 127u) / 255u;
                    uint32_t bl = (p.line.z * a + fill.z * (255u - a) + 127u) / 255u;
                    rgba = r | (g << 8) | (bl << 16) | (255u << 24);
                } else if (fc) {
                    // the outline over a partly covered fill
                    const uint32_t af = (255u * fc + 2u) >> 2;
                    const uint32_t A = (255u * a + af * (255u - a) + 127u) / 255u;
                    const uint32_t den = 255u * A, wf = af * (255u - a), wl = a * 255u;
                    const uint32_t r = (p.line.x * wl + fill.x * wf + 127u * A) / den;
                    const uint32_t g = (p.line.y * wl + fill.y * wf + 127u * A) / den;
                    const uint32_t bl = (p.line.z * wl + fill.z * wf + 127u * A) / den;
                    rgba = r | (g << 8) | (bl << 16) | (A << 24);
                } else if (v) {
                    rgba = (uint32_t)p.line.x | ((uint32_t)p.line.y << 8) | ((uint32_t)p.line.z << 16) | (a << 24);
                }
                w[b] = rgba;
            }
            *(uint4*)(out + px_offset(p.mode, strip * rows + jl, c)) = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
}

#include "hv_sweep.cuh"

TreeArg tree_arg(const TreeView& v) {
    TreeArg a;
    a.nodes = v.nodes;
    for (int l = 0; l <= kMaxLevels; l++) {
        a.level_off[l] = v.level_off[l];
        a.level_n[l] = v.level_n[l];
    }
    a.top = v.top;
    a.n_obj = v.n_obj;
    a.root_box = v.root_box;
    return a;
}

}  // namespace

LModel learned_model(const LearnedView& v);

uint32_t render_launch_count(Layer* L, int) { return L->kind == HV_LAYER_POLYGONS ? 2u : 1u; }

bool fill_style_ok(const hv_fill_style* f) {
    if (!f) return true;
    if (f->flags & ~(uint32_t)HV_FILL_AA) return false;
    if (f->pattern_w == 0 && f->pattern_h == 0) return true;
    if (f->pattern_w < 1 || f->pattern_h < 1 || f->pattern_w > kMaxPattern || f->pattern_h > kMaxPattern ||
        !f->pattern_rgba)
        return false;
    for (uint32_t k = 0; k < f->pattern_w * f->pattern_h; k++)
        if (f->pattern_rgba[4 * k + 3] != 0 && f->pattern_rgba[4 * k + 3] != 255) return false;
    return true;
}

int launch_render(Layer* L, const hv_tile_req* d_reqs, uint32_t n, int mode, int index_kind,
                  const hv_style* style, uint8_t* d_out, cudaStream_t stream, const RenderLog* log,
                  const uint32_t* n_dev, int32_t R_units, const hv_fill_style* fill, const void* pattern_dev) {
    (void)index_kind;
    if (n == 0) return HV_OK;
    Params p;
    memset(&p, 0, sizeof(p));
    p.R_units = R_units < 0 ? -1 : R_units;
    if (fill && L->kind == HV_LAYER_POLYGONS) {
        if (!fill_style_ok(fill)) {
            set_error("invalid fill style (flags, pattern size 1..16, texel alpha 0 or 255)");
            return HV_EINVAL;
        }
        p.fill_aa = (fill->flags & HV_FILL_AA) ? 1 : 0;
        if (fill->pattern_w) {
            if (!pattern_dev) {
                set_error("a fill pattern needs its device copy");
                return HV_EINVAL;
            }
            p.pat_w = (int)fill->pattern_w;
            p.pat_h = (int)fill->pattern_h;
            p.pattern = (const uchar4*)pattern_dev;
        }
    }
    p.reqs = d_reqs;
    p.n = n;
    p.n_dev = n_dev;
    p.mode = mode;
    if (style) {
        p.line = make_uchar4(style->line_rgba[0], style->line_rgba[1], style->line_rgba[2], 0);
        p.fill = make_uchar4(style->fill_rgba[0], style->fill_rgba[1], style->fill_rgba[2], 0);
    }
    p.out = d_out;
    p.tile_bytes = (uint32_t)hv_tile_bytes(mode);
    p.tree = tree_arg(L->tree.view);
    p.obj = L->obj;
    p.mtree = tree_arg(L->mbr_tree.view);
    p.mbr_obj = L->mbr_obj;
    p.mbr_ids = L->mbr_ids;
    p.poly_edges = L->poly_edges;
    p.poly_edge_off = L->poly_edge_off;
    p.status = L->status;
    p.fault = (unsigned long long*)(L->status + 2);
    p.n_poly = L->n_poly;
    p.n_edges = L->n_src;
    if (index_kind == HV_INDEX_LEARNED) {
        const LearnedView& a = L->learned.view;
        const LearnedView& b = L->mbr_learned.view;
        if (!a.ready || (L->kind == HV_LAYER_POLYGONS && !b.ready)) {
            set_error("learned index not built");
            return HV_ESTATE;
        }
        p.use_learned = 1;
        p.lm = learned_model(a);
        p.halo = a.halo;
        p.side = tree_arg(a.outliers);
        p.side_obj = a.outlier_obj;
        p.side_ids = a.outlier_ids;
        if (L->kind == HV_LAYER_POLYGONS) {
            p.mlm = learned_model(b);
            p.mhalo = b.halo;
            p.mside = tree_arg(b.outliers);
            p.mside_obj = b.outlier_obj;
            p.mside_ids = b.outlier_ids;
        }
    }
    if (log) {
        p.log = (unsigned long long*)log->log;
        p.log_cap = log->cap;
        p.log_n = (unsigned long long*)log->count;
        p.phases = (unsigned long long*)log->phases;
    }
    const bool prof = p.phases != nullptr;
    // Strip height: 16 rows (16 CTAs per tile) when the batch fills the GPU, 8 or
    // 4 rows for small batches so that the densest strips, which end last, are
    // shared over more SMs.  Smaller strips repeat the cull.  Measured at z 8-14 on
    // three layers each: points and polygons gain from 8 rows up to 151 tiles
    // (90 tiles: 117 -> 99 us and 208 -> 174 us; 250 tiles would lose: 177 -> 191
    // us for points), points from 4 rows up to 75 tiles (45 tiles: 75 -> 68 us), polygons
    // only up to 37 (60 tiles: 150 -> 175 us).  Segments, whose strips cost
    // little more than their cull, change at 76 and 38 tiles (60 tiles in 4 rows:
    // 18 -> 27 us).
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const uint64_t resident = (uint64_t)sms * 4;
    const uint64_t few16 = (L->kind == HV_LAYER_LINES ? 2 : 4) * resident, few8 = (L->kind == HV_LAYER_POINTS ? 4 : 2) * resident;
    p.rows = (uint64_t)n * 16 >= few16 ? 16 : ((uint64_t)n * 32 >= few8 ? 8 : 4);
    p.strips = kTile / p.rows;
    // batches too small for the GPU even in 4-row strips also split each
    // strip into 2, 4 or 8 column parts (a CTA per 128, 64 or 32 columns), as
    // long as every CTA is resident at once: a tile's densest part decides its
    // time.  36 single tiles of 10M points: 933 us in all with at most 4 parts, 776
    // with 8; of 200,000 polygons 1,852 -> 1,665; of 5M segments 467 -> 472.  Twice as
    // many CTAs (8 parts for two tiles) made sparse tiles slower (6.4 -> 9.2 us).
    p.parts = 1;
    if (p.rows == 4 && !prof)
        while (p.parts < 8 && (uint64_t)n * p.strips * p.parts * 2 <= resident) p.parts *= 2;
    uint64_t grid = (uint64_t)n * p.strips * p.parts;
    if (grid > 0x7fffffffull) {
        set_error("too many tiles in one call");
        return HV_EINVAL;
    }
    if (prof) {
        // the instrumented instantiations (phase profile, full-width strips);
        // polygon layers profile their two launches (fill, outline) into two
        // sets of counters
        if (L->kind == HV_LAYER_POINTS)
            k_sweep<HV_LAYER_POINTS, true, false><<<(unsigned)grid, kThreads, 0, stream>>>(p);
        else if (L->kind == HV_LAYER_LINES)
            k_sweep<HV_LAYER_LINES, true, false><<<(unsigned)grid, kThreads, 0, stream>>>(p);
        else {
            k_sweep<kPolyFill, true, false><<<(unsigned)grid, kThreads, 0, stream>>>(p);
            Params q = p;
            q.phases = p.phases + kPN;
            k_sweep<HV_LAYER_POLYGONS, true, false><<<(unsigned)grid, kThreads, 0, stream>>>(q);
        }
    } else if (p.parts > 1) {
        if (L->kind == HV_LAYER_POINTS)
            k_sweep<HV_LAYER_POINTS, false, true><<<(unsigned)grid, kThreads, 0, stream>>>(p);
        else if (L->kind == HV_LAYER_LINES)
            k_sweep<HV_LAYER_LINES, false, true><<<(unsigned)grid, kThreads, 0, stream>>>(p);
        else {
            k_sweep<kPolyFill, false, true><<<(unsigned)grid, kThreads, 0, stream>>>(p);
            k_sweep<HV_LAYER_POLYGONS, false, true><<<(unsigned)grid, kThreads, 0, stream>>>(p);
        }
    } else if (L->kind == HV_LAYER_POINTS)
        k_sweep<HV_LAYER_POINTS, false, false><<<(unsigned)grid, kThreads, 0, stream>>>(p);
    else if (L->kind == HV_LAYER_LINES)
        k_sweep<HV_LAYER_LINES, false, false><<<(unsigned)grid, kThreads, 0, stream>>>(p);
    else {
        // the fill first: the outline reads its bits and writes the tile
        k_sweep<kPolyFill, false, false><<<(unsigned)grid, kThreads, 0, stream>>>(p);
        k_sweep<HV_LAYER_POLYGONS, false, false><<<(unsigned)grid, kThreads, 0, stream>>>(p);
    }
    HV_CUDA(cudaGetLastError());
    return HV_OK;
}

}  // namespace hv
