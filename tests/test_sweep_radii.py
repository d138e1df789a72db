"""Segment rows of the strip sweep at every ratio of radius to sample spacing
(ground radii at street zooms reach 2^26 spacings): the kernel's own piece_row
and draw_row, compiled for the host, against the 128-bit predicate on every
column in reach, for pieces whose capsule passes within a few units, or a few
spacings, of a sample of the strip, at every slope, with contacts at the
segment's inside and at its ends."""
import ctypes
import math
import random

import pytest

import sweep_host

ENTRIES = r"""
static bool inside(int4 o, int64_t x, int64_t y, int64_t R) {   // the definition, in 128 bits
    typedef __int128 W;
    const W dx = (int64_t)o.z - o.x, dy = (int64_t)o.w - o.y, wx = x - o.x, wy = y - o.y, R2 = (W)R * R;
    const W t = wx * dx + wy * dy, L = dx * dx + dy * dy;
    if (t <= 0) return wx * wx + wy * wy <= R2;
    if (t >= L) return (W)(x - o.z) * (x - o.z) + (W)(y - o.w) * (y - o.w) <= R2;
    const W c = wx * dy - wy * dx;                               // |c| < 2^64, L < 2^63, R2 < 2^59
    const unsigned __int128 a = (unsigned __int128)(c < 0 ? -c : c);
    return a < ((unsigned __int128)1 << 64) && a * a <= (unsigned __int128)R2 * (unsigned __int128)L;
}
static int64_t fdiv(int64_t a, int64_t b) { return a / b - (a % b != 0 && (a < 0) != (b < 0)); }
// the box of piece k of m, as the index build forms it
static int4 piece_box(int4 s, int64_t k, int64_t m) {
    const int64_t dx = (int64_t)s.z - s.x, dy = (int64_t)s.w - s.y;
    const int64_t xa = s.x + fdiv(dx * k, m), xb = s.x + fdiv(dx * (k + 1), m);
    const int64_t ya = s.y + fdiv(dy * k, m), yb = s.y + fdiv(dy * (k + 1), m);
    return make_int4((int)max(min(xa, xb), (int64_t)min(s.x, s.z)), (int)max(min(ya, yb), (int64_t)min(s.y, s.w)),
                     (int)min(max(xa, xb) + 1, (int64_t)max(s.x, s.z)), (int)min(max(ya, yb) + 1, (int64_t)max(s.y, s.w)));
}
struct Result { int64_t wrong, columns, covered, rows; };
// the rows of one piece, at most `most` of them
static void compare(const Lattice& g, int4 o, int4 pb, int most, std::mt19937_64& rng, Result* res) {
    const int32_t x0 = rel32(pb.x, g.xc), y0 = rel32(pb.y, g.yc), x1 = rel32(pb.z, g.xc), y1 = rel32(pb.w, g.yc);
    const int r0 = max(g.hh - ((g.R - y0) >> g.s), 0), r1 = min(((y1 + g.R) >> g.s) + g.hh, 2 * g.hh - 1);
    const int clo = max(g.hw - ((g.R - x0) >> g.s), 0), chi = min(((x1 + g.R) >> g.s) + g.hw, 2 * g.hw - 1);
    if (r0 > r1 || clo > chi) return;
    const PieceRow q = piece_row(g, o, x0, y0, x1, y1, clo, chi);
    for (int n = 0; n < most && n <= r1 - r0; n++) {
        const int r = r1 - r0 < most ? r0 + n : r0 + (int)(rng() % (uint64_t)(r1 - r0 + 1));
        uint32_t bits[kSampleRows * kBitStride] = {};
        draw_row(bits, g, q, &o, r);
        for (int c = 0; c < 2 * g.hw; c++) {
            const bool got = (bits[r * kBitStride + (c >> 5)] >> (c & 31)) & 1u;
            const bool want = c >= clo && c <= chi &&
                              inside(o, (int64_t)g.xc + (int64_t)(c - g.hw) * (1 << g.s), (int64_t)g.yc + (int64_t)(r - g.hh) * (1 << g.s), g.R);
            res->wrong += got != want;
            res->covered += want;
        }
        res->columns += 2 * g.hw;
        res->rows++;
    }
}
static Lattice lattice(int s, int hw, int hh, int32_t xc, int32_t yc, int32_t R) {
    Lattice g;
    g.s = s, g.hw = hw, g.hh = hh, g.xc = xc, g.yc = yc, g.R = R, g.R2 = (int64_t)R * R;
    g.rs = max(32 - __clz(R) - 6, 0), g.narrow = R <= kNarrow;
    return g;
}
// radii of 2^lo .. 2^hi sample spacings
extern "C" void fuzz_rows(uint64_t seed, int64_t n, double lo, double hi, Result* res) {
    std::mt19937_64 rng(seed);
    auto u = [&](double a, double b) { return a + (b - a) * ((double)(rng() >> 11) * 0x1p-53); };
    auto pick = [&](int64_t a, int64_t b) { return a + (int64_t)(rng() % (uint64_t)(b - a + 1)); };
    const double kPi = 3.14159265358979323846;
    for (int64_t i = 0; i < n;) {
        const int s = (int)pick(3, 21);
        const double h = std::ldexp(1.0, s), Rd = std::exp2(u(lo, hi)) * h;
        if (Rd > 536870912.0) continue;
        const int32_t R = (int32_t)Rd;
        const int hw = 16 << pick(0, 4), hh = 2 << pick(0, 3);
        const int64_t zone = ((1ll << 30) >> s) - hw;
        if (zone < 0) continue;
        const Lattice g = lattice(s, hw, hh, (int32_t)(pick(-zone, zone) * (1 << s) + (1 << s >> 1)),
                                  (int32_t)(pick(-zone, zone) * (1 << s) + (1 << s >> 1)), R);
        const double px = g.xc + (double)pick(-hw, hw - 1) * h, py = g.yc + (double)pick(-hh, hh - 1) * h;
        const int slope = (int)pick(0, 5);
        double th = slope == 0 ? 0.0 : slope == 1 ? kPi / 2 : u(0, 2 * kPi);
        if (slope == 2) th = std::pow(10.0, u(-7, -0.5)) * (rng() & 1 ? 1 : -1);
        if (slope == 3) th = kPi / 2 + std::pow(10.0, u(-7, -0.5)) * (rng() & 1 ? 1 : -1);
        const double d = R + (rng() & 1 ? (double)pick(-3, 3) : u(-2, 2) * h);
        const double size = rng() & 1 ? h * std::exp2(u(-3, 12)) : std::exp2(u(s, 30));
        const double side = rng() & 1 ? 1 : -1, along = rng() % 4 ? u(0, 1) : (double)(rng() & 1);
        const double turn = along == 0.0 || along == 1.0 ? u(-kPi / 2, kPi / 2) : 0.0;   // end caps: any direction outwards
        const double nx = -std::sin(th + turn) * side, ny = std::cos(th + turn) * side;
        const double ax = px + nx * d - std::cos(th) * size * along, ay = py + ny * d - std::sin(th) * size * along;
        const double bx = ax + std::cos(th) * size, by = ay + std::sin(th) * size;
        const double e = 1073741823.0;
        if (std::fabs(ax) > e || std::fabs(ay) > e || std::fabs(bx) > e || std::fabs(by) > e) {
            if (rng() % 8) continue;   // mostly drawn again; some cut off at the grid
        }
        const int4 o = make_int4((int)std::lround(max(min(ax, e), -e)), (int)std::lround(max(min(ay, e), -e)),
                                 (int)std::lround(max(min(bx, e), -e)), (int)std::lround(max(min(by, e), -e)));
        const int64_t m = rng() & 1 ? 1 : pick(1, 64);
        compare(g, o, piece_box(o, pick(0, m - 1), m), 4, rng, res);
        i++;
    }
}
"""


ENTRIES += r"""
extern "C" int reach_table(int32_t R, int32_t* reach) {
    const Lattice g = lattice(3, 256, 16, 0, 0, R);
    for (int tid = 0; tid < 256; tid++) fill_reach(reach, g, tid);
    return g.rs;
}
extern "C" int covers(int s, int hw, int hh, int32_t xc, int32_t yc, int32_t R, int32_t x0, int32_t y0, int32_t x1, int32_t y1) {
    const Lattice g = lattice(s, hw, hh, xc, yc, R);
    return covers_strip(g, rel32(x0, xc), rel32(y0, yc), rel32(x1, xc), rel32(y1, yc));
}
extern "C" int32_t reach_by_root(int32_t R, int32_t f) { return reach_width<true>(nullptr, lattice(3, 256, 16, 0, 0, R), f); }
"""
ENTRIES += r"""
static int4 turned(int4 o, int how) {   // mirrored, transposed, ends exchanged
    if (how & 1) o = make_int4(o.y, o.x, o.w, o.z);
    if (how & 2) o = make_int4(o.z, o.w, o.x, o.y);
    return o;
}
// strips along the grid's borders at zooms 0 to 2 and segments from there to the
// opposite border, cut into many pieces: coordinate differences of up to 2^31 + half a spacing
extern "C" void border_rows(uint64_t seed, int64_t n, Result* res) {
    std::mt19937_64 rng(seed);
    auto pick = [&](int64_t a, int64_t b) { return a + (int64_t)(rng() % (uint64_t)(b - a + 1)); };
    const int64_t lo = -(1ll << 30), hi = (1ll << 30) - 1;
    for (int64_t i = 0; i < n; i++) {
        const int z = (int)pick(0, 2), centres = (int)(rng() & 1), L = 23 - z, s = centres ? L : L - 1;
        const int rows = 4 << pick(0, 2), cols = rows == 4 ? 32 << pick(0, 3) : 256;
        const int64_t half = 1ll << s >> 1, ps = 1ll << L;
        const int64_t col0 = rng() & 1 ? 0 : pick(0, 256 / cols - 1) * cols, strip = rng() & 1 ? 0 : pick(0, 256 / rows - 1);
        const int32_t R = (int32_t)(pick(1, rng() & 1 ? 3 : 64) << (19 - z));
        Lattice g = lattice(s, centres ? cols / 2 : cols, centres ? rows / 2 : rows,
                                  (int32_t)(lo + (col0 + cols / 2) * ps + half), (int32_t)(lo + (strip * rows + rows / 2) * ps + half), R);
        const int64_t far_end = pick(0, 3) ? (1ll << 30) - half + pick(-2, 1) : hi - pick(0, 1 << 23);
        const int64_t x = max(lo, min(hi, lo + pick(0, 40) * half + pick(-2, 2)));
        const int64_t slant = pick(0, 2) == 0 ? pick(0, 1 << 24) : 0;
        const int how = (int)pick(0, 3);
        int4 o = turned(make_int4((int)x, (int)(lo + (rng() & 1 ? 0 : pick(0, 1 << 22))), (int)min(hi, x + slant), (int)min(hi, far_end)), how);
        if (rng() & 1) {   // the right and bottom borders
            g.xc = -g.xc + (1 << s), g.yc = -g.yc + (1 << s);
            o = make_int4((int)min(hi, -(int64_t)o.x), (int)min(hi, -(int64_t)o.y), (int)min(hi, -(int64_t)o.z), (int)min(hi, -(int64_t)o.w));
        }
        const int64_t m = 1 << pick(0, 12), k = rng() & 1 ? pick(0, min(m - 1, (int64_t)8)) : pick(0, m - 1);
        compare(g, o, piece_box(o, how & 2 ? m - 1 - k : k, m), 6, rng, res);
    }
}
"""
ENTRIES += r"""
// grid-wide segments in wide pieces (or whole) over strips that their boxes cover: exact tests taken
extern "C" int64_t wide_pieces(uint64_t seed, int64_t n, int32_t R, Result* res) {
    std::mt19937_64 rng(seed);
    auto pick = [&](int64_t a, int64_t b) { return a + (int64_t)(rng() % (uint64_t)(b - a + 1)); };
    const int64_t before = g_tests, e = (1ll << 30) - 1;
    for (int64_t i = 0; i < n; i++) {
        const int s = (int)pick(6, 18), hw = 256, hh = 2 << pick(0, 3);
        const int64_t zone = ((1ll << 30) >> s) - hw;
        const Lattice g = lattice(s, hw, hh, (int32_t)(pick(-zone, zone) * (1 << s) + (1 << s >> 1)),
                                  (int32_t)(pick(-zone, zone) * (1 << s) + (1 << s >> 1)), R < 0 ? -R << s >> 3 : R);
        // through a point within a piece's extent of the strip
        const int64_t m = pick(1, 4), near = 1ll << pick(s, 29);
        const int64_t px = max(-e, min(e, g.xc + pick(-near, near))), py = max(-e, min(e, g.yc + pick(-near, near)));
        const int4 o = make_int4((int)pick(-e, e), (int)pick(-e, e), 0, 0);
        const int64_t bx = 2 * px - o.x, by = 2 * py - o.y;
        if (bx < -e || bx > e || by < -e || by > e) continue;
        compare(g, make_int4(o.x, o.y, (int)bx, (int)by), piece_box(make_int4(o.x, o.y, (int)bx, (int)by), pick(0, m - 1), m), 4, rng, res);
    }
    return g_tests - before;
}
"""
ENTRIES += r"""
// level segments (edges of large squares) whose border lies within a unit or so of a sample row: the most tests of one row
extern "C" int64_t grazing_level(uint64_t seed, int64_t n, Result* res) {
    std::mt19937_64 rng(seed);
    auto pick = [&](int64_t a, int64_t b) { return a + (int64_t)(rng() % (uint64_t)(b - a + 1)); };
    int64_t most = 0;
    for (int64_t i = 0; i < n; i++) {
        const int s = (int)pick(6, 14), hw = 256, hh = 2 << pick(0, 3);
        const int64_t zone = (1ll << 24) >> s, h = 1ll << s;
        const Lattice g = lattice(s, hw, hh, (int32_t)(pick(-zone, zone) * h + h / 2), (int32_t)(pick(-zone, zone) * h + h / 2),
                                  (int32_t)max(h * pick(1, 64) / 16, (int64_t)1));
        const int64_t y = g.yc + pick(-hh, hh - 1) * h + (rng() & 1 ? 1 : -1) * (g.R + pick(-2, 1));
        const int64_t x = g.xc + pick(-300, 300) * h, d = pick(h, 1 << 24), a = pick(0, d);
        const int4 o = make_int4((int)(x - a), (int)y, (int)(x - a + d), (int)y);
        for (int k = 0; k < 3; k++) {
            const int64_t before = g_tests, rows = res->rows;
            compare(g, o, piece_box(o, 0, 1), 1, rng, res);
            if (res->rows > rows) most = max(most, g_tests - before);
        }
    }
    return most;
}
"""


class Result(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int64) for n in ("wrong", "columns", "covered", "rows")]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return sweep_host.library(tmp_path_factory.mktemp("sweep"), ENTRIES)


@pytest.mark.parametrize("lo, hi", [(-4, 7), (7, 10), (10, 14), (14, 18), (18, 22), (22, 26)])
def test_rows_equal_the_predicate(lib, lo, hi):
    res = Result()
    lib.fuzz_rows(ctypes.c_uint64(1000 + lo), ctypes.c_int64(60_000), ctypes.c_double(lo), ctypes.c_double(hi),
                  ctypes.byref(res))
    assert res.rows > 50_000 and 0.05 < res.covered / res.columns < 0.95
    assert res.wrong == 0, (res.wrong, res.columns)


@pytest.mark.parametrize("lo, hi", [(-24, -10), (-10, -4)])
def test_rows_at_radii_of_a_few_units(lib, lo, hi):
    res = Result()
    lib.fuzz_rows(ctypes.c_uint64(7 - lo), ctypes.c_int64(60_000), ctypes.c_double(lo), ctypes.c_double(hi),
                  ctypes.byref(res))
    assert res.rows > 20_000 and res.covered > 0
    assert res.wrong == 0, (res.wrong, res.columns)


@pytest.mark.parametrize("R", [0, 1, 999, -1, -8, -64])     # units; below zero: eighths of a spacing
def test_wide_pieces_take_few_exact_tests(lib, R):
    """A piece's box may cover the strip while its line passes far away or crosses
    a few columns of a row: an exact test for a column of every other row at most
    on average, where testing the box's columns would take up to 512 a row."""
    res = Result()
    lib.wide_pieces.restype = ctypes.c_int64
    tests = lib.wide_pieces(ctypes.c_uint64(9), ctypes.c_int64(40_000), ctypes.c_int32(R), ctypes.byref(res))
    assert res.rows > 10_000 and res.wrong == 0, (res.rows, res.wrong)
    assert tests < res.rows / 2, (tests, res.rows)


def test_grazing_level_segments_take_no_run_of_tests(lib):
    """A level segment just above or below a row left up to 512 columns doubtful; its
    distance from the row is a whole number, so that the row is decided at once (rows
    that do not graze: one test at most at either end)."""
    res = Result()
    lib.grazing_level.restype = ctypes.c_int64
    most = lib.grazing_level(ctypes.c_uint64(2), ctypes.c_int64(100_000), ctypes.byref(res))
    assert res.rows > 30_000 and res.covered > 0 and res.wrong == 0
    assert most <= 2, most


def test_rows_at_the_grid_border(lib):
    res = Result()
    lib.border_rows(ctypes.c_uint64(3), ctypes.c_int64(40_000), ctypes.byref(res))
    assert res.rows > 20_000 and res.covered > 0
    assert res.wrong == 0, (res.wrong, res.columns)


def test_reach_table_is_an_upper_bound(lib):
    """reach[k] bounds the half-width of every row distance f with f >> rs = k
    (the largest is f = k << rs), at radii that are no float (above 2^24) as well."""
    rng = random.Random(5)
    radii = [0, 1, 2, 63, 64, 65, 46340, 46341] + [(1 << b) + d for b in range(6, 29) for d in (-1, 0, 1, 15)]
    radii += [(1 << 29) - 1, 1 << 29] + [int(2 ** rng.uniform(0, 29)) for _ in range(2000)]
    radii += [rng.randrange(1 << 24, 1 << 29) for _ in range(4000)]
    radii += [(rng.randrange(33, 64) << (24 - 5 + b)) + rng.randrange(1, 40) for b in range(5) for _ in range(400)]
    table = (ctypes.c_int32 * 64)()
    for R in (r for r in radii if 0 <= r <= 1 << 29):
        rs = lib.reach_table(R, table)
        for k in range((R >> rs) + 1):
            f = k << rs
            assert math.isqrt(R * R - f * f) <= table[k] <= R, (R, k, table[k])


def test_reach_by_root_is_a_close_upper_bound(lib):
    rng = random.Random(6)
    lib.reach_by_root.restype = ctypes.c_int32
    for i in range(100_000):
        R = rng.randrange(1, 1 << 29) >> rng.randrange(0, 22) if i > 100 else (1 << 29) - i
        f = rng.choice([0, R, max(R - rng.randrange(0, 50), 0), rng.randrange(0, R + 1)])
        w = math.isqrt(R * R - f * f)
        assert w <= lib.reach_by_root(R, f) <= min(R, w + 2 + (w >> 18)), (R, f)


def test_box_that_covers_a_strip(lib):
    """covers_strip against the distances of the strip's corner samples to the box's
    corners: never true for a box that does not cover, and true unless it only just does."""
    rng = random.Random(7)
    seen = [0, 0]
    for _ in range(50_000):
        s, hw, hh = rng.randrange(3, 23), 16 << rng.randrange(5), 2 << rng.randrange(4)
        h = 1 << s
        if hw * h > 1 << 30:
            continue
        zone = ((1 << 30) - hw * h) // h
        xc, yc = (rng.randrange(-zone, zone + 1) * h + h // 2 for _ in range(2))
        R = min(1 << 29, int(hw * h * rng.choice([1, 1.001, 1.01, 1.5, 4])) + rng.randrange(-2, 3))
        near = rng.choice([4, h, R // 8 + 1, 1 << 30])
        x0, y0 = (max(-2 ** 30, min(2 ** 30 - 1, c + rng.randrange(-near, near))) for c in (xc, yc))
        x1, y1 = (min(2 ** 30 - 1, v + rng.randrange(0, rng.choice([2, h, R // 8 + 1]))) for v in (x0, y0))
        far = max((x - a) ** 2 + (y - b) ** 2 for x in (x0, x1) for y in (y0, y1)
                  for a in (xc - hw * h, xc + (hw - 1) * h) for b in (yc - hh * h, yc + (hh - 1) * h))
        got = bool(lib.covers(s, hw, hh, xc, yc, R, x0, y0, x1, y1))
        assert not got or far <= R * R
        assert got or far + 3 * h * R + (R * R >> 17) > R * R      # (a column and row more than the strip has, and rounding)
        seen[got] += 1
    assert min(seen) > 5000, seen
