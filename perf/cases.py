"""The work a user of the tile renderer has it do, as measurable cases.

Each case is a plain dict.  ``prepare`` makes the layer (and its index, the
requests, the style, the output buffer or the server) that a user's program
holds before a call; ``run`` is one pass through the public entry points of
``paper_2005_12489_gb300.hv``; ``work`` is what a pass cannot do without.

Layers are synthetic and made on the GPU from the seed alone: clustered points
(a Gaussian mixture with uniform noise, like GPS or cell-tower points),
polylines as random walks around city centres (like roads), star polygons
around mixture centres (like building footprints).  Requested tiles are
density weighted: a random object, a random zoom, the tile that holds it.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2005_12489_gb300 import hv

GRID = 1 << 31
HALF = 1 << 30
MODES = {"mask": hv.HV_MODE_MASK, "coverage": hv.HV_MODE_COVERAGE, "rgba": hv.HV_MODE_RGBA}
OPS = {"and": hv.HV_OVERLAY_AND, "or": hv.HV_OVERLAY_OR, "xor": hv.HV_OVERLAY_XOR, "diff": hv.HV_OVERLAY_DIFF}
LINE, FILL = (230, 40, 20), (30, 90, 200)


def listed():
    return [
        # one tile for an interactive client: latency and launches are what counts
        dict(name="points_one_tile", do="render", kind="points", n=10_000_000, tiles=1, z0=8, z1=14, r16=32,
             mode="rgba", index="rtree", host=False),
        # a small layer's whole low-zoom pyramid, 1 px, as hit-test masks
        dict(name="points_pyramid", do="render", kind="uniform", n=100_000, tiles=0, z0=0, z1=4, r16=16,
             mode="mask", index="rtree", host=False),
        # the headline batch: 100M clustered points, 2 px, RGBA
        dict(name="points_batch", do="render", kind="points", n=100_000_000, tiles=4000, z0=8, z1=14, r16=32,
             mode="rgba", index="rtree", host=False),
        # heat-map input: coverage counts at 3 px through the learned index
        dict(name="points_coverage_learned", do="render", kind="points", n=12_345_679, tiles=317, z0=6, z1=15,
             r16=48, mode="coverage", index="learned", host=False),
        # a browser's screen of road tiles, host requests in, pinned host tiles out
        dict(name="lines_view", do="render", kind="lines", n=5_000_000, tiles=24, z0=8, z1=16, r16=16,
             mode="rgba", index="rtree", host=True),
        # the linestring batch: 50M segments, 1 px half-width
        dict(name="lines_batch", do="render", kind="lines", n=50_000_000, tiles=4000, z0=6, z1=16, r16=16,
             mode="rgba", index="rtree", host=False),
        # the polygon batch: 2M polygons, fill and 1 px outline
        dict(name="polygons_batch", do="render", kind="polygons", n=2_000_000, tiles=1000, z0=4, z1=14, r16=8,
             mode="rgba", index="rtree", host=False),
        # a screen of styled polygons: anti-aliased fill with a pattern
        dict(name="polygons_styled", do="styled", kind="polygons", n=200_000, tiles=33, z0=6, z1=15, r16=16,
             mode="rgba", index="rtree", host=False),
        # buffer and overlay analysis: roads' buffer within polygons' buffer, one ground radius for all tiles
        dict(name="overlay_lines_polygons", do="overlay", n=5_000_000, n2=200_000, tiles=60, z0=8, z1=13,
             radius=60_000, radius2=25_000, op="and"),
        # a burst of requests of browsing sessions to the tile server (a point and a line layer)
        dict(name="serve_burst", do="serve", n=10_000_000, n2=5_000_000, tiles=64, z0=6, z1=16, r16=24, mode="rgba"),
        # registering a layer: load, index, first view
        dict(name="points_register", do="register", kind="points", n=100_000_000, tiles=24, z0=8, z1=14, r16=32,
             mode="rgba", index="rtree"),
        # registering a road layer with the learned index as well
        dict(name="lines_register_learned", do="register", kind="lines", n=5_000_000, tiles=24, z0=8, z1=16, r16=16,
             mode="rgba", index="learned"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["render"] * 6 + ["styled", "overlay", "serve", "register"])
    z0 = rng.randint(4, 9)
    z1 = z0 + rng.randint(3, 8)
    r16 = rng.randint(8, 48)
    mode = rng.choice(["rgba", "rgba", "coverage", "mask"])
    index = rng.choice(["rtree", "rtree", "rtree", "learned"])
    if do == "overlay":
        return dict(do=do, n=_log(rng, 100_000, 5_000_000), n2=_log(rng, 10_000, 200_000), tiles=rng.randint(4, 60),
                    z0=8, z1=rng.randint(10, 13), radius=_log(rng, 2_000, 60_000), radius2=_log(rng, 2_000, 60_000),
                    op=rng.choice(sorted(OPS)))
    if do == "serve":
        return dict(do=do, n=_log(rng, 300_000, 20_000_000), n2=_log(rng, 100_000, 5_000_000),
                    tiles=rng.randint(8, 96), z0=z0, z1=z1, r16=r16, mode=mode)
    if do == "styled":
        return dict(do=do, kind="polygons", n=_log(rng, 10_000, 300_000), tiles=_log(rng, 1, 100), z0=z0, z1=z1,
                    r16=rng.randint(4, 24), mode=rng.choice(["rgba", "coverage"]), index=index, host=False)
    kind = rng.choice(["points", "lines", "polygons"])
    n = {"points": _log(rng, 100_000, 60_000_000), "lines": _log(rng, 100_000, 30_000_000),
         "polygons": _log(rng, 10_000, 1_000_000)}[kind]
    if do == "register":
        # training takes a fixed time per index, and polygon layers have two: points and lines, no larger than listed
        index = "rtree" if kind == "polygons" else rng.choice(["rtree", "learned"])
        n = n // 8 if kind == "polygons" else min(n, 5_000_000) if index == "learned" else n
        return dict(do=do, kind=kind, n=n, tiles=rng.randint(1, 30), z0=z0, z1=z1, r16=r16, mode=mode, index=index)
    return dict(do=do, kind=kind, n=n, tiles=_log(rng, 1, 300 if kind == "polygons" else 1200), z0=z0, z1=z1, r16=r16,
                mode=mode, index=index, host=rng.random() < 0.25)


# ---- synthetic layers, made on the GPU -----------------------------------------

def _uniform(g, n, lo, hi):
    return torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float32).double()


def _mixture(g, n, k, sigma_lo, sigma_hi):
    """Positions around k random centres (float64, (n, 2))."""
    centre = _uniform(g, (k, 2), -0.8 * HALF, 0.8 * HALF)
    sigma = torch.exp(_uniform(g, k, math.log(sigma_lo), math.log(sigma_hi))) * GRID
    weight = -torch.log(_uniform(g, k, 1e-12, 1.0))
    bound = torch.cumsum(weight.cpu(), 0).cuda()
    bound = bound / bound[-1]
    which = torch.searchsorted(bound, _uniform(g, n, 0.0, 1.0)).clamp_(max=k - 1)
    return centre[which] + sigma[which, None] * _normal(g, n, 2)


def _to_grid(v):
    """Fold back into the grid at its border and quantise."""
    w = torch.remainder(v + HALF, 2.0 * GRID)
    w = torch.where(w >= GRID, 2.0 * GRID - w, w)
    return torch.clamp(torch.floor(w) - HALF, -HALF, HALF - 1).to(torch.int32).contiguous()


def make_points(g, n, uniform=False):
    noise = n if uniform else n // 20
    spread = _uniform(g, (noise, 2), -HALF, HALF)
    return _to_grid(spread if uniform else torch.cat([_mixture(g, n - noise, 64, 1e-4, 1e-2), spread]))


def make_lines(g, n_segments):
    """Random walks of 1..19 log-normal steps: (xy on the GPU, line offsets on the host, anchors)."""
    n = max(1, n_segments // 10)
    segs = torch.randint(1, 20, (n,), generator=g, device="cuda")
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cumsum(segs + 1, 0)
    # a row of 20 vertices per line, the first `segs + 1` of them kept (sums along
    # rows: the same from run to run)
    step = torch.exp(_normal(g, n, 20) + (math.log(1e-4 * GRID) - 0.5))
    step[:, 0] = 0.0
    turn = _uniform(g, (n, 20), -math.pi / 6, math.pi / 6)
    turn[:, 0] = _uniform(g, n, 0.0, 2 * math.pi)
    turn = torch.cumsum(turn, 1)
    start = _mixture(g, n, 1000, 1e-3, 1e-2)
    kept = torch.arange(20, device="cuda") <= segs[:, None]
    xy = torch.stack([(start[:, k:k + 1] + torch.cumsum(step * f(turn), 1))[kept]
                      for k, f in enumerate((torch.cos, torch.sin))], 1)
    xy = _to_grid(xy)
    return xy, off.cpu().numpy().astype(np.uint64), xy


def make_polygons(g, n):
    """Star polygons of 8..64 vertices: (xy on the GPU, ring offsets, polygon offsets, anchors)."""
    nv = torch.randint(8, 65, (n,), generator=g, device="cuda")
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cumsum(nv, 0)
    v = int(off[-1])
    poly = torch.repeat_interleave(torch.arange(n, device="cuda"), nv)
    rank = torch.arange(v, device="cuda") - off[:-1][poly]
    angle = 2 * math.pi * (rank + _uniform(g, v, 0.0, 1.0)) / nv[poly]
    rho = torch.exp(0.75 * _normal(g, n) + math.log(2e-4 * GRID))
    rad = rho[poly] * _uniform(g, v, 0.5, 1.0)
    centre = _mixture(g, n, 256, 1e-4, 1e-2)
    xy = centre[poly] + torch.stack([rad * torch.cos(angle), rad * torch.sin(angle)], 1)
    return (_to_grid(xy), off.cpu().numpy().astype(np.uint64), np.arange(n + 1, dtype=np.uint64), _to_grid(centre))


def density_tiles(g, anchors, case, r16):
    """(n, 4) [z, x, y, r16]: the tiles of random anchors at random zooms."""
    if case["tiles"] == 0:   # every tile of the zooms
        rows = [[z, x, y, r16] for z in range(case["z0"], case["z1"] + 1) for y in range(1 << z) for x in range(1 << z)]
        return np.array(rows, dtype=np.int64)
    n = case["tiles"]
    a = anchors[torch.randint(0, anchors.shape[0], (n,), generator=g, device="cuda")].long()
    z = torch.randint(case["z0"], case["z1"] + 1, (n,), generator=g, device="cuda")
    t = (a + HALF) >> (31 - z)[:, None]
    return torch.cat([z[:, None], t, torch.full_like(z[:, None], r16)], 1).cpu().numpy()


# ---- what a user's program holds --------------------------------------------------

class Held:
    """A context with its layers (and server), freed with the last reference."""

    def __init__(self):
        self.ctx = hv.hv_create(0)
        self.layers, self.server = [], None

    def load(self, kind, data):
        if kind in ("points", "uniform"):
            layer = hv.hv_layer_load_points(self.ctx, data[0], data[0].shape[0])
        elif kind == "lines":
            layer = hv.hv_layer_load_linestrings(self.ctx, data[0], data[1])
        else:
            layer = hv.hv_layer_load_polygons(self.ctx, data[0], data[1], data[2])
        self.layers.append(layer)
        return layer

    def drop(self, layer):
        self.layers.remove(layer)
        hv.hv_layer_free(layer)

    def __del__(self):
        if self.server is not None:
            hv.hv_server_stop(self.server)
        for layer in self.layers:
            hv.hv_layer_free(layer)
        hv.hv_destroy(self.ctx)


def _data(g, kind, n):
    """The layer's arrays, the anchors of density-weighted tiles last."""
    if kind in ("points", "uniform"):
        xy = make_points(g, n, kind == "uniform")
        return xy, xy
    return make_lines(g, n) if kind == "lines" else make_polygons(g, n)


def _pattern(g):
    """12 x 10 texels: diagonal stripes, a third of them transparent."""
    y, x = np.mgrid[0:10, 0:12]
    texel = np.zeros((10, 12, 4), dtype=np.uint8)
    texel[..., :3] = torch.randint(0, 256, (10, 12, 3), generator=g, device="cuda").cpu().numpy()
    texel[..., 3] = np.where((x + y) % 3 == 0, 0, 255)
    return texel


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    do = case["do"]
    held = Held()
    s = dict(case=case, held=held, style=hv.make_style(LINE, FILL))
    kinds = {"overlay": ["lines", "polygons"], "serve": ["points", "lines"]}.get(do) or [case["kind"]]
    anchors = []
    for kind, n in zip(kinds, (case["n"], case.get("n2"))):
        data = _data(g, kind, n)
        anchors.append(data[-1])
        torch.cuda.synchronize()   # the layer calls read the arrays on the default stream's order
        if do == "register":
            s["data"] = data
        else:
            layer = held.load(kind, data)
            hv.hv_layer_build_index(layer, hv.HV_INDEX_RTREE | (
                hv.HV_INDEX_LEARNED if case.get("index") == "learned" else 0))
        del data
    s["index"] = hv.HV_INDEX_LEARNED if case.get("index") == "learned" else hv.HV_INDEX_RTREE
    s["mode"] = MODES[case.get("mode", "mask")]
    rows = density_tiles(g, anchors[0], case, case.get("r16", 16))
    tile = hv.hv_tile_bytes(s["mode"])
    if do == "serve":
        # half of the requests for the line layer, arriving interleaved
        rows[1::2] = density_tiles(g, anchors[1], case, case["r16"])[1::2]
        reqs = hv.make_requests(rows, mode=s["mode"])
        reqs["layer"][1::2] = 1
        s["reqs"] = [reqs[i:i + 1].copy() for i in range(len(reqs))]
        s["out"] = np.zeros((len(reqs), tile), dtype=np.uint8)
        s["done"] = (hv.hv_done * len(reqs))()
        held.server = hv.hv_server_start(held.ctx, held.layers, hv.make_server_opts(
            max_batch=16, queue_capacity=1024, scratch_bytes=256 << 20, style=s["style"]))
        return s
    reqs = hv.make_requests(rows)
    s["n"] = len(reqs)
    if case.get("host"):
        s["reqs"] = reqs
        s["out"] = torch.zeros((len(reqs), tile), dtype=torch.uint8).pin_memory()
    else:
        s["reqs"] = torch.from_numpy(reqs.view(np.uint8)).cuda()
        s["out"] = torch.zeros((len(reqs), tile), dtype=torch.uint8, device="cuda")
    if do == "styled":
        s["fill"] = hv.make_fill_style(aa=True, pattern=_pattern(g))
    if do == "register":
        # room for the sorted keys: a record per point, at most four per segment or edge
        room = {"points": 1, "lines": 4 * 2, "polygons": 4 * 64}[case["kind"]] * case["n"]
        s["sorted"] = torch.zeros(room, dtype=torch.int64, device="cuda")
    if case.get("index") == "learned" and do == "register":
        # keys to look up: Hilbert keys are 62 bits
        s["keys"] = torch.randint(0, 1 << 62, (100_000,), generator=g, device="cuda")
        s["pos"] = torch.zeros(100_000, dtype=torch.int64, device="cuda")
    return s


# ---- one pass -----------------------------------------------------------------------

def run(s):
    return {"render": _render, "styled": _styled, "overlay": _overlay, "serve": _serve,
            "register": _register}[s["case"]["do"]](s)


def _render(s):
    hv.hv_render_tiles(s["held"].layers[0], s["reqs"], s["n"], s["mode"], s["index"], s["style"], s["out"],
                       s["out"].numel(), torch.cuda.current_stream())
    return s["out"]


def _styled(s):
    hv.hv_render_tiles_styled(s["held"].layers[0], s["reqs"], s["n"], s["mode"], s["index"], s["style"], s["fill"],
                              s["out"], s["out"].numel(), torch.cuda.current_stream())
    return s["out"]


def _overlay(s):
    a, b = s["held"].layers
    c = s["case"]
    hv.hv_overlay_tiles(a, c["radius"], b, c["radius2"], OPS[c["op"]], s["reqs"], s["n"], s["index"], s["out"],
                        s["out"].numel(), torch.cuda.current_stream())
    return s["out"]


def _serve(s):
    """Submit the burst, take every tile as it completes, in the order of completion."""
    srv, out, done = s["held"].server, s["out"], s["done"]
    base, tile, left, status = out.ctypes.data, out.shape[1], len(s["reqs"]), 0
    for tag, req in enumerate(s["reqs"]):
        while hv.hv_server_submit(srv, req, tag) != hv.HV_OK:
            pass
    while left:
        for d in done[:hv.hv_server_poll(srv, done)]:
            ctypes.memmove(base + d.tag * tile, d.data, d.bytes)
            status |= d.status
            left -= 1
    return out, status


def _register(s):
    """Load, index and render the first view; the sorted keys are the index's order."""
    held, c = s["held"], s["case"]
    layer = held.load(c["kind"], s["data"])
    learned = c["index"] == "learned"
    hv.hv_layer_build_index(layer, hv.HV_INDEX_RTREE | (hv.HV_INDEX_LEARNED if learned else 0))
    n = hv.hv_layer_info_get(layer).index_records
    hv.hv_layer_keys(layer, 0, s["sorted"], n)
    hv.hv_render_tiles(layer, s["reqs"], s["n"], s["mode"], s["index"], s["style"], s["out"], s["out"].numel(),
                       torch.cuda.current_stream())
    got = [s["sorted"], s["out"]]
    if learned:
        hv.hv_learned_lookup(layer, 0, s["keys"], s["keys"].numel(), s["pos"], torch.cuda.current_stream())
        got.append(s["pos"])
    held.drop(layer)
    return got


# ---- what a pass cannot do without ---------------------------------------------------

def work(case):
    """Bytes: requests in, tiles out; registering also reads the coordinates and
    writes the sorted records and keys.  Which objects a tile needs depends on
    the data, so the records a pass reads are not counted.  Operations: a
    multiply, an add and a compare per sample (four samples a pixel, one in a
    mask) and layer."""
    tiles = case["tiles"] or sum(4 ** z for z in range(case["z0"], case["z1"] + 1))
    mode = case.get("mode", "mask")
    layers = 2 if case["do"] == "overlay" else 1
    total = tiles * (16 + hv.hv_tile_bytes(MODES[mode]))
    flops = 3.0 * tiles * 65536 * (1 if mode == "mask" else 4) * layers
    if case["do"] == "register":
        n = case["n"] * (36 if case["kind"] == "polygons" else 1)
        total += n * (8 + (16 if case["kind"] == "points" else 48))
    return {"bytes": float(total), "flops": flops}


def exact(case, seed):
    """Every output is whole bytes or whole numbers, which stay the same; there is nothing to round."""
    return None
