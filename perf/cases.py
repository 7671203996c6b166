"""Frames, list builds and scans that a program using this library has it do.

Line sets are drawn on the GPU with the shapes of the repository's own
workloads (random walks, tractography-like bundles, ABC-flow pathlines, random
polylines), over the grid sides, image sizes, opacities, shading modes and
culling modes that its benchmark, server and tests use.

A case's ``kind`` says what a pass calls:
  frame    vrt.frame: vertex update + voxelization + (pyramid) + cull + trace
  calls    Renderer.frame: the same chain as separate calls, no update
  static   Renderer.trace_only: the lists of an earlier build, a new image
  serve    Server.submit for every set, then Server.poll until all are done
  scan     scan_counts_noalloc over a grid's packed words
"""
import math

import numpy as np
import torch

import paper_2510_09081_gb300 as vrt

LIGHT = (0.4, 0.5, 0.77)
UNITS = 16384.0            # the library snaps coordinates and radii to 2^-14 voxel
LIST_MARGIN = 32 / UNITS   # a voxel lists a segment within radius + this of its box
OCC_SCALE = 32.0           # occupancy codes per unit occupancy (the default)
R_MIN = 0.5


# ------------------------------------------------------------------ the cases
def _case(name, kind, lines, size, n, radius, width, height, alpha, ao=0, shading=0, cull=0,
          update=0.0, mips=0, ortho=0, graph=0):
    return {"name": name, "kind": kind, "lines": lines, "size": size, "n": n, "radius": radius,
            "width": width, "height": height, "alpha": alpha, "ao": ao, "shading": shading,
            "cull": cull, "update": update, "mips": mips, "ortho": ortho, "graph": graph}


def listed():
    return [
        # the smallest dynamic frame of the benchmark: 98k short segments, a
        # thumbnail-sized orthographic view, every launch counts
        _case("walks_ortho_256", "frame", "walks50", 2000, 64, 0.4, 256, 256, 1.0, update=0.05,
              ortho=1, graph=1),
        # odd image size, thick tubes, low opacity, irregular polylines: what the
        # tests and an inset view render, through the separate calls
        _case("polylines_157x93", "calls", "poly", 300, 32, 1.3, 157, 93, 0.1, cull=1),
        # one interactive view of a small set, automatic culling, 2% of it edited
        _case("walks_720p", "frame", "walks", 20_011, 128, 0.4, 1280, 720, 0.5, cull=2,
              update=0.02),
        # several resident sets viewed at once through the server
        _case("serve_8_sets", "serve", "walks", 200_000, 128, 0.4, 1280, 720, 0.6, cull=2,
              update=0.02),
        # flow lines around the viewer with ambient occlusion at every hit; all
        # vertices move
        _case("flow_ao_720p", "frame", "abc", 15_625, 128, 0.25, 1280, 720, 1.0, ao=6, cull=1,
              update=1.0),
        # opaque tractography in an ordinary window
        _case("bundles_opaque_1366", "frame", "bundles", 50_000, 256, 0.35, 1366, 768, 1.0,
              cull=1, update=0.05, graph=1),
        # the paper's shading: AO and shadows once per voxel, half-precision pyramid
        _case("bundles_voxel_shading", "frame", "bundles", 25_000, 256, 0.35, 1920, 1080, 0.3,
              ao=6, shading=1, cull=1, update=0.05, mips=1),
        # the benchmark's headline frame: 9.9M segments, transparent, 5% replaced
        _case("bundles_1080p", "frame", "bundles", 100_000, 256, 0.35, 1920, 1080, 0.3, cull=1,
              update=0.05, graph=1),
        # a camera moving around a set that does not change: trace only
        _case("bundles_static_1080p", "static", "bundles", 100_000, 256, 0.35, 1920, 1080, 0.3),
        # the server's heaviest request: long sparse walks in the largest grid at 4K
        _case("walks_4k", "frame", "walks", 4_960_000, 512, 0.4, 3840, 2160, 0.2, cull=2,
              update=0.02),
        # 31M segments, all moving, largest grid, ambient occlusion
        _case("flow_1080p", "frame", "abc", 1_000_000, 512, 0.25, 1920, 1080, 1.0, ao=6, cull=1,
              update=1.0, graph=1),
        # list offsets of a whole grid without allocation, as an arena's owner calls it
        _case("scan_256", "scan", "counts", 256 ** 3, 256, 0.0, 0, 0, 0.0),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["walks", "walks", "bundles", "bundles", "abc", "poly", "static", "serve",
                       "scan"])
    if what == "scan":
        return _unnamed(_case("", "scan", "counts", 4096 * _spread(rng, 1, 32768), 0, 0.0, 0, 0, 0.0))
    width, height = _spread(rng, 96, 1920), _spread(rng, 64, 1080)
    alpha = rng.choice([1.0, 1.0, 0.5, 0.3, round(rng.uniform(0.1, 0.9), 3)])
    cull = rng.choice([0, 1, 1, 2])
    graph = rng.choice([0, 1])
    if what == "serve":
        return _unnamed(_case("", "serve", "walks", _spread(rng, 20_000, 200_000), 128, 0.4,
                              min(width, 1280), min(height, 720), alpha, cull=cull, update=0.02))
    if what == "poly":
        return _unnamed(_case("", "calls", "poly", _spread(rng, 30, 3000), rng.choice([32, 64]),
                              rng.choice([0.05, 0.4, 1.3]), min(width, 640), min(height, 480), alpha,
                              cull=rng.choice([0, 1]), ortho=rng.choice([0, 1])))
    if what == "walks":
        size = _spread(rng, 10_000, 4_960_000)
        n = 128 if size < 200_000 else (256 if size < 1_500_000 else 512)
        if size >= 200_000 and rng.random() < 0.3:
            width, height = 3840, 2160
        return _unnamed(_case("", "frame", "walks", size, n, 0.4, width, height, alpha, cull=cull,
                              update=0.02, graph=graph))
    if what == "abc":
        n = rng.choice([128, 256, 512])
        size = int(1_000_000 * (n / 512) ** 3 * rng.uniform(0.2, 1.0))
        return _unnamed(_case("", "frame", "abc", size, n, 0.25, width, height, 1.0,
                              ao=rng.choice([0, 6]), cull=rng.choice([0, 1]), update=1.0,
                              mips=rng.choice([0, 1, 2]), graph=graph))
    n = rng.choice([128, 256, 256])
    size = _spread(rng, 1000, 12_000 if n == 128 else 100_000)
    shading = rng.choice([0, 0, 1])
    return _unnamed(_case("", "static" if what == "static" else "frame", "bundles", size, n, 0.35,
                          width, height, alpha, ao=6 if shading else 0, shading=shading,
                          cull=0 if what == "static" else cull,
                          update=0.0 if what == "static" else 0.05, mips=rng.choice([0, 1]),
                          graph=graph))


def _unnamed(case):
    del case["name"]
    return case


# ------------------------------------------------------------------ line sets
def _unit(v):
    return v / v.norm(dim=-1, keepdim=True).clamp_min(1e-30)


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 1_000_003 + 17)


def _uniform(g, shape, lo, hi):
    return lo + (hi - lo) * torch.rand(shape, generator=g, device="cuda", dtype=torch.float64)


def _normal(g, shape):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)


def _walks(g, lens, n, start_lo):
    """Random walks of half-voxel steps turning by about 10 degrees, reflected
    inside the grid; walk i keeps its first lens[i] vertices."""
    count, longest = len(lens), int(lens.max())
    p = _uniform(g, (count, 3), start_lo, n - start_lo)
    u = _unit(_normal(g, (count, 3)))
    out = torch.empty((count, longest, 3), device="cuda", dtype=torch.float32)
    out[:, 0] = p
    lo, hi = 1.0, n - 1.0
    for s in range(1, longest):
        w = _normal(g, (count, 3))
        w = _unit(w - (w * u).sum(-1, keepdim=True) * u)
        th = _normal(g, (count, 1)) * math.radians(10.0)
        u = _unit(u * th.cos() + torch.linalg.cross(w, u) * th.sin())
        p = p + 0.5 * u
        low, high = p < lo, p > hi
        p = torch.where(low, 2 * lo - p, torch.where(high, 2 * hi - p, p))
        u = torch.where(low | high, -u, u)
        out[:, s] = p
    keep = torch.arange(longest)[None, :] < torch.from_numpy(lens)[:, None]
    return out[keep.cuda()], np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)


def _polylines(rng, count, n):
    """Polylines of 2 to 30 vertices with steps of 0.2 to 3 voxels in any direction."""
    lens = rng.integers(2, 31, count)
    p = rng.uniform(1.0, n - 1.0, (count, 3))
    out = np.empty((count, 30, 3))
    for s in range(30):
        out[:, s] = p
        d = rng.normal(size=(count, 3))
        p = np.clip(p + d / np.linalg.norm(d, axis=1, keepdims=True) * rng.uniform(0.2, 3.0, (count, 1)),
                    1.0, n - 1.0)
    keep = np.arange(30)[None, :] < lens[:, None]
    xyz = torch.from_numpy(out[keep].astype(np.float32)).cuda()
    return xyz, np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)


def _bundles(rng, g, lines, n, verts=100, bundles=30):
    """Streamlines around 30 cubic centrelines inside an ellipsoid."""
    scale = n / 256.0
    centre, axes = np.full(3, 128.0) * scale, np.array([110.0, 90.0, 100.0]) * scale

    def inside():
        while True:
            q = rng.uniform(-1.0, 1.0, 3)
            if (q * q).sum() <= 1.0:
                return centre + 0.9 * q * axes
    ctrl, width = np.empty((bundles, 7, 3)), rng.uniform(2.0, 6.0, bundles) * scale
    for b in range(bundles):
        while True:
            s, e = inside(), inside()
            if np.linalg.norm(e - s) >= 80.0 * scale:
                break
        mid = [s + (e - s) * k / 4.0 + rng.normal(0.0, 20.0 * scale, 3) for k in (1, 2, 3)]
        mid = [m if (rr := np.linalg.norm((m - centre) / axes)) <= 0.9 else centre + (m - centre) * 0.9 / rr
               for m in mid]
        c = [s, *mid, e]
        ctrl[b] = [2 * c[0] - c[1], *c, 2 * c[-1] - c[-2]]
    which = torch.arange(lines, device="cuda") * bundles // lines
    ctrl = torch.from_numpy(ctrl).cuda()
    sig = torch.from_numpy(width / 2).cuda()[which][:, None, None]
    line = torch.linspace(0.0, 1.0, verts, device="cuda", dtype=torch.float64)
    t0, t1 = _uniform(g, (lines, 1), 0.0, 0.05), _uniform(g, (lines, 1), 0.95, 1.0)
    x = (t0 + (t1 - t0) * line) * 4
    k = x.long().clamp_max(3)
    f = (x - k)[..., None]
    p0, p1, p2, p3 = (ctrl[which[:, None], k + j] for j in range(4))
    pos = 0.5 * (2 * p1 + (p2 - p0) * f + (2 * p0 - 5 * p1 + 4 * p2 - p3) * f ** 2
                 + (3 * p1 - p0 - 3 * p2 + p3) * f ** 3)
    tan = _unit(0.5 * ((p2 - p0) + 2 * (2 * p0 - 5 * p1 + 4 * p2 - p3) * f
                       + 3 * (3 * p1 - p0 - 3 * p2 + p3) * f ** 2))
    ref = torch.zeros_like(tan).scatter_(2, tan.mean(1, keepdim=True).abs().argmin(2, keepdim=True)
                                         .expand(-1, verts, 1), 1.0)
    n1 = _unit(torch.linalg.cross(tan, ref))
    n2 = torch.linalg.cross(tan, n1)
    off = _normal(g, (lines, 1, 2)) * sig
    off = off + 0.15 * sig * torch.sin(2 * math.pi * _uniform(g, (lines, 1, 2), 1.0, 4.0) * line[:, None]
                                       + _uniform(g, (lines, 1, 2), 0.0, 2 * math.pi))
    p = (pos + off[..., :1] * n1 + off[..., 1:] * n2).clamp(1.0, n - 1.0)
    return p.float().reshape(-1, 3), np.arange(0, lines * verts + 1, verts, dtype=np.int64)


def _flow(g, particles, n, phase, verts=32):
    """Lines of about one voxel per segment through the ABC flow."""
    a, b, c = math.sqrt(3.0), math.sqrt(2.0), 1.0
    scale = 2 * math.pi / n
    dt = scale / 2.2

    def vel(q):
        s, k = torch.sin(q + phase), torch.cos(q + phase)
        return torch.stack([a * s[:, 2] + c * k[:, 1], b * s[:, 0] + a * k[:, 2],
                            c * s[:, 1] + b * k[:, 0]], -1)
    x = _uniform(g, (particles, 3), n / 8.0, 7.0 * n / 8.0) * scale
    out = torch.empty((particles, verts, 3), device="cuda", dtype=torch.float32)
    out[:, 0] = x / scale
    for s in range(1, verts):
        k1 = vel(x)
        k2 = vel(x + 0.5 * dt * k1)
        k3 = vel(x + 0.5 * dt * k2)
        k4 = vel(x + dt * k3)
        x = x + dt / 6.0 * (k1 + 2 * k2 + 2 * k3 + k4)
        out[:, s] = x / scale
    return (out.clamp_(0.5, n - 0.5).reshape(-1, 3),
            np.arange(0, particles * verts + 1, verts, dtype=np.int64))


def _line_set(case, seed, size=None):
    rng, g = np.random.default_rng([int(seed), 5]), _generator(seed)
    n, size = case["n"], case["size"] if size is None else size
    if case["lines"] == "poly":
        return _polylines(rng, size, n)
    if case["lines"] == "walks50":
        return _walks(g, np.full(size, 50, np.int64), n, 8.0)
    if case["lines"] == "walks":  # 20 to 200 vertices each, `size` segments in all
        lens = rng.integers(20, 201, size // 19 + 1)
        ends = np.cumsum(lens - 1)
        m = int(np.searchsorted(ends, size)) + 1
        lens = lens[:m].astype(np.int64)
        lens[-1] -= ends[m - 1] - size
        return _walks(g, lens, n, 2.0)
    if case["lines"] == "bundles":
        return _bundles(rng, g, size, n)
    return _flow(g, size, n, 0.1 * int(seed) % (2 * math.pi))


class _Camera:
    """A camera with the attributes the library reads."""

    def __init__(self, case, turn=0.0):
        n = float(case["n"])
        c = n / 2.0
        self.width, self.height, self.ortho = case["width"], case["height"], case["ortho"]
        self.target, self.up, self.fovy_deg, self.ortho_h = (c, c, c), (0.0, 0.0, 1.0), 45.0, n
        if case["ortho"]:
            self.eye, self.target, self.up = (c, c, -1.0), (c, c, n), (0.0, 1.0, 0.0)
        elif case["lines"] == "abc":  # inside the flow
            self.eye = (c, c, c)
            self.target = (c + 10 * math.cos(turn), c + 10 * math.sin(turn), c + 2.0)
        elif case["lines"] == "bundles":
            r, el = 300.0 * n / 256.0, math.radians(20.0)
            self.eye = (c + r * math.cos(el) * math.cos(turn), c + r * math.cos(el) * math.sin(turn),
                        c + r * math.sin(el))
        else:
            self.eye = (c + 1.7 * n * math.cos(turn), c + 1.7 * n * math.sin(turn), c + 0.5 * n)


def _turn(seed, k=0):
    return float(np.random.default_rng([int(seed), 9, k]).uniform(0, 2 * math.pi))


def _update(case, seed, xyz):
    """The block of vertices a frame replaces: (first vertex, coordinates)."""
    total = xyz.shape[0]
    count = max(1, int(round(total * case["update"])))
    first = int(np.random.default_rng([int(seed), 3]).integers(0, total - count + 1))
    g = _generator(seed + 7)
    moved = xyz[first:first + count].double() + 0.05 * _normal(g, (count, 3))
    return first, moved.clamp(1.0, case["n"] - 1.0).float().contiguous()


def _server_sets(case, seed):
    """Eight sets, log-uniformly sized up to case["size"] segments, with their views."""
    rng = np.random.default_rng([int(seed), 11])
    sizes = np.exp(rng.uniform(math.log(case["size"] / 20), math.log(case["size"]), 8)).astype(int)
    alphas = np.clip(case["alpha"] * rng.uniform(0.5, 1.6, 8), 0.1, 1.0)
    for k in range(8):
        xyz, off = _line_set(case, 101 * int(seed) + k, max(100, int(sizes[k])))
        first, moved = _update(case, 101 * int(seed) + k, xyz)
        yield xyz, off, first, moved, _Camera(case, _turn(seed, k)), float(alphas[k])


# ------------------------------------------------------------ prepare and run
def _scan_inputs(case, seed):
    """Packed words and marks of a grid's voxels: most are empty, a few very full."""
    g, m = _generator(seed), case["size"]
    counts = torch.rand(m, generator=g, device="cuda").pow(6.0).mul(60.0).int()
    occ = torch.randint(0, 2048, (m,), generator=g, device="cuda", dtype=torch.int32)
    marks = torch.randint(-2 ** 31, 2 ** 31, (m // 32,), generator=g, device="cuda",
                          dtype=torch.int64).int()
    return torch.where(counts > 0, occ * 65536 + counts, 0).int(), marks


def prepare(case, seed):
    if case["kind"] == "scan":
        words, marks = _scan_inputs(case, seed)
        return {"kind": "scan", "words": words, "marks": marks, "offsets": torch.empty_like(words),
                "total": torch.zeros(1, dtype=torch.int32, device="cuda"),
                "status": torch.zeros(1, dtype=torch.int32, device="cuda")}
    if case["kind"] == "serve":
        server, requests = vrt.Server(hbm_budget=16 << 30, max_inflight=4), []
        for xyz, off, first, moved, cam, alpha in _server_sets(case, seed):
            sid = server.add_set(xyz.cpu().numpy(), off, case["n"], case["radius"])
            bufs = _images(cam)
            requests.append((sid, cam, bufs, alpha, first, moved.cpu().numpy()))
        torch.cuda.synchronize()  # the server works on streams of its own
        return {"kind": "serve", "server": server, "requests": requests, "cull": case["cull"]}
    xyz, off = _line_set(case, seed)
    cam = _Camera(case, _turn(seed))
    r = vrt.Renderer(case["n"], case["radius"])
    r.upload(xyz, off)
    vrt.set_option(r.h, vrt.OPT_MIPS_FORMAT, case["mips"])
    vrt.set_option(r.h, vrt.OPT_GRAPH, case["graph"])
    params = vrt.params_c(case["alpha"], case["ao"], case["cull"], 0, case["shading"], LIGHT)
    state = {"kind": case["kind"], "renderer": r, "cam": cam, "cam_c": vrt.camera_c(cam),
             "params": params, "case": dict(case), "images": _images(cam)}
    if case["update"]:
        state["first"], state["moved"] = _update(case, seed, xyz)
    if case["kind"] == "static":
        # the set's one build; each pass then draws it from the turned camera
        r.frame(_Camera(case, 0.0), case["alpha"], case["ao"], 0, 0, True, case["shading"], LIGHT)
    if case["cull"] == 2:
        # automatic culling goes by the visible share of the frames seen so far
        vrt.frame(r.h, state["cam_c"], params, *state["images"])
        vrt.sync(r.h)
    return state


def _images(cam):
    h, w = cam.height, cam.width
    return (torch.empty((h, w, 4), device="cuda"), torch.empty((h, w), dtype=torch.int32, device="cuda"),
            torch.empty((h, w), device="cuda"))


def run(state):
    if state["kind"] == "scan":
        vrt.scan_counts_noalloc(state["words"], state["offsets"], state["marks"], state["total"],
                                state["status"])
        return [state["offsets"], state["total"], state["status"]]
    if state["kind"] == "serve":
        for sid, cam, (rgba, fid, ft), alpha, first, moved in state["requests"]:
            state["server"].submit(sid, cam, rgba, alpha, 0, state["cull"], fid, ft, first, moved)
        done = state["server"].poll(wait=True)
        if any(d["status"] for d in done):
            raise RuntimeError("a served frame failed")
        return [list(q[2]) for q in state["requests"]]
    case = state["case"]
    if state["kind"] == "static":
        return list(state["renderer"].trace_only(state["cam"], case["alpha"], case["ao"], 0,
                                                 case["shading"], LIGHT))
    if state["kind"] == "calls":
        return list(state["renderer"].frame(state["cam"], case["alpha"], case["ao"], case["cull"], 0,
                                            True, case["shading"], LIGHT))
    vrt.frame(state["renderer"].h, state["cam_c"], state["params"], *state["images"],
              first_vertex=state["first"], update=state["moved"])
    return list(state["images"])


def work(case):
    """Bytes: each vertex of the set (12) and of the update (12) and the output
    image (colour, id and depth: 24 per pixel) once. Operations: one
    capsule-box decision per segment (about 40) and one ray-capsule test per
    pixel (82)."""
    if case["kind"] == "scan":
        return {"bytes": case["size"] * 8.125, "flops": case["size"]}
    px = case["width"] * case["height"]
    verts = case["size"] * {"poly": 16, "walks50": 50, "walks": 1.01, "bundles": 100, "abc": 32}[case["lines"]]
    frames = 1
    if case["kind"] == "serve":  # eight log-uniform sets: mean size 0.32 of the largest
        frames, verts = 8, verts * 0.32
    if case["kind"] == "static":
        return {"bytes": 24 * px + 12 * verts, "flops": 82 * px}
    return {"bytes": frames * (12 * verts * (1 + case["update"]) + 24 * px),
            "flops": frames * (40 * verts + 82 * px)}


# ----------------------------------------------------------------- 64-bit images
MOST_PAIRS = 1_500_000_000  # (pixel, segment) pairs an image may take
MOST_HITS = 150_000_000


def exact(case, seed):
    if case["kind"] == "scan":
        return None  # whole numbers
    if case["kind"] == "serve":
        out = []
        for xyz, off, first, moved, cam, alpha in _server_sets(case, seed):
            xyz[first:first + moved.shape[0]] = moved
            out.append(_exact_frame(case, xyz, off, cam, alpha))
        return None if any(v is None for v in out) else out
    # voxel-space shading marches every voxel to the light; the largest sets
    # give too many hits
    if case["shading"] or case["size"] * (case["lines"] in ("abc", "bundles")) > 60_000:
        return None
    if case["lines"] == "walks" and case["size"] > 1_000_000:
        return None
    xyz, off = _line_set(case, seed)
    if case["update"]:
        first, moved = _update(case, seed, xyz)
        xyz[first:first + moved.shape[0]] = moved
    return _exact_frame(case, xyz, off, _Camera(case, _turn(seed)), case["alpha"])


def _f32(v):
    return torch.tensor(np.asarray(v, np.float32).astype(np.float64), device="cuda")


def _dot(a, b):
    return (a * b).sum(-1)


class _Scene:
    """Snapped segments with their clip planes, in 64 bits."""

    def __init__(self, xyz, off, radius):
        p = torch.round(xyz.double() * UNITS) / UNITS  # half to even, as the library
        total = p.shape[0]
        off = torch.from_numpy(off).cuda()
        first = torch.zeros(total, dtype=torch.bool, device="cuda")
        last = torch.zeros_like(first)
        first[off[:-1]] = True
        last[off[1:] - 1] = True
        tan = torch.zeros_like(p)
        tan[1:-1] = p[2:] - p[:-2]
        tan[first | last] = 0.0
        ids = torch.nonzero(~last).squeeze(1)
        self.ids, self.a, self.b = ids, p[ids], p[ids + 1]
        self.na, self.nb = _unit(tan[ids]) * (tan[ids].abs().amax(-1, keepdim=True) > 0), \
            _unit(tan[ids + 1]) * (tan[ids + 1].abs().amax(-1, keepdim=True) > 0)
        self.ca, self.cb = _dot(tan[ids], tan[ids]) > 0, _dot(tan[ids + 1], tan[ids + 1]) > 0
        self.r = round(float(np.float32(radius)) * UNITS) / UNITS


class _View:
    """Rays of a camera, and which pixels may see a ball."""

    def __init__(self, cam):
        self.w, self.h, self.ortho = cam.width, cam.height, cam.ortho
        eye, tgt, up = _f32(cam.eye), _f32(cam.target), _f32(cam.up)
        self.eye = eye
        self.f = _unit(tgt - eye)
        self.right = _unit(torch.linalg.cross(self.f, up))
        self.up = torch.linalg.cross(self.right, self.f)
        if cam.ortho:
            self.sy = float(np.float32(cam.ortho_h)) / 2
        else:
            self.sy = math.tan(math.radians(float(np.float32(cam.fovy_deg))) / 2)
        self.sx = self.sy * self.w / self.h

    def rays(self, pix):
        u = (2 * (pix % self.w + 0.5) / self.w - 1) * self.sx
        v = (1 - 2 * (torch.div(pix, self.w, rounding_mode="floor") + 0.5) / self.h) * self.sy
        side = u[:, None] * self.right + v[:, None] * self.up
        if self.ortho:
            return self.eye + side, self.f.expand(pix.shape[0], 3)
        return self.eye.expand(pix.shape[0], 3), _unit(self.f + side)

    def boxes(self, centre, rad):
        """Pixel rectangles [x0, x1) x [y0, y1) that hold every ray meeting the balls."""
        v = centre - self.eye
        x, y, z = _dot(v, self.right), _dot(v, self.up), _dot(v, self.f)
        if self.ortho:
            lo = [(x - rad) / self.sx, (y - rad) / self.sy]
            hi = [(x + rad) / self.sx, (y + rad) / self.sy]
            out = torch.zeros_like(z, dtype=torch.bool)
        else:
            d = v.norm(dim=-1)
            wide = math.atan(math.hypot(self.sx, self.sy)) + 1e-6
            out = (d > rad) & (torch.acos((z / d).clamp(-1, 1)) - torch.asin((rad / d).clamp(max=1)) > wide)
            near, far = z - rad, z + rad
            whole = near <= 1e-3
            lo, hi = [], []
            for q, s in ((x, self.sx), (y, self.sy)):
                a, b = (q - rad) / s, (q + rad) / s
                lo.append(torch.where(whole, -2.0, a / torch.where(a < 0, near, far)))
                hi.append(torch.where(whole, 2.0, b / torch.where(b < 0, far, near)))
        px0 = torch.floor((lo[0] + 1) / 2 * self.w - 0.5 - 1e-3).clamp(0, self.w)
        px1 = torch.ceil((hi[0] + 1) / 2 * self.w - 0.5 + 1e-3).add(1).clamp(0, self.w)
        py0 = torch.floor((1 - hi[1]) / 2 * self.h - 0.5 - 1e-3).clamp(0, self.h)
        py1 = torch.ceil((1 - lo[1]) / 2 * self.h - 0.5 + 1e-3).add(1).clamp(0, self.h)
        wd = torch.where(out, 0.0, (px1 - px0).clamp_min(0)).long()
        ht = torch.where(out, 0.0, (py1 - py0).clamp_min(0)).long()
        return px0.long(), py0.long(), wd, ht


def _ball(oc, d, r2):
    b = _dot(oc, d)
    disc = r2 - _dot(oc - b[:, None] * d, oc - b[:, None] * d)
    return torch.where(disc >= 0, -b - disc.clamp_min(0).sqrt(), math.inf)


def _entry(o, d, a, b, r):
    """First entry of each line o + t d into the capsule (a, b, r); inf when it misses."""
    oa, ba, r2 = o - a, b - a, r * r
    l2 = _dot(ba, ba)
    inv = 1.0 / torch.where(l2 > 0, l2, 1.0)
    dp = d - (_dot(d, ba) * inv)[:, None] * ba
    op = oa - (_dot(oa, ba) * inv)[:, None] * ba
    q = _dot(dp, dp)
    qs = torch.where(q > 1e-24, q, 1.0)
    ts = -_dot(op, dp) / qs
    w = op + ts[:, None] * dp
    disc = r2 - _dot(w, w)
    t = ts - (disc.clamp_min(0) / qs).sqrt()
    y = _dot(oa + t[:, None] * d, ba)
    ea, eb = _ball(oa, d, r2), _ball(o - b, d, r2)
    t = torch.where(y < 0, ea, torch.where(y > l2, eb, t))
    t = torch.where(disc < 0, math.inf, t)
    t = torch.where(q > 1e-24, t, torch.minimum(ea, eb))
    return torch.where(l2 > 0, t, ea)


def _hits(scene, view, n):
    """(pixel, depth, segment row) of every accepted hit, in chunks."""
    mid, half = (scene.a + scene.b) / 2, (scene.b - scene.a).norm(dim=-1) / 2
    x0, y0, wd, ht = view.boxes(mid, half + scene.r + 1e-6)
    count = wd * ht
    ends = torch.cumsum(count, 0)
    total = int(ends[-1])
    if total > MOST_PAIRS:
        return None

    def chunks():
        step = 8_000_000
        for lo in range(0, total, step):
            k = torch.arange(lo, min(total, lo + step), device="cuda")
            s = torch.searchsorted(ends, k, right=True)
            q = k - (ends[s] - count[s])
            pix = (y0[s] + torch.div(q, wd[s], rounding_mode="floor")) * view.w + x0[s] + q % wd[s]
            o, d = view.rays(pix)
            a, b = scene.a[s], scene.b[s]
            t = _entry(o, d, a, b, scene.r)
            ok = torch.isfinite(t) & (t >= 0)
            p = o + torch.where(ok, t, 0.0)[:, None] * d
            ok &= ((p >= 0) & (p <= n)).all(-1)
            ok &= ~scene.ca[s] | (_dot(p - a, scene.na[s]) >= 0)
            ok &= ~scene.cb[s] | (_dot(p - b, scene.nb[s]) <= 0)
            yield pix[ok], t[ok], s[ok]
    return chunks()


def _exact_frame(case, xyz, off, cam, alpha):
    n, alpha = case["n"], float(np.float32(alpha))
    scene, view = _Scene(xyz, off, case["radius"]), _View(cam)
    chunks = _hits(scene, view, n)
    if chunks is None:
        return None
    npx = view.w * view.h
    if alpha >= 1.0:
        depth = torch.full((npx,), math.inf, device="cuda", dtype=torch.float64)
        seg = torch.full((npx,), -1, device="cuda", dtype=torch.long)
        for pix, t, s in chunks:
            before = depth.clone()
            depth.scatter_reduce_(0, pix, t, "amin")
            win = t == depth[pix]
            seg = torch.where(depth < before, 2 ** 40, seg)
            seg.scatter_reduce_(0, pix[win], s[win], "amin")
        pix = torch.nonzero(seg >= 0).squeeze(1)
        t, s = depth[pix], seg[pix]
    else:
        got, hits = [], 0
        for c in chunks:
            got.append(c)
            hits += c[0].shape[0]
            if hits > MOST_HITS:
                return None
        pix, t, s = (torch.cat(v) for v in zip(*got))
        order = torch.argsort(s, stable=True)
        order = order[torch.argsort(t[order], stable=True)]
        order = order[torch.argsort(pix[order], stable=True)]
        pix, t, s = pix[order], t[order], s[order]
    d = scene.b[s] - scene.a[s]
    colour = torch.where(_dot(d, d)[:, None] > 0, _unit(d).abs(), 1.0)
    if case["ao"] and pix.shape[0]:
        o, dv = view.rays(pix)
        colour = colour * _ambient(_pyramid(scene, n), o + t[:, None] * dv)[:, None]
    new = torch.ones_like(pix, dtype=torch.bool)
    new[1:] = pix[1:] != pix[:-1]
    start = torch.nonzero(new).squeeze(1)
    rank = torch.arange(pix.shape[0], device="cuda") - start[torch.cumsum(new, 0) - 1]
    # composited front to back until the transmittance falls below 1e-4
    w = alpha * (1.0 - alpha) ** rank.double()
    w = torch.where((rank == 0) | (w / alpha >= 1e-4), w, 0.0)
    rgba = torch.zeros((npx, 4), device="cuda", dtype=torch.float64)
    rgba[:, :3].index_add_(0, pix, w[:, None] * colour)
    rgba[:, 3].index_add_(0, pix, w)
    depth = torch.full((npx,), math.inf, device="cuda", dtype=torch.float64)
    depth[pix[start]] = t[start]
    return [rgba.reshape(view.h, view.w, 4), None, depth.reshape(view.h, view.w)]


def _box_distance(a, d):
    """Distance of the segments a + t d, 0 <= t <= 1, to the unit box: the squared
    distance is convex and quadratic between the t where a coordinate meets a face."""
    safe = torch.where(d != 0, d, 1.0)
    t = torch.cat([torch.where(d != 0, -a / safe, 0.0), torch.where(d != 0, (1 - a) / safe, 0.0),
                   torch.zeros_like(a[:, :1]), torch.ones_like(a[:, :1])], 1).clamp(0, 1).sort(1).values

    def square(t):
        p = a[:, None] + t[..., None] * d[:, None]
        return ((-p).clamp_min(0) + (p - 1).clamp_min(0)).square().sum(-1)
    lo, hi = t[:, :-1], t[:, 1:]
    p = a[:, None] + ((lo + hi) / 2)[..., None] * d[:, None]
    act = ((p < 0) | (p > 1)).double()
    e0 = act * (a[:, None] - (p > 1).double())
    dd = act * d[:, None]
    q = _dot(dd, dd)
    best = torch.where(q > 0, -_dot(e0, dd) / torch.where(q > 0, q, 1.0), lo)
    best = torch.minimum(torch.maximum(best, lo), hi)
    return torch.minimum(square(best).amin(1), square(t).amin(1)).sqrt()


def _pyramid(scene, n):
    """Averaging pyramid of the occupancy codes of every listed (segment, voxel) pair."""
    rl = scene.r + LIST_MARGIN
    rc = max(scene.r, R_MIN)
    lo = torch.floor(torch.minimum(scene.a, scene.b) - rl).clamp(0, n - 1).long()
    hi = torch.floor(torch.maximum(scene.a, scene.b) + rl).clamp(0, n - 1).long()
    ext = hi - lo + 1
    count = ext.prod(-1)
    ends = torch.cumsum(count, 0)
    level = torch.zeros(n ** 3, device="cuda", dtype=torch.float64)
    for k0 in range(0, int(ends[-1]), 4_000_000):
        k = torch.arange(k0, min(int(ends[-1]), k0 + 4_000_000), device="cuda")
        s = torch.searchsorted(ends, k, right=True)
        q = k - (ends[s] - count[s])
        x = lo[s, 0] + q % ext[s, 0]
        q = torch.div(q, ext[s, 0], rounding_mode="floor")
        y, z = lo[s, 1] + q % ext[s, 1], lo[s, 2] + torch.div(q, ext[s, 1], rounding_mode="floor")
        v = torch.stack([x, y, z], -1).double()
        a, b = scene.a[s] - v, scene.b[s] - v
        d = b - a
        near = _box_distance(a, d) <= rl
        pa, pb, dd = 0.5 - a, 0.5 - b, _dot(d, d)
        h = torch.where(dd > 0, _dot(pa, d) / torch.where(dd > 0, dd, 1.0), 0.0).clamp(0, 1)
        sd = (pa - h[:, None] * d).norm(dim=-1) - rc
        sd = torch.where(scene.ca[s], torch.maximum(sd, -_dot(pa, scene.na[s])), sd)
        sd = torch.where(scene.cb[s], torch.maximum(sd, _dot(pb, scene.nb[s])), sd)
        code = torch.floor(OCC_SCALE * (0.5 - sd).clamp(0, 1) * (scene.r / rc) ** 2 + 0.5)
        level.index_add_(0, (z * n + y) * n + x, torch.where(near, code, 0.0))
    levels = [(level / OCC_SCALE).clamp_max(1.0).reshape(n, n, n)]
    while levels[-1].shape[0] > 1:
        m = levels[-1].shape[0] // 2
        levels.append(levels[-1].reshape(m, 2, m, 2, m, 2).mean((1, 3, 5)))
    return levels


def _trilinear(level, p, scale):
    m = level.shape[0]
    u = p * scale - 0.5
    base = torch.floor(u)
    f, base, acc = u - base, base.long(), 0.0
    for k in range(8):
        bit = torch.tensor([k & 1, k >> 1 & 1, k >> 2], device="cuda")
        q = base + bit
        w = torch.where(bit.bool(), f, 1.0 - f).prod(-1)
        ok = ((q >= 0) & (q < m)).all(-1)
        q = q.clamp(0, m - 1)
        acc = acc + torch.where(ok, w * level[q[:, 2], q[:, 1], q[:, 0]], 0.0)
    return acc


def _ambient(levels, p):
    """Six cones along the axes, cos(half angle) = 2/3, samples half a diameter apart."""
    tan = math.sqrt(5.0) / 2
    total = 0.0
    for c in range(6):
        clear, t = 1.0, 1.0
        while t <= 16.0:
            dia = max(1.0, 2 * t * tan)
            lam = min(math.log2(dia), len(levels) - 1)
            l0 = int(lam)
            q = p.clone()
            q[:, c >> 1] += -t if c & 1 else t
            s = _trilinear(levels[l0], q, 0.5 ** l0)
            if lam > l0:
                s = (1 - (lam - l0)) * s + (lam - l0) * _trilinear(levels[l0 + 1], q, 0.5 ** (l0 + 1))
            clear = clear * (1 - s)
            t += 0.5 * dia
        total = total + clear
    return total / 6.0
