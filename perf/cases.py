"""Measured cases: what a program that uses this library has it do.

Every case goes through the public entry points of ``lod.py``: building the
octree of one cloud in device memory (all five sampling modes, with and
without kept indices), the same from host memory with the octree read back,
many small clouds in one call, a burst of requests to the serving loop, and
drawing a frame of a finished octree.  Clouds follow the repository's three
recipes (an even sphere, an aerial survey, an indoor scan), drawn here on the
device from the seed, each vectorised so that hundreds of millions of points
take about a second.

All results are whole numbers (node records, voxel records, packed colours,
64-bit depth|colour keys), so there is nothing to state in 64-bit floating
point and the file defines no ``exact``.  The order of the points inside one
leaf is free by the library's contract and differs from run to run, so
builds return what does not depend on it: the node table and every voxel,
copied into buffers of the caller's own as a viewer does (their sizes follow
from the case, the rest stays zero); a build that keeps the input indices
returns, per input point, the leaf that holds it, and the cases that draw
return the frame (a pixel keeps the nearest of the samples, whatever their
order).  A weighted build's voxels come in a free order inside a node too: it
returns the node table and a frame.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2302_14801_gb300 import camera, lod, synth_gpu

_CHUNK = 1 << 24


def listed():
    return [
        # the smallest call: a small scan or one object, where launches, host
        # synchronisations and allocations are all there is
        {"name": "build_20k", "kind": "build", "cloud": "sphere", "n": 20_000, "leaf_threshold": 1000, "mode": "filter"},
        # one object scan at the default leaf size
        {"name": "build_1m", "kind": "build", "cloud": "sphere", "n": 1_000_000, "leaf_threshold": 50_000, "mode": "filter"},
        # a room-scale scan in host memory, built and read back whole (a file
        # converter's inner step), first-come sampling
        {"name": "host_10m_first", "kind": "host", "cloud": "indoor", "n": 10_000_000, "leaf_threshold": 50_000, "mode": "first"},
        # a survey tile with small leaves and kept indices: per-point
        # attributes are joined to the leaves afterwards
        {"name": "build_12m_pick_index", "kind": "build", "cloud": "aerial", "n": 12_000_001, "leaf_threshold": 3000, "mode": "pick",
         "keep_index": True},
        # the paper's own random key, with the picked points at full precision
        {"name": "build_20m_random_full", "kind": "build", "cloud": "indoor", "n": 20_000_000, "leaf_threshold": 50_000, "mode": "random",
         "full_precision": True},
        # an aerial survey block, averaged colours
        {"name": "build_50m", "kind": "build", "cloud": "aerial", "n": 50_000_000, "leaf_threshold": 50_000, "mode": "filter"},
        # a large building scan, sample picking, a ragged size
        {"name": "build_200m_pick", "kind": "build", "cloud": "indoor", "n": 200_000_003, "leaf_threshold": 50_000, "mode": "pick"},
        # the largest: half of the billion-point scan (three inputs, their
        # octrees and the scratch fit the card together)
        {"name": "build_500m", "kind": "build", "cloud": "indoor", "n": 500_000_000, "leaf_threshold": 50_000, "mode": "filter"},
        # independent scan tiles of very uneven size in one call
        {"name": "batched_48_tiles", "kind": "batched", "tiles": 48, "smallest": 10_000, "largest": 2_000_000,
         "leaf_threshold": 50_000, "mode": "filter"},
        # a burst of requests to the serving loop, mixed sizes and modes
        {"name": "serve_16_requests", "kind": "serve", "requests": 16, "inflight": 8, "smallest": 100_000, "largest": 8_000_000,
         "leaf_threshold": 50_000},
        # the neighbourhood-weighted average, and the first frame of it
        {"name": "weighted_20m_frame", "kind": "weighted", "cloud": "aerial", "n": 20_000_000, "leaf_threshold": 50_000,
         "view": "overview", "width": 1920, "height": 1080, "lod_pixels": 100.0},
        # one full-HD frame of a resident octree, as a viewer draws it
        {"name": "frame_50m", "kind": "frame", "cloud": "indoor", "n": 50_000_000, "leaf_threshold": 50_000, "mode": "filter",
         "view": "overview", "width": 1920, "height": 1080, "lod_pixels": 100.0},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["build"] * 6 + ["host", "batched", "serve", "weighted", "frame"])
    cloud = rng.choice(["sphere", "aerial", "indoor"])
    if kind == "batched":
        big = _log_uniform(rng, 50_000, 3_000_000)
        return {"kind": kind, "tiles": rng.randint(2, 60), "smallest": _log_uniform(rng, 1000, big // 4), "largest": big,
                "leaf_threshold": _log_uniform(rng, 1000, 100_000), "mode": rng.choice(["filter", "pick", "first", "random"])}
    if kind == "serve":
        big = _log_uniform(rng, 400_000, 16_000_000)
        return {"kind": kind, "requests": rng.randint(3, 24), "inflight": rng.choice([2, 4, 8]), "smallest": _log_uniform(rng, 100_000, big // 2),
                "largest": big, "leaf_threshold": _log_uniform(rng, 10_000, 100_000)}
    n = _log_uniform(rng, 10_000, {"build": 300_000_000, "host": 40_000_000, "weighted": 40_000_000, "frame": 100_000_000}[kind])
    # leaves from 1000 points, and at most about 20,000 leaves
    case = {"kind": kind, "cloud": cloud, "n": n, "leaf_threshold": _log_uniform(rng, max(1000, n // 20_000), 100_000)}
    if kind in ("weighted", "frame"):
        case.update(view=rng.choice(["overview", "close"]), width=rng.randint(320, 3840), height=rng.randint(240, 2160),
                    lod_pixels=float(_log_uniform(rng, 30, 400)))
    if kind != "weighted":
        case["mode"] = rng.choice(["filter", "filter", "pick", "first", "random"])
    if kind == "build":
        case["keep_index"] = rng.random() < 0.25
        case["full_precision"] = case["mode"] != "filter" and rng.random() < 0.25
    return case


# ------------------------------------------------------------------- clouds

def _pack(r, g, b):
    """RGBA8 in an int32 (R in the low byte, A = 255) from int32 channels."""
    return r.clamp(0, 255) + g.clamp(0, 255) * 256 + b.clamp(0, 255) * 65536 - (1 << 24)


def _noise(gen, m):
    return torch.randint(-16, 17, (m, 3), generator=gen, device="cuda", dtype=torch.int32)


def _gradient(gen, p, hi):
    c = torch.round(p * (255.0 / hi)).to(torch.int32) + _noise(gen, p.shape[0])
    return _pack(c[:, 0], c[:, 1], c[:, 2])


def _aerial(n, seed, buildings=2000):
    """synth.aerial on the device: 90 % terrain (6-octave value noise over a
    2^24 square, in random order), 10 % on the walls and roofs of boxes,
    building by building."""
    gen = torch.Generator(device="cuda").manual_seed(seed)

    def uni(*shape):
        return torch.rand(shape, generator=gen, device="cuda")

    dom, amp = float(1 << 24), float(1 << 18)
    norm = sum(0.5 ** o for o in range(6))
    layers = [(4 << o, amp * 0.5 ** o / norm, uni((4 << o) + 2, (4 << o) + 2)) for o in range(6)]

    def height(x, y):
        z = torch.zeros_like(x)
        for cells, a, tab in layers:
            u, v = x * (cells / dom), y * (cells / dom)
            iu, iv = u.floor(), v.floor()
            fu, fv = u - iu, v - iv
            fu, fv = fu * fu * (3 - 2 * fu), fv * fv * (3 - 2 * fv)
            at = iu.long() * (cells + 2) + iv.long()
            t = tab.reshape(-1)
            z += a * (t[at] * (1 - fu) * (1 - fv) + t[at + cells + 2] * fu * (1 - fv) + t[at + 1] * (1 - fu) * fv
                      + t[at + cells + 3] * fu * fv)
        return z

    def colour(z):
        t = (z / (amp + float(1 << 14))).clamp(0, 1)
        c = _noise(gen, z.shape[0])
        return _pack(torch.round(255 * t).int() + c[:, 0], torch.round(255 * (1 - (2 * t - 1).abs())).int() + c[:, 1],
                     torch.round(255 * (1 - t)).int() + c[:, 2])

    out = torch.empty((n, 4), dtype=torch.int32, device="cuda")
    n_t = n - n // 10

    def put(s, x, y, z):
        z = torch.round(z + 64.0 * torch.randn(z.shape, generator=gen, device="cuda"))
        e = s + x.shape[0]
        out[s:e, 0] = x.clamp(0, dom - 1).int()
        out[s:e, 1] = y.clamp(0, dom - 1).int()
        out[s:e, 2] = z.int()
        out[s:e, 3] = colour(z)

    for s in range(0, n_t, _CHUNK):
        m = min(_CHUNK, n_t - s)
        x, y = torch.floor(uni(m) * dom), torch.floor(uni(m) * dom)
        put(s, x, y, height(x, y))
    cx, cy = uni(buildings) * dom, uni(buildings) * dom
    wx, wy = torch.exp2(8 + 4 * uni(buildings)), torch.exp2(8 + 4 * uni(buildings))
    h = (1 << 10) + uni(buildings) * ((1 << 14) - (1 << 10))
    z0 = height(cx, cy)
    area = torch.stack([wx * wy, wy * h, wy * h, wx * h, wx * h], 1).double().cumsum(1)
    cum = area[:, -1].cumsum(0)
    cum = (cum / cum[-1] * (n - n_t)).contiguous()
    face_cum = (area / area[:, -1:]).float()
    for s in range(n_t, n, _CHUNK):
        m = min(_CHUNK, n - s)
        i = torch.arange(s - n_t, s - n_t + m, device="cuda", dtype=torch.float64)
        b = torch.searchsorted(cum, i, right=True).clamp_(max=buildings - 1)
        face = (uni(m)[:, None] >= face_cum[b]).sum(1)
        u, v = uni(m), uni(m)
        x0, y0 = cx[b] - wx[b] / 2, cy[b] - wy[b] / 2
        wall_x, wall_y = (face == 1) | (face == 2), face >= 3
        x = torch.where(wall_x, x0 + (face == 2) * wx[b], x0 + u * wx[b])
        y = torch.where(wall_y, y0 + (face == 4) * wy[b], y0 + torch.where(wall_x, u, v) * wy[b])
        put(s, x, y, torch.where(face == 0, z0[b] + h[b], z0[b] + v * h[b]))
    return out


def _indoor(n, seed, prims=4096):
    """synth.indoor on the device: planes of random orientation and box
    surfaces in a 2^22 cube, log-normal point shares, one after another as a
    scanner delivers them."""
    gen = torch.Generator(device="cuda").manual_seed(seed)

    def uni(*shape, **kw):
        return torch.rand(shape, generator=gen, device="cuda", **kw)

    def nrm(*shape, **kw):
        return torch.randn(shape, generator=gen, device="cuda", **kw)

    hi = float((1 << 22) - 1)
    cum = torch.exp(1.5 * nrm(prims, dtype=torch.float64)).cumsum(0)
    cum = (cum / cum[-1] * n).contiguous()
    size = torch.exp2(10 + 10 * uni(prims, 3))
    centre = uni(prims, 3) * hi
    t1 = nrm(prims, 3)
    t1 = t1 / t1.norm(dim=1, keepdim=True)
    t2 = nrm(prims, 3)
    t2 = t2 - (t2 * t1).sum(1, keepdim=True) * t1
    t2 = t2 / t2.norm(dim=1, keepdim=True)
    t3 = torch.linalg.cross(t1, t2)
    a = torch.stack([size[:, 1] * size[:, 2], size[:, 0] * size[:, 2], size[:, 0] * size[:, 1]], 1).repeat_interleave(2, 1).cumsum(1)
    a = a / a[:, -1:]
    out = torch.empty((n, 4), dtype=torch.int32, device="cuda")
    step = _CHUNK // 2
    for s in range(0, n, step):
        m = min(step, n - s)
        k = torch.searchsorted(cum, torch.arange(s, s + m, device="cuda", dtype=torch.float64), right=True).clamp_(max=prims - 1)
        sz = size[k]
        uvw, g = uni(m, 3) - 0.5, nrm(m, 1) * 32.0
        plane = uvw[:, :1] * sz[:, :1] * t1[k] + uvw[:, 1:2] * sz[:, 1:2] * t2[k] + g * t3[k]
        face = (uni(m)[:, None] >= a[k]).sum(1).clamp_(max=5)
        on = torch.arange(3, device="cuda")[None, :] == (face // 2)[:, None]
        box = torch.where(on, ((face % 2).float()[:, None] - 0.5) * sz + g, uvw * sz)
        p = torch.round(centre[k] + torch.where((k % 2 == 0)[:, None], plane, box)).clamp_(0, hi)
        out[s:s + m, :3] = p.int()
        out[s:s + m, 3] = _gradient(gen, p, hi)
    return out


def _cloud(name, n, seed):
    if name == "sphere":
        return synth_gpu.sphere(n, seed=seed)
    return _aerial(n, seed) if name == "aerial" else _indoor(n, seed)


# ------------------------------------------------------------------ workloads

class _Array:
    """A device array of the library, kept alive by its result."""

    def __init__(self, owner, ptr, shape):
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": shape, "typestr": "<i4", "data": (ptr, False), "version": 3, "strides": None}


def _on_device(owner, ptr, n, width):
    if not n:
        return torch.empty((0, width), dtype=torch.int32, device="cuda")
    return torch.as_tensor(_Array(owner, ptr, (n, width)), device="cuda")


def _buffer(n, width):
    return torch.zeros((n, width), dtype=torch.int32, device="cuda")


def _room(n, leaf_threshold):
    """Places for the nodes and voxels of a cloud of n points."""
    return 256 + 32 * (n // leaf_threshold + 1), 100_000 + int(2.0 * _voxels(n, leaf_threshold))


def _own(n, leaf_threshold):
    nodes, voxels = _room(n, leaf_threshold)
    return {"nodes": _buffer(nodes, 14), "voxels": _buffer(voxels, 4)}


def _take_nodes(r, own):
    v = r.view()
    nodes = _on_device(r, v.nodes, v.n_nodes, 14)
    own["nodes"][:v.n_nodes] = nodes
    return nodes


def _take(r, own):
    """Node table and voxels of one result, into the caller's buffers."""
    v = r.view()
    own["voxels"][:v.n_voxels] = _on_device(r, v.voxels, v.n_voxels, 4)
    return _take_nodes(r, own)


def _build_args(case):
    return {"leaf_threshold": case["leaf_threshold"], "mode": case["mode"]}


def _eye(case, pts, seed):
    """A view of the cloud: from outside over the whole of it, or close above
    one of its points; the seed moves the eye."""
    gen = torch.Generator().manual_seed(seed)
    t = torch.rand(4, generator=gen).tolist()
    lo, top = pts[:, :3].min(0).values.cpu().numpy().astype(np.float64), pts[:, :3].max(0).values.cpu().numpy().astype(np.float64)
    size = float((top - lo).max()) + 1.0
    if case["view"] == "overview":
        at = lo + (top - lo) / 2
        eye = at + size * np.array([1.5 + t[0], -0.5 - t[1], 0.8 + 0.4 * t[2]])
        fov = 50
    else:
        at = pts[int(t[3] * (pts.shape[0] - 1)), :3].cpu().numpy().astype(np.float64)
        eye = at + size * np.array([0.05 + 0.02 * t[0], 0.03 + 0.01 * t[1], 0.05 + 0.02 * t[2]])
        fov = 70
    return camera.perspective(eye, at, fovy_deg=fov, aspect=case["width"] / case["height"], near=1, far=1e9)


def _pinned(shape):
    return torch.zeros(shape, dtype=torch.int32, pin_memory=True)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batched":
        rng = np.random.default_rng(seed)
        # sizes over the whole range in a fixed spread, so that the work does
        # not depend on the seed; every tile has its own place and points
        sizes = np.rint(np.exp(np.linspace(math.log(case["smallest"]), math.log(case["largest"]), case["tiles"]))).astype(np.int64)
        rng.shuffle(sizes)
        offsets = rng.integers(0, (1 << 30) - (1 << 21), size=(case["tiles"], 3))
        tiles = [synth_gpu.sphere(int(m), seed=seed * 1000 + t, offset=tuple(int(o) for o in offsets[t])) for t, m in enumerate(sizes)]
        rooms = [_room(int(m), case["leaf_threshold"]) for m in sizes]
        return {"case": case, "tiles": tiles, "nodes": _buffer(sum(r[0] for r in rooms), 14), "voxels": _buffer(sum(r[1] for r in rooms), 4)}
    if kind == "serve":
        rng = np.random.default_rng(seed)
        sizes = np.rint(np.exp(np.linspace(math.log(case["smallest"]), math.log(case["largest"]), case["requests"]))).astype(np.int64)
        rng.shuffle(sizes)
        clouds = [_cloud("sphere", case["largest"], seed), _cloud("aerial", case["largest"], seed)]
        clouds = [c[torch.randperm(c.shape[0], device="cuda", generator=torch.Generator(device="cuda").manual_seed(seed))] for c in clouds]
        requests = [(clouds[i % 2][:int(m)], ("filter", "pick")[(i // 2) % 2]) for i, m in enumerate(sizes)]
        # room for the largest behind every request
        own = [_own(case["largest"], case["leaf_threshold"]) for _ in requests]
        return {"case": case, "requests": requests, "own": own, "server": lod.Server(120_000_000_000, case["inflight"])}
    pts = _cloud(case["cloud"], case["n"], seed)
    if kind == "build":
        own = _own(case["n"], case["leaf_threshold"])
        if case.get("full_precision"):
            own["voxel_points"] = torch.zeros_like(own["voxels"])
        return {"case": case, "points": pts, "own": own}
    if kind == "host":
        host = _pinned((case["n"], 4))
        host.copy_(pts)
        # page-locked places for the octree that comes back
        nodes, voxels = _room(case["n"], case["leaf_threshold"])
        out = {"nodes": _pinned((nodes, 14)).numpy().view(lod.NODE_DTYPE).reshape(-1), "points": _pinned((case["n"], 4)).numpy(),
               "voxels": _pinned((voxels, 4)).numpy().view(np.uint32)}
        if case["mode"] != "filter":
            out["index"] = _pinned((case["n"],)).numpy().view(np.uint32)
        return {"case": case, "points": host, "out": out}
    view_proj, origin = _eye(case, pts, seed)
    state = {"case": case, "view_proj": view_proj, "origin": origin}
    if kind == "weighted":
        state["points"] = pts
        state["own"] = {"nodes": _buffer(_room(case["n"], case["leaf_threshold"])[0], 14)}
    else:
        state["octree"] = lod.build(pts, **_build_args(case))
    return state


def _frame(state, octree):
    case = state["case"]
    return lod.render(octree, state["view_proj"], state["origin"], case["width"], case["height"], case["lod_pixels"])


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "frame":
        return _frame(state, state["octree"])
    if kind == "weighted":
        r = lod.build(state["points"], leaf_threshold=case["leaf_threshold"], mode="weighted")
        _take_nodes(r, state["own"])
        return {"nodes": state["own"]["nodes"], "frame": _frame(state, r)}
    if kind == "serve":
        server = state["server"]
        tickets = [server.submit(p, leaf_threshold=case["leaf_threshold"], mode=m) for p, m in state["requests"]]
        rs = [server.wait(t) for t in tickets]
        for r, own in zip(rs, state["own"]):
            _take(r, own)
        # the server's streams may reuse a result's memory once it is given back
        torch.cuda.current_stream().synchronize()
        return state["own"]
    if kind == "batched":
        rs = lod.build_batched(state["tiles"], **_build_args(case))
        views = [r.view() for r in rs]
        # one node table, and the one array of voxels that the nodes index
        total = sum(int(v.n_nodes) for v in views)
        torch.cat([_on_device(r, v.nodes, v.n_nodes, 14) for r, v in zip(rs, views)], out=state["nodes"][:total])
        total = sum(int(v.n_voxels) for v in views)
        state["voxels"][:total] = _on_device(rs, views[0].voxels, total, 4)
        return {"nodes": state["nodes"], "voxels": state["voxels"]}
    if kind == "host":
        r = lod.build_from_host(state["points"], **_build_args(case))
        r.to_host(out=state["out"])
        r.free()
        return {"nodes": state["out"]["nodes"].view(np.int32).reshape(-1, 14), "voxels": state["out"]["voxels"].view(np.int32)}
    own = state["own"]
    r = lod.build(state["points"], keep_index=case.get("keep_index", False), full_precision=case.get("full_precision", False),
                  **_build_args(case))
    nodes = _take(r, own)
    if case.get("full_precision"):
        ptr, n_voxels = ctypes.c_void_p(), r.view().n_voxels
        if n_voxels:
            lod.lib().lod_result_voxel_points(r.handle, ctypes.byref(ptr))
            own["voxel_points"][:n_voxels] = _on_device(r, ptr.value, n_voxels, 4)
    if not case.get("keep_index"):
        return own
    # which leaf (in point order) holds each input point: every node's range
    # starts where its first leaf's does
    n = case["n"]
    first = torch.zeros(n, dtype=torch.int32, device="cuda")
    first[nodes[:, 6:8].contiguous().view(torch.int64)[:, 0]] = 1
    leaf = torch.cumsum(first, 0, dtype=torch.int32)
    index = r.tensors()["index"]
    return own | {"leaf_of_point": torch.empty(n, dtype=torch.int32, device="cuda").scatter_(0, index.long(), leaf)}


# ----------------------------------------------------------------- what it takes

def _voxels(n, leaf_threshold):
    """About how many voxels a cloud of surfaces gives: a node of m points on
    a surface occupies about 20,000 (1 - exp(-m / 20,000)) cells of its 128^3
    grid, and every level up holds four times the points per node."""
    total, m = 0.0, 2.0 * leaf_threshold
    while m < 4.0 * n:
        k = min(m, n)
        total += n / k * 20000.0 * (1.0 - math.exp(-k / 20000.0))
        m *= 4.0
    return total if n > leaf_threshold else 0.0


def _build_bytes(n, case, mode):
    """Points read and written once, indices where the mode keeps them,
    voxels written once."""
    index = 4 if mode in ("pick", "first", "random") or case.get("keep_index") else 0
    voxel = 32 if case.get("full_precision") else 16
    return n * (32.0 + index) + _voxels(n, case["leaf_threshold"]) * voxel


def work(case):
    kind = case["kind"]
    if kind in ("batched", "serve"):
        count = case["tiles"] if kind == "batched" else case["requests"]
        sizes = np.exp(np.linspace(math.log(case["smallest"]), math.log(case["largest"]), count))
        modes = [case["mode"]] * count if kind == "batched" else [("filter", "pick")[(i // 2) % 2] for i in range(count)]
        b = sum(_build_bytes(float(m), case, mode) for m, mode in zip(sizes, modes))
    elif kind == "frame":
        # the samples a frame draws: a node whose projection is lod_pixels
        # wide holds about (128 / lod_pixels)^2 of them a pixel, on a few
        # layers of surface, as far as the octree has them
        pixels = case["width"] * case["height"]
        b = 8.0 * pixels + 16.0 * min(pixels * (128.0 / case["lod_pixels"]) ** 2 * 4.0, case["n"])
    else:
        b = _build_bytes(case["n"], case, case.get("mode", "weighted"))
        if kind == "weighted":
            b += 8.0 * case["width"] * case["height"]
    # integer work throughout; the frames' projections are counted as what
    # they are, 40 operations a sample
    return {"bytes": b, "flops": 0.0 if kind != "frame" else 40.0 * b / 16.0}
