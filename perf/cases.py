"""The work that users have this library do, as cases to be timed and compared.

Each case is one pass through the package's public calls, on inputs drawn
from a seed on the GPU (the recipes are those of the package's synthetic
workloads: uniform, clustered and mixed frames, a camera lattice round one
scene, anisotropic 3D Gaussians):

* ``frame``       one frame of projected Gaussians, ``Context.sort_frame``:
                  a viewer or trainer sorting its frame, from thumbnail to 4K;
* ``views``       several cameras of one scene in one ``sort_views`` batch;
* ``graph``       a served batch of requests of mixed sizes and resolutions,
                  reserved once and replayed from a CUDA graph;
* ``frame3d``     preprocessing and sort from 3D Gaussians and a camera;
* ``render``      the blend of one sorted frame into an image;
* ``pairs``       ``sort_pairs`` alone on the pairs of a frame;
* ``steps``       the five steps called one by one;
* ``normalized``  the frame with the 32-bit normalised key;
* ``host``        frames from pinned host memory and back, two in flight.

A case fixes its number of Gaussian-tile pairs (about nine tenths of what
its Gaussians would give: the rest of them are culled, as outside the view
frustum), so that its outputs have the same shapes for every seed.
"""
from __future__ import annotations

import collections
import functools
import math

import numpy as np
import torch

from paper_2511_16298_gb300 import host_pipeline, synth, tdgs

TILE = 16
RESOLUTIONS = ((640, 360), (1280, 720), (1920, 1080))  # of the request stream

# Distributions of projected Gaussians: clustered share of the means, number
# of centres, their spread (px), log-median / log-sd / clip of sigma, depth
# (None: uniform in [0.2, 50]; else log-median, log-sd), share of depths on a
# coarse grid (exact ties) and its step, share culled, margin off the image.
SCENES = {
    "uniform": dict(cl=0.0, centres=1, sd=0.0, sig=(math.log(3.0), 0.6, 64.0), depth=None, ties=(0.0, 1.0),
                    culled=0.0, margin=0.0),
    "clustered": dict(cl=0.70, centres=32, sd=60.0, sig=(math.log(4.0), 0.8, 256.0), depth=(math.log(5.0), 0.7),
                      ties=(0.0, 1.0), culled=0.0, margin=0.0),
    "dense": dict(cl=0.85, centres=128, sd=40.0, sig=(math.log(3.0), 1.0, 512.0), depth=(math.log(8.0), 0.9),
                  ties=(0.05, 0.125), culled=0.0, margin=0.0),
    "mixed": dict(cl=0.0, centres=1, sd=0.0, sig=(math.log(3.0), 0.9, 64.0), depth=(math.log(6.0), 0.8),
                  ties=(0.2, 0.5), culled=0.05, margin=51.2),
}


def listed():
    return [
        # a thumbnail or a small synthetic object: launches and latency count
        dict(name="frame 10k 256x256", kind="frame", scene="uniform", n=10_000, width=256, height=256),
        # a trained scene at 720p: the frame that the benchmark is quoted on
        dict(name="frame 1M 720p", kind="frame", scene="clustered", n=1_000_000, width=1280, height=720),
        # a large scene at 1080p, with many equal depths
        dict(name="frame 3M 1080p", kind="frame", scene="dense", n=3_000_000, width=1920, height=1080),
        # an odd 4K window with Gaussians culled, off the image and tied in depth
        dict(name="frame 778k odd 4K", kind="frame", scene="mixed", n=777_777, width=3839, height=2161),
        # a training step's or a flythrough's cameras in one call
        dict(name="views 16x500k", kind="views", n=500_000, views=16, width=1280, height=720),
        # six requests of a server, their batch replayed from a graph
        dict(name="graph 6 requests", kind="graph", scene="clustered", n=600_000, views=6),
        # from 3D Gaussians: projection and sort of one image
        dict(name="frame3d 500k 720p", kind="frame3d", n=500_000, width=1280, height=720),
        # the image of a sorted frame
        dict(name="render 500k 720p", kind="render", n=500_000, width=1280, height=720),
        # the sort step alone, as a program with its own duplication calls it
        dict(name="pairs of 1M 720p", kind="pairs", scene="clustered", n=1_000_000, width=1280, height=720),
        # the five steps one by one, at a small frame of the request stream
        dict(name="steps 250k 360p", kind="steps", scene="clustered", n=250_007, width=640, height=360),
        # the paper's 32-bit key
        dict(name="normalized 1M 720p", kind="normalized", scene="clustered", n=1_000_000, width=1280, height=720),
        # frames that live in host memory, two in flight
        dict(name="host 2x250k 720p", kind="host", scene="clustered", n=250_000, width=1280, height=720),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("frame", "frame", "frame", "views", "graph", "frame3d", "render", "pairs", "steps",
                       "normalized", "host"))
    case = dict(kind=kind)
    if kind in ("frame", "pairs", "steps", "normalized", "host", "graph"):
        case["scene"] = rng.choice(("uniform", "clustered", "dense", "mixed"))
    if kind == "graph":
        case.update(n=_log_uniform(rng, 5_000, 600_000), views=rng.randint(2, 8))
        return case
    case["width"] = _log_uniform(rng, 160, 1280 if kind == "views" else 3840)
    case["height"] = max(120, min(2160, int(case["width"] * rng.uniform(0.45, 0.8))))
    top = {"frame": 2_900_000, "views": 450_000, "frame3d": 1_500_000, "render": 700_000, "pairs": 1_500_000,
           "steps": 1_000_000, "normalized": 1_500_000, "host": 400_000}[kind]
    case["n"] = _log_uniform(rng, 4_000, top)
    if kind == "views":
        case["views"] = rng.randint(2, 16)
    return case


# ------------------------------------------------------------------- inputs
def _gen(seed, device="cuda"):
    g = torch.Generator(device=device)
    g.manual_seed(int(seed))
    return g


def _uniform(g, lo, hi, *shape):
    return torch.rand(*shape, generator=g, device=g.device, dtype=torch.float64) * (hi - lo) + lo


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device=g.device, dtype=torch.float64)


def _means(g, n, width, height, sc):
    size = torch.tensor([width, height], device=g.device, dtype=torch.float64)
    m = sc["margin"]
    xy = torch.rand(n, 2, generator=g, device=g.device, dtype=torch.float64) * (size + 2 * m) - m
    n_cl = int(round(sc["cl"] * n))
    if n_cl:
        centres = torch.rand(sc["centres"], 2, generator=g, device=g.device, dtype=torch.float64) * size
        which = torch.randint(0, sc["centres"], (n_cl,), generator=g, device=g.device)
        xy[:n_cl] = centres[which] + sc["sd"] * _normal(g, n_cl, 2)
        xy = xy[torch.randperm(n, generator=g, device=g.device)]
    return xy


def _depth(g, n, sc):
    if sc["depth"] is None:
        d = _uniform(g, 0.2, 50.0, n)
    else:
        d = torch.exp(sc["depth"][0] + sc["depth"][1] * _normal(g, n))
    share, step = sc["ties"]
    if share:
        tied = torch.rand(n, generator=g, device=g.device) < share
        d = torch.where(tied, torch.clamp(torch.round(d / step) * step, min=step), d)
    return d


def _pack(xy, depth, radius):
    rec = torch.empty(xy.shape[0], 4, device=xy.device, dtype=torch.int32)
    f = rec.view(torch.float32)
    f[:, :2] = xy.float()
    f[:, 2] = depth.float()
    rec[:, 3] = radius.to(torch.int32)
    return rec


def _grid(width, height):
    return (width + TILE - 1) // TILE, (height + TILE - 1) // TILE


def _boxes(rec, width, height):
    """First column and row, columns and rows of each record's tile box."""
    f, r = rec.view(torch.float32), rec[:, 3].float()
    box = []
    for k, top in enumerate(_grid(width, height)):
        lo = torch.clamp(torch.floor((f[:, k] - r) * 0.0625), 0, top).long()
        hi = torch.clamp(torch.floor(((f[:, k] + r) + 15.0) * 0.0625), 0, top).long()
        box.append((lo, torch.where(rec[:, 3] > 0, torch.clamp(hi - lo, min=0), torch.zeros_like(lo))))
    (x0, w), (y0, h) = box
    return x0, y0, w, h


def _count(rec, width, height):
    _, _, w, h = _boxes(rec, width, height)
    return w * h


def _squares(rest, width, height):
    """Tile squares that sum to `rest` pairs: (side in tiles) of each."""
    side, out = min(_grid(width, height)), []
    while rest:
        k = min(side, math.isqrt(rest))
        out.append(k)
        rest -= k * k
    return out


def _keep(counts, pairs, g):
    """The Gaussians to keep (a random subset of at most `pairs` pairs), the
    ones left out, and the pairs still missing; None if all are too few."""
    order = torch.randperm(counts.shape[0], generator=g, device=counts.device)
    cum = torch.cumsum(counts[order], 0)
    if int(cum[-1]) < pairs:
        return None
    kept = int((cum <= pairs).sum())
    return order[:kept], order[kept:], pairs - (int(cum[kept - 1]) if kept else 0)


def _fix(rec, width, height, pairs, g):
    """The same records with exactly `pairs` pairs: surplus Gaussians are
    culled, and a few of those cover tile squares that make up the rest."""
    while True:
        counts = _count(rec, width, height)
        found = _keep(counts, pairs, g)
        if found:
            break
        rec[:, 3] = torch.ceil(rec[:, 3] * 1.15).to(torch.int32)
    _, out, rest = found
    rec[out, 3] = 0
    for i, k in zip(out[counts[out] > 0].tolist(), _squares(rest, width, height)):
        rec.view(torch.float32)[i, :2] = 8.0 * k
        rec[i, 3] = max(1, 8 * k - 1)
    return rec


@functools.lru_cache(maxsize=None)
def _pairs_of(scene, n, width, height):
    ns = min(n, 20_000)
    return int(0.9 * int(_count(_drawn(scene, ns, width, height, _gen(1, "cpu")), width, height).sum()) * n / ns) + 1


def _records(scene, n, width, height, g):
    return _fix(_drawn(scene, n, width, height, g), width, height, _pairs_of(scene, n, width, height), g)


def _drawn(scene, n, width, height, g):
    """(n, 4) int32 view of n 16-byte records (x, y, depth, radius)."""
    sc = SCENES[scene]
    xy = _means(g, n, width, height, sc)
    mu, sd, top = sc["sig"]
    radius = torch.ceil(3.0 * torch.clamp(torch.exp(mu + sd * _normal(g, n)), 1.0, top))
    if sc["culled"]:
        radius[torch.rand(n, generator=g, device=g.device) < sc["culled"]] = 0
    return _pack(xy, _depth(g, n, sc), radius)


def _scene_means(n, g):
    return _uniform(g, -5.0, 5.0, n, 3)


def _scene_scales(n, g):
    return torch.exp(math.log(0.05) + 0.5 * _normal(g, n))


def _cameras(count, width, height, radius, jitter, near=(1.0, 1.0)):
    """`count` CAMERA records on a Fibonacci lattice, looking near the origin."""
    g = _gen(7, "cpu")
    u = _normal(g, count, 3)
    u = (u / u.norm(dim=1, keepdim=True) * (jitter * _uniform(g, 0.0, 1.0, count, 1) ** (1 / 3))).numpy()
    lo, hi = near
    dist = (radius * lo * (hi / lo) ** _uniform(g, 0.0, 1.0, count)).numpy()
    i = np.arange(count) + 0.5
    phi, theta = np.arccos(1.0 - 2.0 * i / count), math.pi * (1.0 + 5.0 ** 0.5) * i
    eye = np.stack([np.cos(theta) * np.sin(phi), np.cos(phi), np.sin(theta) * np.sin(phi)], 1) * dist[:, None]
    return np.stack([synth.camera(eye[v], u[v], width, height) for v in range(count)])


def _view_records(mean, scale, cam):
    """Isotropic splats of one camera as projected records."""
    rot = torch.tensor(np.asarray(cam["rot"], np.float64).reshape(3, 3), device=mean.device)
    t = mean @ rot.T + torch.tensor(np.asarray(cam["trans"], np.float64), device=mean.device)
    ok = t[:, 2] > 0.2
    z = torch.where(ok, t[:, 2], torch.ones_like(t[:, 2]))
    fx = float(cam["fx"])
    xy = torch.stack([fx * t[:, 0] / z + float(cam["cx"]), fx * t[:, 1] / z + float(cam["cy"])], 1)
    radius = torch.where(ok, torch.ceil(3.0 * fx * scale / z), torch.zeros_like(z))
    return _pack(xy, z, radius)


@functools.lru_cache(maxsize=None)
def _pairs_of_views(n, views, width, height):
    ns, g = min(n, 20_000), _gen(1, "cpu")
    mean, scale = _scene_means(ns, g), _scene_scales(ns, g)
    return [int(0.9 * int(_count(_view_records(mean, scale, c), width, height).sum()) * n / ns) + 1
            for c in _cameras(views, width, height, 15.0, 8.0, (0.25, 1.0))]


def _gaussians3d(n, g):
    """Means + opacity (n, 4) and covariances (n, 8), float32."""
    s2 = torch.exp(2.0 * (math.log(0.03) + 0.5 * _normal(g, n, 3)))
    q = _normal(g, n, 4)
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    r = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                     2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                     2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).view(n, 3, 3)
    s3 = (r * s2[:, None, :]) @ r.transpose(1, 2)
    g3 = torch.cat([_scene_means(n, g), _uniform(g, 0.05, 1.0, n, 1)], 1).float()
    cov = torch.zeros(n, 8, device=g.device, dtype=torch.float32)
    for k, (i, j) in enumerate(((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))):
        cov[:, k] = s3[:, i, j].float()
    return g3, cov


def _covariance2d(g3, cov, cam):
    """EWA projection in 64 bits: camera-space means, whether they are in
    front, and the entries xx, xy, yy of the 2D covariance."""
    dev = g3.device
    rot = torch.tensor(np.asarray(cam["rot"], np.float64).reshape(3, 3), device=dev)
    t = g3[:, :3].double() @ rot.T + torch.tensor(np.asarray(cam["trans"], np.float64), device=dev)
    fx, fy = float(cam["fx"]), float(cam["fy"])
    seen = t[:, 2] > float(cam["near_z"])
    z = torch.where(seen, t[:, 2], torch.ones_like(t[:, 2]))
    lx, ly = 0.65 * int(cam["width"]) / fx, 0.65 * int(cam["height"]) / fy
    u, v = torch.clamp(t[:, 0] / z, -lx, lx), torch.clamp(t[:, 1] / z, -ly, ly)
    o = torch.zeros_like(z)
    jac = torch.stack([torch.stack([fx / z, o, -fx * u / z], 1), torch.stack([o, fy / z, -fy * v / z], 1)], 1)
    xx, xy, xz, yy, yz, zz = cov[:, :6].double().unbind(1)
    s3 = torch.stack([xx, xy, xz, xy, yy, yz, xz, yz, zz], 1).view(-1, 3, 3)
    p = jac @ rot
    s2 = p @ s3 @ p.transpose(1, 2) + 0.3 * torch.eye(2, device=dev, dtype=torch.float64)
    return t, seen, s2[:, 0, 0], s2[:, 0, 1], s2[:, 1, 1]


@functools.lru_cache(maxsize=None)
def _pairs_of_3d(n, width, height):
    ns = min(n, 20_000)
    g3, cov = _gaussians3d(ns, _gen(1, "cpu"))
    cam = _camera3d(width, height)
    t, seen, a, b, d = _covariance2d(g3, cov, cam)
    mid = 0.5 * (a + d)
    radius = torch.ceil(3.0 * torch.sqrt(mid + torch.sqrt(torch.clamp(mid * mid - a * d + b * b, min=0.1))))
    z = torch.where(seen, t[:, 2], torch.ones_like(t[:, 2]))
    xy = torch.stack([float(cam["fx"]) * t[:, 0] / z + float(cam["cx"]),
                      float(cam["fy"]) * t[:, 1] / z + float(cam["cy"])], 1)
    rec = _pack(xy, z, torch.where(seen, radius, torch.zeros_like(radius)))
    return int(0.9 * int(_count(rec, width, height).sum()) * n / ns) + 1


def _camera3d(width, height):
    return _cameras(1, width, height, 15.0, 4.0)[0]


def _scene3d(n, width, height, g):
    """3D Gaussians with a fixed number of pairs in the camera's image:
    surplus ones lie behind the camera, a few points make up the rest."""
    g3, cov = _gaussians3d(n, g)
    cam, pairs = _camera3d(width, height), _pairs_of_3d(n, width, height)
    while True:
        counts = _count(_context().preprocess(g3, cov, cam, with_conic=False)[0], width, height)
        found = _keep(counts, pairs, g)
        if found:
            break
        cov *= 1.2
    _, out, rest = found
    rot = np.asarray(cam["rot"], np.float64).reshape(3, 3)

    def world(p):  # camera space to world space
        return torch.tensor(rot.T @ (np.asarray(p) - np.asarray(cam["trans"], np.float64)), device=g3.device).float()

    g3[out, :3] = world([0.0, 0.0, -5.0])
    point = out[counts[out] > 0][:rest]  # one tile each: points at the centre of an inner tile
    at = [(16 * (size // 32) + 8 - c) / f for size, c, f in ((width, float(cam["cx"]), float(cam["fx"])),
                                                             (height, float(cam["cy"]), float(cam["fy"])))]
    g3[point, :3] = world([4.0 * at[0], 4.0 * at[1], 4.0])
    cov[point] = 0.0
    return g3, cov


def _splats(n, width, height, g):
    """Records, conic + opacity and colours of projected anisotropic splats."""
    sc = SCENES["clustered"]
    s = torch.clamp(torch.exp(math.log(1.8) + 0.5 * _normal(g, n, 2)), 0.3, 60.0)
    a = _uniform(g, 0.0, math.pi, n)
    c, d = torch.cos(a), torch.sin(a)
    v0, v1 = s[:, 0] ** 2, s[:, 1] ** 2
    xx, yy, xy = c * c * v0 + d * d * v1 + 0.3, d * d * v0 + c * c * v1 + 0.3, c * d * (v0 - v1)
    det = xx * yy - xy * xy
    mid = 0.5 * (xx + yy)
    radius = torch.ceil(3.0 * torch.sqrt(mid + torch.sqrt(torch.clamp(mid * mid - det, min=0.1))))
    rec = _pack(_means(g, n, width, height, sc), _depth(g, n, sc), radius)
    conic = torch.stack([yy / det, -xy / det, xx / det, _uniform(g, 0.05, 1.0, n)], 1).float()
    rgb = _uniform(g, 0.0, 1.0, n, 3).float()
    return rec.contiguous(), conic.contiguous(), rgb.contiguous()


def _pairs(rec, width, height):
    """Gaussian-tile pairs in Gaussian order: (tile << 32 | depth bits), index."""
    gx, _ = _grid(width, height)
    x0, y0, w, h = _boxes(rec, width, height)
    cnt = w * h
    idx = torch.repeat_interleave(torch.arange(rec.shape[0], device=rec.device), cnt)
    first = torch.cumsum(cnt, 0) - cnt
    at = torch.arange(idx.shape[0], device=rec.device) - first[idx]
    wi = w[idx]
    tile = (y0[idx] + torch.div(at, wi, rounding_mode="floor")) * gx + x0[idx] + at % wi
    return (tile << 32) | rec[:, 2].long()[idx], idx.to(torch.int32)


_shared = {}
# A result is a view of its context's buffers: the contexts of the last few
# graphs outlive their states, as a program keeps its context while it reads.
_kept = collections.deque(maxlen=4)


def _context():
    """The context that a program keeps for the calls that it makes in turn."""
    if "ctx" not in _shared:
        _shared["ctx"] = tdgs.Context(0)
    return _shared["ctx"]


def _pipeline():
    if "pipe" not in _shared:
        _shared["pipe"] = host_pipeline.HostPipeline(0, depth=2)
    return _shared["pipe"]


def prepare(case, seed):
    kind, n, g = case["kind"], case["n"], _gen(seed)
    w, h = case.get("width"), case.get("height")
    st = dict(kind=kind, width=w, height=h)
    if kind == "views":
        mean, scale = _scene_means(n, g), _scene_scales(n, g)
        cams = _cameras(case["views"], w, h, 15.0, 8.0, (0.25, 1.0))
        st.update(ctx=_context(), views=[(_fix(_view_records(mean, scale, c), w, h, m, g), w, h) for c, m in
                                         zip(cams, _pairs_of_views(n, case["views"], w, h))])
    elif kind == "graph":
        ctx = tdgs.Context(0)  # a graph keeps its context's buffers: one of its own
        _kept.append(ctx)
        views = [(_records(case["scene"], nv, vw, vh, g), vw, vh) for nv, vw, vh in _request_shapes(case)]
        m = sum(r[3] for r in ctx.sort_views(views))
        ctx.reserve_views(views, m + m // 8 + 1024)
        ctx.sort_views_async(views)
        ctx.views_results(len(views))
        graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            with torch.cuda.graph(graph, stream=side):
                ctx.sort_views_async(views)
        torch.cuda.current_stream().wait_stream(side)
        st.update(ctx=ctx, views=views, graph=graph)
    elif kind == "frame3d":
        g3, cov = _scene3d(n, w, h, g)
        st.update(ctx=_context(), g3=g3, cov=cov, cam=_camera3d(w, h))
    elif kind == "render":
        rec, conic, rgb = _splats(n, w, h, g)
        _, values, ranges, _ = _context().sort_frame(rec, w, h, copy=True)
        st.update(ctx=_context(), rec=rec, conic=conic, rgb=rgb, values=values, ranges=ranges)
    elif kind == "pairs":
        keys, values = _pairs(_records(case["scene"], n, w, h, g), w, h)
        st.update(ctx=_context(), keys=keys, values=values, bits=tdgs.tile_bits(w, h),
                  work=[torch.empty_like(t) for t in (keys, values, keys, values)])
    elif kind == "host":
        st.update(pipe=_pipeline(), frames=[_records(case["scene"], n, w, h, g).cpu().pin_memory() for _ in range(2)])
    else:
        st.update(ctx=_context(), rec=_records(case["scene"], n, w, h, g))
    return st


def _request_shapes(case):
    """Sizes of a batch's requests: from a sixth of the largest up, resolutions in turn."""
    k = case["views"]
    return [(max(1, case["n"] * (i + 1) // k - 13 * i), *RESOLUTIONS[i % 3]) for i in range(k)]


# --------------------------------------------------------------------- pass
def run(st):
    kind, w, h = st["kind"], st["width"], st["height"]
    if kind == "frame":
        return st["ctx"].sort_frame(st["rec"], w, h)
    if kind == "views":
        return [r[:3] for r in st["ctx"].sort_views(st["views"])]
    if kind == "graph":
        st["graph"].replay()
        return [r[:3] for r in st["ctx"].views_results(len(st["views"]))]
    if kind == "frame3d":
        k, v, r, _, rec, conic = st["ctx"].sort_frame_3d(st["g3"], st["cov"], st["cam"])
        return dict(keys=k, values=v, ranges=r, records=rec, conic=conic)
    if kind == "render":
        return st["ctx"].render(st["rec"], st["conic"], st["rgb"], st["values"], st["ranges"], w, h, (0.1, 0.2, 0.3))
    if kind == "pairs":  # the call sorts in place: the program's pairs are copied first
        k, v, ka, va = st["work"]
        k.copy_(st["keys"])
        v.copy_(st["values"])
        return st["ctx"].sort_pairs(k, v, st["bits"], tdgs.SORT_DEPTH_POSITIVE, ka, va)
    if kind == "steps":
        ctx, rec = st["ctx"], st["rec"]
        counts = ctx.count_tiles(rec, w, h)
        offsets, total = ctx.scan(counts)
        keys, values = ctx.duplicate_keys(rec, offsets, w, h, int(total.item()))
        keys, values = ctx.sort_pairs(keys, values, tdgs.tile_bits(w, h), tdgs.SORT_DEPTH_POSITIVE)
        return counts, offsets, keys, values, ctx.tile_ranges(keys, tdgs.num_tiles(w, h))
    if kind == "normalized":
        return st["ctx"].sort_frame_normalized(st["rec"], w, h)
    pipe = st["pipe"]
    tickets = [pipe.submit(f, w, h) for f in st["frames"]]
    return [(r.keys, r.values, r.ranges) for r in map(pipe.result, tickets)]


# --------------------------------------------------------- accounting, exact
def work(case):
    """Each input read once and each output written once; a blend also needs
    about 20 operations per pixel of each splat's footprint."""
    kind, n = case["kind"], case["n"]
    w, h = case.get("width"), case.get("height")

    def frame_bytes(n, m, w, h):
        return 16.0 * n + 12 * m + 8 * tdgs.num_tiles(w, h)

    if kind == "graph":
        return dict(bytes=sum(frame_bytes(nv, _pairs_of(case["scene"], nv, vw, vh), vw, vh)
                              for nv, vw, vh in _request_shapes(case)), flops=0.0)
    if kind == "views":
        return dict(bytes=sum(frame_bytes(n, m, w, h) for m in _pairs_of_views(n, case["views"], w, h)), flops=0.0)
    if kind == "frame3d":
        m = _pairs_of_3d(n, w, h)
        return dict(bytes=48.0 * n + 32 * n + 12 * m + 8 * tdgs.num_tiles(w, h), flops=150.0 * n)
    if kind == "render":
        ns = min(n, 20_000)
        rec, _, _ = _splats(ns, w, h, _gen(1, "cpu"))
        m = int(_count(rec, w, h).sum()) * n / ns
        area = float((math.pi * rec[:, 3].double() ** 2).sum()) * n / ns
        return dict(bytes=44.0 * n + 4 * m + 8 * tdgs.num_tiles(w, h) + 12.0 * w * h, flops=20.0 * area)
    m = _pairs_of(case["scene"], n, w, h)
    if kind == "pairs":
        return dict(bytes=24.0 * m, flops=0.0)
    if kind == "steps":  # records, counts, offsets, then pairs out, in and out sorted, ranges
        return dict(bytes=16.0 * n + 8 * n + 12 * m * 3 + 8 * tdgs.num_tiles(w, h), flops=0.0)
    if kind == "normalized":
        return dict(bytes=16.0 * n + 8 * m + 8 * tdgs.num_tiles(w, h), flops=0.0)
    return dict(bytes=frame_bytes(n, m, w, h) * (2 if kind == "host" else 1), flops=0.0)


def exact(case, seed):
    """The floating outputs in 64 bits; whole numbers have none."""
    kind, n, g = case["kind"], case["n"], _gen(seed)
    w, h = case.get("width"), case.get("height")
    if kind == "frame3d":
        g3, cov = _scene3d(n, w, h, g)
        _, seen, a, b, d = _covariance2d(g3, cov, _camera3d(w, h))
        det = a * d - b * b
        conic = torch.stack([d / det, -b / det, a / det, g3[:, 3].double()], 1)
        conic = torch.where((seen & (det > 0))[:, None], conic, torch.zeros_like(conic))
        return dict(keys=None, values=None, ranges=None, records=None, conic=conic)
    if kind == "render":
        return _exact_image(*_splats(n, w, h, g), w, h, (0.1, 0.2, 0.3))
    return None


def _exact_image(rec, conic, rgb, width, height, background):
    """Front-to-back blend of every tile in 64 bits, one list position at a time."""
    dev = rec.device
    gx, gy = _grid(width, height)
    keys, values = _pairs(rec, width, height)
    order = torch.sort(keys, stable=True).indices  # pairs come in index order
    tile, g = (keys >> 32)[order], values.long()[order]
    begin = torch.searchsorted(tile, torch.arange(gx * gy + 1, device=dev))
    first, length = begin[:-1], begin[1:] - begin[:-1]
    pix = torch.arange(TILE * TILE, device=dev)
    ids = torch.arange(gx * gy, device=dev)
    px = ((ids % gx) * TILE)[:, None] + (pix % TILE)[None]
    py = (torch.div(ids, gx, rounding_mode="floor") * TILE)[:, None] + torch.div(pix, TILE, rounding_mode="floor")[None]
    inside = (px < width) & (py < height)
    light = torch.ones(gx * gy, TILE * TILE, device=dev, dtype=torch.float64)
    colour = torch.zeros(gx * gy, TILE * TILE, 3, device=dev, dtype=torch.float64)
    mean, con, col = rec.view(torch.float32)[:, :2].double(), conic.double(), rgb.double()
    done = ~inside

    def blend(act, done_a, light_a, colour_a, fx, fy, j):
        i = g[first[act] + j]
        d0, d1 = mean[i, 0][:, None] - fx, mean[i, 1][:, None] - fy
        c = con[i]
        power = -0.5 * (c[:, 0, None] * d0 * d0 + c[:, 2, None] * d1 * d1) - c[:, 1, None] * d0 * d1
        alpha = torch.clamp(c[:, 3, None] * torch.exp(power), max=0.99)
        on = ~done_a & (power <= 0) & (alpha >= 1.0 / 255.0)
        left = light_a * (1.0 - alpha)
        stop = on & (left < 0.0001)
        on = on & ~stop
        colour_a += torch.where(on, alpha * light_a, torch.zeros_like(alpha))[:, :, None] * col[i][:, None, :]
        light_a.copy_(torch.where(on, left, light_a))
        done_a |= stop

    j, longest = 0, int(length.max()) if gx * gy else 0
    while j < longest:
        act = torch.nonzero((length > j) & ~done.all(1)).flatten()
        if act.numel() == 0:
            break
        upto = min(longest, j + 32)
        da, la, ca = done[act], light[act], colour[act]
        fx, fy = px[act].double(), py[act].double()
        short = length[act]
        for q in range(j, upto):
            have = torch.nonzero(short > q).flatten() if int(short.min()) <= q else None
            if have is None:
                blend(act, da, la, ca, fx, fy, q)
            elif have.numel():
                dh, lh, ch = da[have], la[have], ca[have]
                blend(act[have], dh, lh, ch, fx[have], fy[have], q)
                da[have], la[have], ca[have] = dh, lh, ch
        done[act], light[act], colour[act] = da, la, ca
        j = upto
    colour += light[:, :, None] * torch.tensor(background, device=dev, dtype=torch.float64)
    image = torch.empty(height, width, 3, device=dev, dtype=torch.float64)
    image[py[inside], px[inside]] = colour[inside]
    return image
