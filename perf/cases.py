"""What is timed: passes that a program using this package makes, through its public entry points.

A case names its kind, its sizes and its options; the listed cases are points of the ranges that
draw() spreads over:

  trace     rays through a BVH that is built once: camera rays (a row-major image), one diffuse bounce
            per camera hit, one shadow ray per camera hit, or random rays; closest or any hit
  points    closest point queries around a mesh
  train     the differentiable closest hit: forward and gradients of vertices and rays
  backward  the gradient pass alone, for the hits of a rendered image
  batch     many scenes of uneven size in one launch
  rebuild   an animated mesh whose topology is rebuilt every frame on the GPU, then traced
  refit     an animated mesh whose tree is kept and refitted every frame, then traced

Scenes are a terrain (a value-noise height field with spheres on it; indexed) or a soup of random
triangles in the unit cube. Inputs are made on the GPU from the seed alone.
"""
import functools
import math

import torch

from paper_2511_15028_gb300 import scenes, scion

INF = math.inf

# The layouts that the ranges cover; each with triangles copied into the leaves or referred to.
LAYOUTS = {
    "bvh2_f32": dict(width=2, box_layout="aos", box_prec="f32"),
    "bvh2_q16": dict(width=2, box_layout="aos", box_prec="q16"),
    "bvh2_eq10": dict(width=2, box_layout="aos", box_prec="eq10"),
    "bvh4_f32": dict(width=4, box_layout="soa", box_prec="f32"),
    "bvh4_f32_bfs": dict(width=4, box_layout="soa", box_prec="f32", order="bfs"),
    "bvh4_u8_bfs": dict(width=4, box_layout="soa", box_prec="u8", order="bfs"),
    "bvh8_f16": dict(width=8, box_layout="soa", box_prec="f16"),
    "bvh8_u8": dict(width=8, box_layout="aos", box_prec="u8"),
    "bvh8_u16": dict(width=8, box_layout="aos", box_prec="u16"),
}
# The node families of a multi-scene launch among them.
BATCH_LAYOUTS = ("bvh2_f32", "bvh2_q16", "bvh4_f32", "bvh4_u8_bfs", "bvh8_f16", "bvh8_u8")


def listed():
    return [
        # the smallest call: a handful of visibility questions of a game or a planner, on a small level
        dict(name="visibility_1k", kind="trace", scene="terrain", tris=65_000, layout="bvh8_u8", prims="indirect",
             rays="random", n=1_000, query="any", tmax=0.5, fetch=0, order=0),
        # camera rays of a full-HD frame, the first thing a renderer traces
        dict(name="camera_1080p", kind="trace", scene="terrain", tris=1_373_138, layout="bvh4_f32", prims="direct",
             rays="camera", width=1920, height=1080, query="closest", tmax=INF, fetch=0, order=3),
        # global illumination: one diffuse bounce of that frame, in the half-precision 8-wide layout
        dict(name="bounce", kind="trace", scene="terrain", tris=1_373_138, layout="bvh8_f16", prims="direct",
             rays="bounce", n=750_000, width=1920, height=1080, query="closest", tmax=INF, fetch=8, order=3),
        # shadows of that frame toward one light, every parameter left at its default
        dict(name="shadow", kind="trace", scene="terrain", tris=1_373_138, layout="bvh4_f32", prims="indirect",
             rays="shadow", n=750_000, width=1920, height=1080, query="any", tmax=INF, fetch=0, order=0),
        # the largest: random rays in a tree far larger than L2 (particle or radio transport)
        dict(name="soup_closest_8m", kind="trace", scene="soup", tris=1 << 23, layout="bvh4_u8_bfs", prims="direct",
             rays="random", n=1 << 23, query="closest", tmax=INF, fetch=4, order=0),
        # short random rays (ambient occlusion) in the compact binary layout
        dict(name="soup_any_q16", kind="trace", scene="soup", tris=2_000_003, layout="bvh2_q16", prims="direct",
             rays="random", n=1_000_003, query="any", tmax=0.05, fetch=0, order=0),
        # distance field sampling and mesh registration
        dict(name="points_1m", kind="points", scene="terrain", tris=1_373_138, layout="bvh4_f32", prims="direct",
             n=1 << 20),
        # a small optimisation step: 4,096 triangles, 128 x 128 rays, gradients of vertices and rays
        dict(name="train_128", kind="train", scene="terrain", tris=4_096, layout="bvh2_f32", prims="indirect",
             width=128, height=128),
        # the gradient pass of a full-HD image
        dict(name="backward_1080p", kind="backward", scene="terrain", tris=1_373_138, layout="bvh4_f32",
             prims="direct", width=1920, height=1080),
        # asset thumbnails, sensor simulation in many worlds: scenes of uneven size in one launch
        dict(name="batch_48", kind="batch", scenes=48, tris=400_000, n=200_000, layout="bvh4_u8_bfs", prims="direct",
             fetch=0, order=0),
        # a deforming mesh without frame coherence: new tree, then a full-HD frame
        dict(name="rebuild_1080p", kind="rebuild", scene="terrain", tris=1_373_138, layout="bvh4_f32", prims="direct",
             width=1920, height=1080, fetch=0, order=3),
        # an animated mesh: refit the compressed 8-wide tree, then a 720p frame
        dict(name="refit_720p", kind="refit", scene="terrain", tris=1_373_138, layout="bvh8_u8", prims="direct",
             width=1280, height=720, fetch=0, order=3),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("trace", "trace", "trace", "points", "train", "backward", "batch", "rebuild", "refit"))
    layout = rng.choice(sorted(LAYOUTS))
    prims = rng.choice(("direct", "indirect"))
    fetch, order = rng.choice((0, 0, 4, 8)), rng.choice((0, 2, 3))
    case = dict(kind=kind, layout=layout, prims=prims)
    if kind == "batch":
        return dict(case, scenes=rng.randint(3, 60), tris=_log(rng, 2_000, 400_000), n=_log(rng, 1_000, 200_000),
                    layout=rng.choice(BATCH_LAYOUTS), fetch=fetch, order=order)
    case["scene"] = "soup" if kind == "trace" and rng.random() < 0.5 else "terrain"
    case["tris"] = _log(rng, 1_000, 2_000_000)
    w = _log(rng, 17, 1920)
    image = dict(width=w, height=max(1, int(w * rng.uniform(0.4, 1.0) * 9 / 16)))
    if kind == "points":
        return dict(case, n=_log(rng, 300, 700_000))
    if kind in ("train", "backward"):
        return dict(case, **image)
    if kind in ("rebuild", "refit"):
        return dict(case, fetch=fetch, order=order, **image)
    rays = "random" if case["scene"] == "soup" else rng.choice(("camera", "bounce", "shadow", "random"))
    query = "any" if rays == "shadow" else "closest" if rays in ("camera", "bounce") else rng.choice(("closest", "any"))
    case.update(rays=rays, query=query, fetch=fetch, order=order)
    if rays == "random":
        return dict(case, n=_log(rng, 250, 1_500_000), tmax=rng.choice((INF, 0.05, 0.5)) if query == "any" else INF)
    if rays != "camera":
        case["n"] = max(1, int(0.4 * image["width"] * image["height"]))
    return dict(case, tmax=INF, **image)


# ------------------------------------------------------------------ scenes


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)


def _uniform(g, shape, lo=0.0, hi=1.0):
    return lo + (hi - lo) * torch.rand(shape, generator=g, device="cuda", dtype=torch.float64)


def _unit(v):
    return v / v.norm(dim=-1, keepdim=True)


def _noise(g, x, y):
    """Six octaves of value noise over [-1, 1]^2."""
    z, amp, res = torch.zeros_like(x), 0.25, 4
    for _ in range(6):
        table = _uniform(g, (res + 1, res + 1), -1, 1)
        gx, gy = (x + 1) * 0.5 * res, (y + 1) * 0.5 * res
        i, j = gx.floor().long().clamp(0, res - 1), gy.floor().long().clamp(0, res - 1)
        fx, fy = gx - i, gy - j
        fx, fy = fx * fx * (3 - 2 * fx), fy * fy * (3 - 2 * fy)
        low = table[j, i] * (1 - fx) + table[j, i + 1] * fx
        high = table[j + 1, i] * (1 - fx) + table[j + 1, i + 1] * fx
        z += amp * (low * (1 - fy) + high * fy)
        amp, res = amp * 0.5, res * 2
    return z


@functools.lru_cache(maxsize=None)
def _sphere():
    v, f = scenes.icosphere(3)
    return torch.from_numpy(v).cuda(), torch.from_numpy(f).cuda()


def _terrain(g, tris):
    """(vertices float32, indices int32): a quarter of the triangles in spheres of 1,280."""
    spheres = tris // 4 // 1280
    side = max(2, int(math.sqrt((tris - 1280 * spheres) / 2) + 0.5) + 1)
    line = torch.linspace(-1, 1, side, dtype=torch.float64, device="cuda")
    y, x = torch.meshgrid(line, line, indexing="ij")
    ground = torch.stack([x, y, _noise(g, x, y)], -1).reshape(-1, 3)
    j, i = torch.meshgrid(torch.arange(side - 1, device="cuda"), torch.arange(side - 1, device="cuda"), indexing="ij")
    a = j * side + i
    faces = torch.stack([torch.stack([a, a + 1, a + side + 1], -1), torch.stack([a, a + side + 1, a + side], -1)], 2)
    verts, index = [ground], [faces.reshape(-1, 3)]
    if spheres:
        sv, sf = _sphere()
        c = torch.cat([_uniform(g, (spheres, 2), -1, 1), _uniform(g, (spheres, 1), 0, 0.5)], 1)
        r = _uniform(g, (spheres, 1, 1), math.log(0.005), math.log(0.05)).exp()
        verts.append((sv[None] * r + c[:, None]).reshape(-1, 3))
        start = side * side + sv.shape[0] * torch.arange(spheres, device="cuda")
        index.append((sf[None] + start[:, None, None]).reshape(-1, 3))
    return torch.cat(verts).float(), torch.cat(index).int()


def _soup(g, tris):
    """Equilateral triangles, log-normal edges that keep the density of 2^23 triangles of edge 0.002."""
    out = torch.empty((tris, 3, 3), dtype=torch.float32, device="cuda")
    for b in range(0, tris, 1 << 20):
        m = min(1 << 20, tris - b)
        n = _unit(torch.randn((m, 3), generator=g, device="cuda", dtype=torch.float64))
        e = torch.zeros_like(n).scatter_(1, n.abs().argmin(1, keepdim=True), 1.0)
        s = _unit(torch.linalg.cross(n, e))
        t = torch.linalg.cross(n, s)
        edge = 0.002 * math.sqrt((1 << 23) / tris) * torch.exp(
            0.5 * torch.randn((m, 1), generator=g, device="cuda", dtype=torch.float64))
        turn, c = _uniform(g, (m, 1), 0, 2 * math.pi), _uniform(g, (m, 3))
        for k in range(3):
            a = turn + k * 2 * math.pi / 3
            out[b:b + m, k] = (c + edge / math.sqrt(3) * (a.cos() * s + a.sin() * t)).float()
    return out.reshape(-1, 3), None


def _scene(g, case):
    return _soup(g, case["tris"]) if case.get("scene") == "soup" else _terrain(g, case["tris"])


def _triangles(verts, index):
    return verts.reshape(-1, 3, 3) if index is None else verts[index.long()]


def _layout(case):
    return scion.layout(prim_ref=case["prims"], **LAYOUTS[case["layout"]])


def _build(verts, index, case):
    """Scenes up to a few million triangles are built on the host (the better tree), larger ones on the GPU."""
    if case["tris"] > 2_500_000:
        return scion.scion_build_gpu(verts, _layout(case), index)
    return scion.scion_build(verts, _layout(case), index)


# ------------------------------------------------------------------ rays


def _rays(o, d, tmax):
    r = torch.empty((d.shape[0], 8), dtype=torch.float32, device="cuda")
    r[:, 0:3], r[:, 3], r[:, 4:7], r[:, 7] = o.float(), 1e-4, d.float(), tmax
    return r


EYE, LIGHT = (0.0, -2.2, 1.4), (2.0, 2.0, 3.0)


def _camera(w, h):
    """Position, view axes (forward, right, up) and the half extents of the image plane."""
    eye = torch.tensor(EYE, dtype=torch.float64, device="cuda")
    f = _unit(-eye)
    r = _unit(torch.linalg.cross(f, torch.tensor([0.0, 0.0, 1.0], dtype=torch.float64, device="cuda")))
    th = math.tan(math.radians(45.0) / 2)
    return eye, f, r, torch.linalg.cross(r, f), th * w / h, th


def _camera_rays(w, h):
    eye, f, r, u, tx, ty = _camera(w, h)
    sx = ((torch.arange(w, device="cuda", dtype=torch.float64) + 0.5) / w * 2 - 1) * tx
    sy = (1 - (torch.arange(h, device="cuda", dtype=torch.float64) + 0.5) / h * 2) * ty
    d = _unit(f + sx[None, :, None] * r + sy[:, None, None] * u).reshape(-1, 3)
    return _rays(eye.expand_as(d), d, INF)


def _random_rays(g, n, lo, hi, tmax):
    o = lo + (hi - lo) * _uniform(g, (n, 3))
    return _rays(o, _unit(torch.randn((n, 3), generator=g, device="cuda", dtype=torch.float64)), tmax)


def _moeller(o, d, tmin, tmax, p0, p1, p2):
    """t, u, v and whether the ray hits, in 64 bits."""
    e1, e2, s = p1 - p0, p2 - p0, o - p0
    q = torch.linalg.cross(d, e2)
    det = (e1 * q).sum(-1)
    x = torch.linalg.cross(s, e1)
    t, u, v = (e2 * x).sum(-1) / det, (s * q).sum(-1) / det, (d * x).sum(-1) / det
    return t, u, v, (det != 0) & (u >= 0) & (v >= 0) & (u + v <= 1) & (t >= tmin) & (t <= tmax)


def _nearest(n, ray, t, u, v, tri):
    """The nearest hit of each ray (the lowest triangle where two are as near) from a list of hits."""
    bt = torch.full((n,), INF, dtype=torch.float64, device="cuda").scatter_reduce_(0, ray, t, "amin")
    m = t == bt[ray]
    ray, u, v, tri = ray[m], u[m], v[m], tri[m]
    bi = torch.full((n,), 1 << 40, device="cuda").scatter_reduce_(0, ray, tri, "amin")
    m = tri == bi[ray]
    bu = torch.zeros((n,), dtype=torch.float64, device="cuda").index_copy_(0, ray[m], u[m])
    bv = torch.zeros((n,), dtype=torch.float64, device="cuda").index_copy_(0, ray[m], v[m])
    return bt, bu, bv, torch.where(bt < INF, bi, -1)


def _render(verts, index, w, h):
    """Closest hits (t, u, v, triangle or -1) of the camera's rays by drawing every triangle, in 64 bits."""
    rays, tri = _camera_rays(w, h).double(), _triangles(verts, index).double()
    eye, f, r, u, tx, ty = _camera(w, h)
    p = tri - eye
    z = p @ f
    px, py = ((p @ r) / z / tx + 1) / 2 * w - 0.5, (1 - (p @ u) / z / ty) / 2 * h - 0.5
    x0, x1 = (px.amin(1) - 0.01).ceil().clamp(0, w).long(), (px.amax(1) + 0.01).floor().clamp(-1, w - 1).long()
    y0, y1 = (py.amin(1) - 0.01).ceil().clamp(0, h).long(), (py.amax(1) + 0.01).floor().clamp(-1, h - 1).long()
    bw = (x1 - x0 + 1).clamp(min=0)
    count = bw * (y1 - y0 + 1).clamp(min=0)
    seen = count.nonzero()[:, 0]
    ends = count[seen].cumsum(0)
    found, total = [], int(ends[-1]) if len(seen) else 0
    for b in range(0, total, 1 << 22):
        k = torch.arange(b, min(total, b + (1 << 22)), device="cuda")
        at = torch.searchsorted(ends, k, right=True)
        t = seen[at]
        k = k - (ends[at] - count[t])
        pixel = (y0[t] + k // bw[t]) * w + x0[t] + k % bw[t]
        ray, c = rays[pixel], tri[t]
        ht, hu, hv, hit = _moeller(ray[:, 0:3], ray[:, 4:7], 1e-4, INF, c[:, 0], c[:, 1], c[:, 2])
        found.append([x[hit] for x in (pixel, ht, hu, hv, t)])
    if not found:
        found = [[torch.empty(0, dtype=d, device="cuda") for d in (torch.long,) + (torch.float64,) * 3 + (torch.long,)]]
    return _nearest(w * h, *(torch.cat(x) for x in zip(*found)))


def _second_rays(g, verts, index, case):
    """Bounce or shadow rays of n camera hits (about one for each hit there is), in image order."""
    _, u, v, tri = _render(verts, index, case["width"], case["height"])
    m = (tri >= 0).nonzero()[:, 0]
    if not len(m):  # an image too small to hit anything
        return _random_rays(g, case["n"], verts.amin(0).double(), verts.amax(0).double(), case["tmax"])
    m = m[torch.arange(case["n"], device="cuda") * len(m) // case["n"]]
    c, u, v = _triangles(verts, index)[tri[m]].double(), u[m, None], v[m, None]
    p = (1 - u - v) * c[:, 0] + u * c[:, 1] + v * c[:, 2]
    if case["rays"] == "shadow":
        to = torch.tensor(LIGHT, dtype=torch.float64, device="cuda") - p
        dist = to.norm(dim=1, keepdim=True)
        return _rays(p, to / dist, ((1 - 1e-4) * dist[:, 0]).float())
    n = _unit(torch.linalg.cross(c[:, 1] - c[:, 0], c[:, 2] - c[:, 0]))
    n = torch.where((n * (p - torch.tensor(EYE, dtype=torch.float64, device="cuda"))).sum(1, keepdim=True) > 0, -n, n)
    # a cosine-weighted direction: the normal plus a point of the unit sphere
    d = n + _unit(torch.randn(n.shape, generator=g, device="cuda", dtype=torch.float64))
    return _rays(p, _unit(torch.where(d.norm(dim=1, keepdim=True) > 1e-6, d, n)), INF)


def _trace_rays(g, verts, index, case):
    if case["rays"] == "camera":
        return _camera_rays(case["width"], case["height"])
    if case["rays"] == "random":
        lo, hi = verts.amin(0).double(), verts.amax(0).double()
        return _random_rays(g, case["n"], lo, hi, case["tmax"])
    return _second_rays(g, verts, index, case)


def _params(case, raster=0):
    return scion.TraceParams(rays_per_fetch=case["fetch"], ordered_children=case["order"],
                             raster_width=0 if case["fetch"] else raster)


def _points(g, verts, n):
    """Points in the mesh's box, a tenth of its size wider on every side; no limit on the distance."""
    lo, hi = verts.amin(0).double(), verts.amax(0).double()
    p = torch.empty((n, 4), dtype=torch.float32, device="cuda")
    p[:, :3] = (lo + (hi - lo) * _uniform(g, (n, 3), -0.1, 1.1)).float()
    p[:, 3] = INF
    return p


def _batch_sizes(case, s):
    a, b = (0.618034 * s) % 1, (0.754878 * s) % 1
    return int(1_000 * (case["tris"] / 1_000) ** (1 - a)), int(500 * (case["n"] / 500) ** (1 - b))


def _batch_parts(g, case):
    """Per scene: vertices, indices, rays (half a camera's from outside, half random). Sizes are spread over
    their logarithms, the same for every seed; the scenes and rays are not."""
    for s in range(case["scenes"]):
        tris, n = _batch_sizes(case, s)
        verts, index = _soup(g, tris) if s % 2 else _terrain(g, tris)
        lo, hi = verts.amin(0).double(), verts.amax(0).double()
        rays = _random_rays(g, n, lo, hi, INF)
        w = max(1, int(math.sqrt(n / 2)))
        h = n // 2 // w
        if h:
            out = _camera_rays(w, h)
            out[:, 0:3] += ((lo + hi) / 2).float()
            rays[:w * h] = out
        yield verts, index, rays


def _moved(verts):
    """The deformed frame of an animation."""
    return (verts + 0.02 * torch.sin(3.0 * verts[:, [1, 2, 0]])).contiguous()


# ------------------------------------------------------------------ the cases


def _inputs(case, seed):
    """The inputs of a case that are made without the package's kernels."""
    g = _generator(seed)
    verts, index = _scene(g, case)
    s = {"verts": verts, "index": index}
    kind = case["kind"]
    if kind == "trace":
        s["rays"] = _trace_rays(g, verts, index, case)
    elif kind == "points":
        s["points"] = _points(g, verts, case["n"])
    else:
        s["rays"] = _camera_rays(case["width"], case["height"])
        if kind in ("train", "backward"):
            s["grad"] = torch.randn((s["rays"].shape[0], 3), generator=g, device="cuda")
        if kind == "backward":  # the forward's results, as it lays them out
            h = _render(verts, index, case["width"], case["height"])
            s["hits"] = torch.stack([x.float().view(torch.int32) for x in h[:3]] + [h[3].int()], 1)
    return s


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        bvhs, rays = [], []
        for verts, index, r in _batch_parts(_generator(seed), case):
            bvhs.append(scion.scion_build_gpu(verts, _layout(case), index))
            rays.append(r)
        batch = scion.Batch(bvhs, rays, params=[_params(case)] * len(bvhs))
        return {"kind": kind, "batch": batch}
    s = dict(_inputs(case, seed), kind=kind)
    if kind != "rebuild":
        s["bvh"] = _build(s["verts"], s["index"], case)
    if kind == "trace":
        s["params"] = _params(case, case["width"] if case["rays"] == "camera" else 0)
        s["query"] = case["query"]
    elif kind == "train":
        s["verts"].requires_grad_(True)
        s["rays"].requires_grad_(True)
        s["grad"] = [x.contiguous() for x in s["grad"].unbind(1)]
    elif kind in ("rebuild", "refit"):
        s["verts"] = _moved(s["verts"])
        s["params"] = _params(case, case["width"])
        s["layout"] = _layout(case)
    return s


def _hits(h):
    f = h.view(torch.float32)
    return {"t": f[:, 0], "u": f[:, 1], "v": f[:, 2], "prim": h[:, 3]}


def run(s):
    kind = s["kind"]
    if kind == "trace":
        if s["query"] == "any":
            return {"occluded": scion.scion_trace_any(s["bvh"], s["rays"], params=s["params"])}
        return _hits(scion.scion_trace_closest(s["bvh"], s["rays"], params=s["params"]))
    if kind == "points":
        return _hits(scion.scion_query_closest_point(s["bvh"], s["points"]))
    if kind == "train":
        t, u, v, prim = scion.trace_fn().apply(s["verts"], s["rays"], s["bvh"])
        gv, gr = torch.autograd.grad([t, u, v], [s["verts"], s["rays"]], s["grad"])
        return {"t": t.detach(), "u": u.detach(), "v": v.detach(), "prim": prim, "verts": gv, "rays": gr}
    if kind == "backward":
        gv, gr = scion.scion_trace_backward(s["bvh"], s["rays"], s["hits"], s["grad"])
        return {"verts": gv, "rays": gr}
    if kind == "batch":
        return list(s["batch"].launch())
    if kind == "rebuild":  # the last frame's tree goes when this frame's is there
        s["bvh"] = scion.scion_build_gpu(s["verts"], s["layout"], s["index"])
    else:
        scion.scion_refit(s["bvh"], s["verts"])
    return _hits(scion.scion_trace_closest(s["bvh"], s["rays"], params=s["params"]))


def work(case):
    """Rays or points and their results once, the triangles that can be hit once (36 bytes of vertices), the
    built or refitted tree once (at least 8 bytes a triangle of compressed boxes, and the leaves); per ray
    one path down a balanced tree (log2 of the triangles; a box test of 12 operations) and one triangle test (40)."""
    kind = case["kind"]
    if kind == "batch":
        sizes = [_batch_sizes(case, k) for k in range(case["scenes"])]
        return {"bytes": sum(48 * n + 36 * min(t, n) for t, n in sizes),
                "flops": sum(n * (40 + 12 * math.log2(t)) for t, n in sizes)}
    t = case["tris"]
    n = case["n"] if "n" in case else case["width"] * case["height"]
    out = 4 if case.get("query") == "any" else 16
    move = n * ((16 if kind == "points" else 32) + out) + 36 * min(t, n)
    flops = n * (40 + 12 * math.log2(max(2, t)))
    verts = 12 * t // 2
    if kind in ("train", "backward"):
        back = n * (16 + 16 + 12 + 32) + 36 * min(t, n) + verts
        fwd = kind == "train"
        return {"bytes": back + (move if fwd else 0), "flops": 60 * n + (flops if fwd else 0)}
    if kind in ("rebuild", "refit"):
        move += verts + 12 * t + 8 * t + (48 if case["prims"] == "direct" else 4) * t
        flops += 30 * t
    return {"bytes": move, "flops": flops}


def tolerance(case):
    # Hits, occlusion flags and closest points are bit for bit those of a fixed sequence of IEEE operations and
    # do not depend on the layout, the tree or the order of the traversal.
    if case["kind"] not in ("train", "backward"):
        return "exact"
    # Gradients: 32-bit sums, in no fixed order, over the rays that hit a vertex's triangles. Measured on the same
    # inputs twice (another order of the sums): rel 4e-8 to 8e-8, largest single value 1.1e-6 of the root mean
    # square; four times that, and as much again for the last bit of another correct solve of the 3x3 systems.
    return {"rel": 8e-7, "max": 1e-5, "differ": 0.0}


# ------------------------------------------------------------------ the same in 64 bits

MOST_PAIRS = 12_000_000_000  # ray-triangle tests that fit in a few seconds


def _brute_hits(rays, tri, any_hit):
    rays, tri = rays.double(), tri.double()
    n, m = rays.shape[0], tri.shape[0]
    bt = torch.full((n,), INF, dtype=torch.float64, device="cuda")
    bu, bv, bi = torch.zeros_like(bt), torch.zeros_like(bt), torch.full((n,), -1, device="cuda")
    step = max(1, (1 << 22) // n)
    for b in range(0, m, step):
        c = tri[b:b + step]
        for a in range(0, n, 1 << 22):
            r = rays[a:a + (1 << 22), None]
            t, u, v, hit = _moeller(r[..., 0:3], r[..., 4:7], r[..., 3], r[..., 7], c[None, :, 0], c[None, :, 1],
                                    c[None, :, 2])
            t, k = torch.where(hit, t, INF).min(1)
            s = slice(a, a + t.shape[0])
            better = t < bt[s]
            bt[s] = torch.where(better, t, bt[s])
            bu[s] = torch.where(better, u.gather(1, k[:, None])[:, 0], bu[s])
            bv[s] = torch.where(better, v.gather(1, k[:, None])[:, 0], bv[s])
            bi[s] = torch.where(better, b + k, bi[s])
    return (bt < INF).int() if any_hit else (bt, bu, bv, bi)


def _brute_points(points, tri):
    """Squared distance to the nearest triangle."""
    p, tri = points[:, :3].double(), tri.double()
    n = p.shape[0]
    best = torch.full((n,), INF, dtype=torch.float64, device="cuda")
    step = max(1, (1 << 22) // n)
    dot = lambda x, y: (x * y).sum(-1)  # noqa: E731
    for b in range(0, tri.shape[0], step):
        c = tri[None, b:b + step]
        e1, e2, s = c[:, :, 1] - c[:, :, 0], c[:, :, 2] - c[:, :, 0], p[:, None] - c[:, :, 0]
        a11, a12, a22, b1, b2 = dot(e1, e1), dot(e1, e2), dot(e2, e2), dot(s, e1), dot(s, e2)
        det = a11 * a22 - a12 * a12
        u, v = (a22 * b1 - a12 * b2) / det, (a11 * b2 - a12 * b1) / det
        inside = (det > 0) & (u >= 0) & (v >= 0) & (u + v <= 1)
        # the foot on the plane where it is inside, otherwise the best of the three edges
        zero = torch.zeros_like(u)
        e3 = e2 - e1
        k = ((dot(s, e3) - dot(e1, e3)) / dot(e3, e3)).clamp(0, 1)
        tries = [(torch.where(inside, u, 0.0), torch.where(inside, v, 0.0)), ((b1 / a11).clamp(0, 1), zero),
                 (zero, (b2 / a22).clamp(0, 1)), (1 - k, k)]
        for x, y in tries:
            r = s - x[..., None] * e1 - y[..., None] * e2
            best = torch.minimum(best, dot(r, r).nan_to_num(INF, INF).amin(1))
    return best


def _gradients(verts, index, rays, hits, grad):
    """Gradients of the vertices and of the rays for the hit triangles, in 64 bits."""
    t, u, v, tri = hits
    m = (tri >= 0).nonzero()[:, 0]
    ids = index.long()[tri[m]] if index is not None else 3 * tri[m, None] + torch.arange(3, device="cuda")
    c, d = verts.double()[ids], rays[m, 4:7].double()
    j = torch.stack([d, c[:, 0] - c[:, 1], c[:, 0] - c[:, 2]], 1)  # the rows of J^T
    g = grad[m].double()
    x, y, z = (torch.linalg.cross(j[:, k], j[:, (k + 1) % 3]) for k in (1, 2, 0))
    lam = (g[:, :1] * x + g[:, 1:2] * y + g[:, 2:] * z) / (j[:, 0] * x).sum(1, keepdim=True)
    weight = torch.stack([1 - u[m] - v[m], u[m], v[m]], 1)
    gv = torch.zeros(verts.shape, dtype=torch.float64, device="cuda")
    gv.index_add_(0, ids.reshape(-1), (weight[:, :, None] * lam[:, None]).reshape(-1, 3))
    gr = torch.zeros((rays.shape[0], 8), dtype=torch.float64, device="cuda")
    gr[m, 0:3], gr[m, 4:7] = -lam, -t[m, None] * lam
    return gv, gr


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":  # the hits come as one record of bits
        return None
    s = _inputs(case, seed)
    verts, index = s["verts"], s["index"]
    named = lambda h: {"t": h[0], "u": h[1], "v": h[2], "prim": None}  # noqa: E731
    if kind == "trace" and case["rays"] != "camera":
        if s["rays"].shape[0] * case["tris"] > MOST_PAIRS:
            return None  # random rays have no order to draw triangles in
        if case["query"] == "any":
            return {"occluded": _brute_hits(s["rays"], _triangles(verts, index), True)}
        return named(_brute_hits(s["rays"], _triangles(verts, index), False))
    if kind == "points":
        if 3 * s["points"].shape[0] * case["tris"] > MOST_PAIRS:
            return None
        # the nearest point often lies on an edge or a corner: whose triangle's weights come back is no number
        return {"t": _brute_points(s["points"], _triangles(verts, index)), "u": None, "v": None, "prim": None}
    if kind in ("rebuild", "refit"):
        verts = _moved(verts)
    if kind == "backward":
        h = s["hits"].view(torch.float32).double()
        gv, gr = _gradients(verts, index, s["rays"], (h[:, 0], h[:, 1], h[:, 2], s["hits"][:, 3].long()), s["grad"])
        return {"verts": gv, "rays": gr}
    hits = _render(verts, index, case["width"], case["height"])
    if kind != "train":
        return named(hits)
    # In a large image a few rays pass so near an edge that 32 bits find the triangle beside it, and where those
    # graze the surface the gradients, which grow with the slope, are another triangle's.
    few = s["rays"].shape[0] <= 1 << 15
    gv, gr = _gradients(verts, index, s["rays"], hits, s["grad"]) if few else (None, None)
    return dict(named(hits), verts=gv, rays=gr)
