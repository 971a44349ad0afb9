"""The workloads that the performance of this framework is measured on.

Every case is work that a program has the library do through ``Context``: frames (selection and
rendering of a composed scene, one or several views, into device or host images), requests to the
server, and the pair sort on its own.  A frame case is a dict with

* ``assets`` x ``leaves``: the library of assets that the program loads once and keeps (synthetic
  3DGS assets of the kind the tests and the benchmark use: leaves on a jittered unit sphere,
  64-Gaussian Morton clusters, a 4-ary moment-matched tree);
* ``instances``, ``scene``: the composed scene, "orbit" (one asset at the origin, a camera at
  ``distance``) or "crowd" (assets strewn over a ground of half width ``extent``, a camera on its walk);
* ``width``, ``height``, ``fov``, ``tau``, ``views``: the image(s) and the pixel tolerance;
* ``fp16``, ``graphs``, ``host``, ``trans``: FP16 colour storage, CUDA-graph frames, the image
  returned in host memory, the final transmittance wanted too.

The instances (rotations, places, scales, assets) and the camera(s) come from the seed; the library
of assets is the same for every seed, as the loaded scene of a running program is.
"""
import collections
import math
import types

import numpy as np
import torch

from paper_2505_06523_gb300 import Context, _native

MAX_LEAVES, MAX_INSTANCES = 1_000_000, 5000


def _frame(name, **kw):
    c = {"name": name, "kind": "frame", "assets": 1, "leaves": 1_000_000, "instances": 1, "scene": "orbit", "distance": 3.0,
         "extent": 100.0, "width": 1920, "height": 1080, "fov": 45.0, "tau": 1.0, "views": 1, "fp16": False, "graphs": False,
         "host": False, "trans": False}
    c.update(kw)
    return c


def listed():
    return [
        # a thumbnail of a small asset: the smallest call, all launches and latency
        _frame("thumbnail", leaves=20_000, width=96, height=80, fov=60.0, distance=2.6, trans=True),
        # one asset in a small viewer window (the tiny workload)
        _frame("viewer 256x256", leaves=100_000, width=256, height=256, fov=60.0),
        # a preview of a composed scene of two assets (the tests' small crowd)
        _frame("small crowd 640x360", assets=2, leaves=100_000, instances=200, scene="crowd", extent=70.0, width=640, height=360),
        # a ragged window over an FP16 asset close by, a wide lens and a fine tolerance
        _frame("ragged 1001x563 fp16", leaves=300_000, width=1001, height=563, fov=90.0, distance=2.2, tau=0.5, fp16=True, trans=True),
        # inspecting one full-size asset: the camera almost inside it, Gaussians that cover many tiles
        _frame("orbit near 1080p", distance=1.5),
        # the same asset far away, the frame handed to the host (an encoder, a GUI toolkit)
        _frame("orbit far 1080p host", distance=50.0, tau=2.0, host=True),
        # the crowd walk in full HD, FP32, one frame at a time: the headline workload
        _frame("crowd 1080p", assets=10, instances=1000, scene="crowd"),
        # the largest composed scene at 4K with a fine tolerance, FP16 colour, as a CUDA graph
        _frame("crowd 5000 4K fp16", assets=10, instances=5000, scene="crowd", width=3840, height=2160, tau=0.5, fp16=True, graphs=True),
        # sixteen views of the crowd in one batch (multi-view capture, offline rendering)
        _frame("crowd 16 views fp16", assets=10, instances=1000, scene="crowd", views=16, tau=2.0, fp16=True, graphs=True),
        # a burst of independent requests to the server, four slots, FP16 colour
        {"name": "serve 8 requests", "kind": "serve", "assets": 10, "leaves": 1_000_000, "requests": 8, "instances": 1000,
         "width": 1280, "height": 720, "tau": 1.0},
        # the sort stage on its own: depth keys of one large frame
        {"name": "sort 20M depth keys", "kind": "sort", "pairs": 20_000_017, "begin": 0, "end": 32, "noalloc": False},
        # the sort of a host that may not allocate: tile ids of a small frame
        {"name": "sort 300k tile ids noalloc", "kind": "sort", "pairs": 300_001, "begin": 0, "end": 13, "noalloc": True},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["one", "one", "crowd", "crowd", "large crowd", "views", "serve", "sort"])
    width = _log(rng, 64, 3840)
    c = _frame("", width=width, height=max(33, int(width * rng.uniform(0.5, 0.8))), tau=round(2.0 ** rng.uniform(-1, 2), 3),
               fp16=rng.random() < 0.5, trans=rng.random() < 0.3, host=rng.random() < 0.2, fov=round(rng.uniform(40.0, 75.0), 1))
    del c["name"]
    if kind == "one":
        c.update(leaves=_log(rng, 20_000, MAX_LEAVES), distance=round(1.5 * (50.0 / 1.5) ** rng.random(), 3), graphs=rng.random() < 0.2)
    elif kind == "crowd":
        c.update(assets=2, leaves=100_000, instances=_log(rng, 20, 2000), scene="crowd", extent=round(rng.uniform(60.0, 100.0), 1))
    elif kind == "large crowd":
        c.update(assets=10, instances=_log(rng, 100, MAX_INSTANCES), scene="crowd", graphs=c["fp16"])
    elif kind == "views":
        c.update(assets=2, leaves=100_000, instances=_log(rng, 20, 400), scene="crowd", extent=70.0, views=rng.randint(2, 16),
                 width=min(width, 1920), height=min(c["height"], 1080), host=False)
    elif kind == "serve":
        return {"kind": "serve", "assets": 2, "leaves": 100_000, "requests": rng.randint(3, 16), "instances": _log(rng, 20, 1000),
                "width": min(width, 1920), "height": min(c["height"], 1080), "tau": c["tau"]}
    else:
        noalloc = rng.random() < 0.4
        begin = rng.choice([0, 0, 0, 3, 8])
        return {"kind": "sort", "pairs": _log(rng, 1000, 1 << 20) if noalloc else _log(rng, 10_000, 64_000_000), "begin": begin,
                "end": rng.randint(begin + 4, 32), "noalloc": noalloc}
    return c


# ------------------------------------------------------------------------------ synthetic assets

def _eigen3(a):
    """Eigenvalues (descending) and eigenvectors (columns, determinant +1) of symmetric (n, 3, 3) matrices, by Jacobi rotations."""
    a, n = a.clone(), a.shape[0]
    v = torch.eye(3, dtype=a.dtype, device=a.device).repeat(n, 1, 1)
    for _ in range(6):
        for p, q in ((0, 1), (0, 2), (1, 2)):
            off = a[:, p, q]
            theta = (a[:, q, q] - a[:, p, p]) / torch.where(off == 0, torch.ones_like(off), 2 * off)
            t = torch.where(theta < 0, -1.0, 1.0) / (theta.abs() + torch.sqrt(theta * theta + 1))
            t = torch.where(off == 0, torch.zeros_like(t), t)
            c = 1 / torch.sqrt(t * t + 1)
            s = t * c
            for m, axis in ((a, 2), (a, 1), (v, 2)):   # columns, then rows of a; columns of v
                x, y = m.select(axis, p).clone(), m.select(axis, q).clone()
                cc, ss = c[:, None], s[:, None]
                m.select(axis, p).copy_(cc * x - ss * y)
                m.select(axis, q).copy_(ss * x + cc * y)
    lam = torch.diagonal(a, dim1=1, dim2=2)
    order = torch.argsort(lam, dim=1, descending=True, stable=True)
    v = torch.gather(v, 2, order[:, None, :].expand(-1, 3, -1))
    det = (torch.cross(v[:, :, 0], v[:, :, 1], dim=1) * v[:, :, 2]).sum(1)
    v[:, :, 2] *= torch.where(det < 0, -1.0, 1.0)[:, None]
    return torch.gather(lam, 1, order), v


def _rotation(q):
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)


def _quaternion(r):
    d = torch.diagonal(r, dim1=1, dim2=2)
    tr = d.sum(1)
    xy, xz, yz = r[:, 1, 0] + r[:, 0, 1], r[:, 0, 2] + r[:, 2, 0], r[:, 2, 1] + r[:, 1, 2]
    wx, wy, wz = r[:, 2, 1] - r[:, 1, 2], r[:, 0, 2] - r[:, 2, 0], r[:, 1, 0] - r[:, 0, 1]
    rows = torch.stack([torch.stack([1 + tr, wx, wy, wz], 1), torch.stack([wx, 1 + 2 * d[:, 0] - tr, xy, xz], 1),
                        torch.stack([wy, xy, 1 + 2 * d[:, 1] - tr, yz], 1), torch.stack([wz, xz, yz, 1 + 2 * d[:, 2] - tr], 1)], 1)
    best = torch.diagonal(rows, dim1=1, dim2=2).argmax(1)
    q = rows[torch.arange(len(best), device=r.device), best]
    return q / q.norm(dim=1, keepdim=True)


def _merge(g):
    """Moment-matched merge of Gaussians 2k and 2k + 1 of a list (an odd last one is kept); g: (mean, log-scale, quaternion, opacity, SH)."""
    n = g[0].shape[0] // 2 * 2
    a, b = [x[0:n:2].double() for x in g], [x[1:n:2].double() for x in g]
    wa, wb = (x[3] * torch.exp(x[1].sum(1)) for x in (a, b))
    ta = (wa / (wa + wb))[:, None]
    tb = 1 - ta
    mean = ta * a[0] + tb * b[0]
    cov = 0
    for t, x in ((ta, a), (tb, b)):
        rot, d = _rotation(x[2]) * torch.exp(x[1])[:, None, :], x[0] - mean
        cov = cov + t[:, :, None] * (rot @ rot.transpose(1, 2) + d[:, :, None] * d[:, None, :])
    lam, vec = _eigen3(cov)
    sh = (ta * a[4].flatten(1) + tb * b[4].flatten(1)).view_as(a[4])
    out = (mean, 0.5 * torch.log(lam.clamp_min(1e-30)), _quaternion(vec), (1 - (1 - a[3]) * (1 - b[3])).clamp_max(0.999), sh)
    return [torch.cat([x.float(), y[n:]]) for x, y in zip(out, g)]


def _leaves(seed, n):
    gen = torch.Generator("cuda").manual_seed(7919 * seed + n)
    normal = lambda *s: torch.randn(*s, generator=gen, device="cuda", dtype=torch.float64)  # noqa: E731
    mean = normal(n, 3)
    mean = mean / mean.norm(dim=1, keepdim=True) + 0.01 * normal(n, 3)
    g = [mean, -4.0 + 0.5 * normal(n, 3), normal(n, 4), torch.sigmoid(normal(n)), 0.3 * normal(n, 16, 3)]
    lo = mean.amin(0)
    cell = ((mean - lo) / (mean.amax(0) - lo) * (2 ** 21 - 1)).long().clamp(0, 2 ** 21 - 1)
    code = torch.zeros(n, dtype=torch.int64, device="cuda")
    for bit in range(21):
        for axis in range(3):
            code |= ((cell[:, axis] >> bit) & 1) << (3 * bit + axis)
    order = torch.argsort(code, stable=True)
    return [x[order].float() for x in g]


def _up32(x):
    r = np.asarray(x, np.float64).astype(np.float32)
    return np.where(r.astype(np.float64) < x, np.nextafter(r, np.float32(np.inf)), r)


def _asset(seed, n):
    """One asset: 64-Gaussian clusters of the leaves in Morton order; a parent of four clusters merges their Gaussians pairwise down to at most 64."""
    levels = [_leaves(seed, n)]
    while levels[-1][0].shape[0] > 64:
        g = levels[-1]
        full = g[0].shape[0] // 256 * 256
        head, tail = [x[:full] for x in g], [x[full:] for x in g]
        if full:
            head = _merge(_merge(head))
        while tail[0].shape[0] > 64:
            tail = _merge(tail)
        levels.append([torch.cat([x, y]) for x, y in zip(head, tail)])
    spheres = []   # of each level's groups of four clusters
    for g in levels:
        p = g[0].double()
        full = p.shape[0] // 256 * 256
        parts = ([p[:full].view(-1, 256, 3)] if full else []) + ([p[full:][None]] if p.shape[0] > full else [])
        got = []
        for q in parts:
            c = q.mean(1).float()
            r = (q - c.double()[:, None]).norm(dim=2).amax(1)
            got.append(np.concatenate([c.cpu().numpy().astype(np.float64), r.cpu().numpy()[:, None]], 1))
        spheres.append(np.concatenate(got))
    for k in range(1, len(levels)):   # each group holds the groups below its members
        below = spheres[k - 1]
        owner = np.arange(len(below)) // 4
        need = np.linalg.norm(spheres[k][owner, :3] - below[:, :3], axis=1) + below[:, 3]
        np.maximum.at(spheres[k][:, 3], owner, need * (1 + 2.0 ** -16))
        spheres[k][:, 3] = _up32(spheres[k][:, 3])
    out = types.SimpleNamespace(gaussians_per_group=256)
    counts = [np.minimum(64, g[0].shape[0] - 64 * np.arange((g[0].shape[0] + 63) // 64)) for g in levels]
    base = np.concatenate([[0], np.cumsum([len(c) for c in counts])])
    out.node_count = np.concatenate(counts).astype(np.uint32)
    out.node_first = (np.cumsum(out.node_count) - out.node_count).astype(np.uint32)
    out.node_level = np.concatenate([np.full(len(c), k) for k, c in enumerate(counts)]).astype(np.uint8)
    out.node_parent = np.concatenate([base[k + 1] + np.arange(len(c)) // 4 if k + 1 < len(counts) else [-1] for k, c in enumerate(counts)]).astype(np.int32)
    own = np.concatenate([s[np.arange(len(c)) // 4] for s, c in zip(spheres, counts)])
    out.own_sphere = np.concatenate([own[:, :3].astype(np.float32), _up32(own[:, 3:])], 1).astype(np.float32)
    out.gpu = [torch.cat([g[i] for g in levels]) for i in range(5)]
    return out


def _on_host(a):
    a.means, a.log_scales, a.quats, a.opacity, a.sh = (x.cpu().numpy() for x in a.gpu)
    a.gpu = None
    return a


# ------------------------------------------------------------------------------ scenes

def _rotations(rng, n):
    q = rng.standard_normal((n, 4))
    w, x, y, z = (q / np.linalg.norm(q, axis=1, keepdims=True)).T
    return np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                     2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                     2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).reshape(n, 3, 3)


def _camera(eye, forward, width, height, fov):
    forward = forward / np.linalg.norm(forward)
    right = np.cross(forward, (0.0, 0.0, 1.0))
    right /= np.linalg.norm(right)
    r = np.stack([right, np.cross(forward, right), forward])
    f = float(np.float32(0.5 * width / math.tan(math.radians(fov) / 2)))
    return types.SimpleNamespace(world_to_cam=np.concatenate([r, (-r @ eye)[:, None]], 1), fx=f, fy=f, cx=width / 2.0, cy=height / 2.0,
                                 width=width, height=height, near=float(np.float32(0.01)))


def _orbit(c, rng):
    e, a = math.radians(rng.uniform(15.0, 45.0)), rng.uniform(0.0, 2 * math.pi)
    eye = c["distance"] * np.array([math.cos(e) * math.cos(a), math.cos(e) * math.sin(a), math.sin(e)])
    inst = types.SimpleNamespace(asset=np.zeros(1, np.uint32), rot=_rotations(rng, 1), trans=np.zeros((1, 3)), scale=np.ones(1))
    return inst, [_camera(eye, -eye, c["width"], c["height"], c["fov"])]


def _crowd_instances(c, rng, n, extent):
    xy = np.empty((0, 2))
    while len(xy) < n:   # clear of the circle that the camera walks
        new = rng.uniform(-extent, extent, (2 * n, 2))
        xy = np.concatenate([xy, new[np.abs(np.linalg.norm(new, axis=1) - 0.6 * extent) >= 3.5]])
    scale = rng.uniform(0.5, 2.0, n)
    return types.SimpleNamespace(asset=rng.integers(0, c["assets"], n).astype(np.uint32), rot=_rotations(rng, n),
                                 trans=np.concatenate([xy[:n], scale[:, None]], 1), scale=scale)


def _walk_camera(t, extent, width, height, fov):
    out, along = np.array([math.cos(t), math.sin(t), 0.0]), np.array([-math.sin(t), math.cos(t), 0.0])
    eye = 0.6 * extent * out + np.array([0.0, 0.0, 1.7])
    return _camera(eye, math.cos(math.radians(20)) * along - math.sin(math.radians(20)) * out, width, height, fov)


def _scene(c, seed):
    rng = np.random.default_rng([seed, 1])
    if c["scene"] == "orbit":
        return _orbit(c, rng)
    inst = _crowd_instances(c, rng, c["instances"], c["extent"])
    t = rng.uniform(0, 2 * math.pi)
    return inst, [_walk_camera(t + 0.02 * v, c["extent"], c["width"], c["height"], c["fov"]) for v in range(c["views"])]


# ------------------------------------------------------------------------------ the calls

_handles = collections.OrderedDict()   # the last few libraries of assets, each with the context that a program keeps for it


def _handle(assets, leaves, fp16, graphs, slots):
    key = (assets, leaves, fp16, graphs, slots)
    if key not in _handles:
        while len(_handles) >= 4:
            _handles.popitem(last=False)
        ctx = Context(0)
        ctx.set_option(_native.V3DG_OPT_ATTR_FP16, int(fp16))
        ctx.set_option(_native.V3DG_OPT_GRAPHS, int(graphs))
        for k in range(assets):
            ctx.load_hierarchy(_on_host(_asset(k, leaves)))
        if slots:
            ctx.server_start(slots)
        _handles[key] = types.SimpleNamespace(ctx=ctx, images={})
    _handles.move_to_end(key)
    return _handles[key]


def _images(h, c):
    """The output images of a program that keeps its own: one set for a library and an image size."""
    shape = ((c["views"],) if c["views"] > 1 else ()) + (c["height"], c["width"])
    key = (shape, c["host"], c["trans"])
    if key not in h.images:
        h.images.clear()
        new = (lambda *s: torch.empty(s, pin_memory=True).numpy()) if c["host"] else (lambda *s: torch.empty(s, device="cuda"))
        h.images[key] = (new(*shape, 3), new(*shape) if c["trans"] else None)
    return h.images[key]


def _keys(c, seed):
    """Depth keys of clusters (64 neighbours at nearly one depth; a few culled), or the ids of the tiles that Gaussians cover, in depth order."""
    gen = torch.Generator("cuda").manual_seed(seed)
    n = c["pairs"]
    if c["end"] >= 24:
        depth = 0.5 + 150 * torch.rand((n + 63) // 64, generator=gen, device="cuda") ** 2
        depth = depth.repeat_interleave(64)[:n] * (1 + 0.01 * torch.rand(n, generator=gen, device="cuda"))
        keys = torch.where(torch.rand(n, generator=gen, device="cuda") < 0.02, -1, depth.view(torch.int32))
    else:
        first = torch.randint(0, 1 << c["end"], ((n + 3) // 4,), generator=gen, device="cuda")
        keys = (first.repeat_interleave(4)[:n] + torch.randint(0, 3, (n,), generator=gen, device="cuda")).to(torch.int32)
    return keys.contiguous()


def prepare(case, seed):
    c = case
    s = types.SimpleNamespace(case=c)
    if c["kind"] == "sort":
        s.keys = _keys(c, seed)
        s.vals = torch.arange(c["pairs"], dtype=torch.int32, device="cuda")
        s.k, s.v = torch.empty_like(s.keys), torch.empty_like(s.vals)
        s.ctx = None if c["noalloc"] else _sorter()
    elif c["kind"] == "serve":
        s.ctx = _handle(c["assets"], c["leaves"], True, True, 4).ctx
        rng = np.random.default_rng([seed, 2])
        s.requests = []
        for k in range(c["requests"]):   # scenes, image sizes and tolerances about the case's own
            n, f = max(1, c["instances"] // (1, 2, 10)[k % 3]), (1.0, 1.5, 1.0, 0.6)[k % 4]
            inst = _crowd_instances(c, rng, n, 100.0)
            cam = _walk_camera(rng.uniform(0, 2 * math.pi), 100.0, int(c["width"] * f), int(c["height"] * f), 45.0)
            s.requests.append((inst, cam, c["tau"] * (1.0, 2.0, 0.5)[k % 3]))
    else:
        # the large FP16 library is also the one that a server shares
        h = _handle(c["assets"], c["leaves"], c["fp16"], c["graphs"], 4 if c["fp16"] and c["graphs"] and c["assets"] > 1 else 0)
        s.ctx, (s.inst, s.cams) = h.ctx, _scene(c, seed)
        s.images = _images(h, c) if c["host"] or c["graphs"] else (None, None)
    return s


_sort_context = []


def _sorter():
    if not _sort_context:
        _sort_context.append(Context(0))
    return _sort_context[0]


def run(state):
    s, c = state, state.case
    if c["kind"] == "sort":
        s.k.copy_(s.keys)
        s.v.copy_(s.vals)
        if c["noalloc"]:
            _native.v3dg_sort_pairs_noalloc(s.k.data_ptr(), s.v.data_ptr(), c["pairs"], c["begin"], c["end"], torch.cuda.current_stream().cuda_stream)
        else:
            s.ctx.sort_pairs(s.k, s.v, c["begin"], c["end"])
        return {"keys": s.k, "vals": s.v}
    if c["kind"] == "serve":
        tickets = [s.ctx.submit(inst, cam, tau) for inst, cam, tau in s.requests]
        images = []
        for t in tickets:
            got = None
            while got is None:
                got = s.ctx.poll(t, 1_000_000)
            images.append(got[1])
        return images
    s.ctx.set_instances(s.inst)
    if c["views"] > 1:
        s.ctx.select_views(s.cams, c["tau"])
    else:
        s.ctx.select(s.cams[0], c["tau"])
    rgb, T = (s.ctx.render_host if c["host"] else s.ctx.render)(*s.images, want_T=c["trans"])
    return {"rgb": rgb, "T": T} if c["trans"] else {"rgb": rgb}


# ------------------------------------------------------------------------------ the work

def _drawn(c, n_assets):
    """About how many distinct Gaussians a frame draws: the cut stays at the leaves until the groups' footprints fall below the tolerance."""
    if c.get("scene") == "orbit":
        x = c["tau"] * c["distance"] * math.sqrt(c["leaves"] / 1e6) * 2318.0 / (0.5 * c["width"] / math.tan(math.radians(c["fov"]) / 2))
        return c["leaves"] * min(1.0, 30.0 / x) ** 1.2 * (0.25 if c["distance"] < 2.0 else 1.0)
    in_view = c["instances"] / 8
    return c["leaves"] * n_assets * (1 - (1 - 1 / n_assets) ** in_view)


def work(case):
    """Bytes: the attributes of the drawn Gaussians and the instances once, the image once.  Flops: about 250 for each projected Gaussian, 10 for each of the
    about 60 that a pixel blends."""
    c = case
    if c["kind"] == "sort":
        return {"bytes": 16 * c["pairs"], "flops": 0}
    frames = c["requests"] if c["kind"] == "serve" else c["views"]
    pixels = c["width"] * c["height"] * frames
    attr = 138 if c.get("fp16", True) else 236
    distinct = _drawn(c, c["assets"])
    visible = distinct if c.get("scene") == "orbit" else 63.0 * c["instances"] * c["leaves"] / 1e3 / math.sqrt(max(c["tau"], 0.25))
    shared = frames if c["kind"] == "serve" else 1   # views of one batch read the attributes once
    return {"bytes": attr * distinct * shared + 104 * c["instances"] * shared + (16 if c.get("trans") else 12) * pixels,
            "flops": 250 * visible * frames + 600 * pixels}


# ------------------------------------------------------------------------------ the same in 64 bits

def _cut_and_cull(a, M, s, tau, cam):
    """(instance, node) of the cut of instances with transforms M (n, 3, 4) of asset `a`, without clusters that are surely out of view."""
    own = torch.from_numpy(a.own_sphere).cuda().double()
    level, parent = torch.from_numpy(a.node_level).cuda(), torch.from_numpy(a.node_parent).cuda().long()
    z = own[:, :3] @ M[:, 2, :3].T + M[:, 2, 3]
    r = own[:, 3:] * s
    F = torch.where(z.abs() <= r, math.inf, math.pi * cam.fx * cam.fy * r * r / (z * z))
    own_ok = (level == 0)[:, None] | (F <= tau)
    par_out = (parent < 0)[:, None] | (F[parent.clamp_min(0)] > tau)
    count = torch.from_numpy(a.node_count.astype(np.int64)).cuda()
    first = torch.from_numpy(a.node_first.astype(np.int64)).cuda()
    index = (first[:, None] + torch.arange(64, device="cuda")).clamp_max(a.gpu[0].shape[0] - 1)
    valid = torch.arange(64, device="cuda") < count[:, None]
    p = a.gpu[0].double()[index]
    centre = (p * valid[:, :, None]).sum(1) / count[:, None]
    radius = ((p - centre[:, None]).norm(dim=2) * valid).amax(1)
    sigma = (torch.exp(a.gpu[1].double().amax(1))[index] * valid).amax(1)
    view = torch.einsum("irc,nc->nir", M[:, :, :3], centre) + M[:, :, 3]
    reach = radius[:, None] * s + 0.05
    far = view[:, :, 2] + reach < cam.near
    for axis, half, f in ((0, cam.width / 2 + 2, cam.fx), (1, cam.height / 2 + 2, cam.fy)):
        slope = half / f   # 3.33 sigma is where alpha falls below 1/255; the Jacobian's clamp lies 1.3 half images out
        far |= view[:, :, axis].abs() - reach - 3.4 * sigma[:, None] * s * math.sqrt(1 + (1.3 * slope) ** 2) > slope * (view[:, :, 2] + reach).clamp_min(0)
    node, inst = torch.nonzero(own_ok & par_out & ~far, as_tuple=True)
    return node, inst, index, valid


def _project(a, node, inst, index, valid, M, cam_a, cam, gid0, fp16):
    """Visible Gaussians of (instance, node) pairs of one asset: their float32 depth keys, ids and (u, v, conic, opacity, rgb, box), in 64 bits."""
    keep = valid[node]
    g = index[node][keep]
    i = inst[:, None].expand(-1, 64)[keep]
    mean32 = a.gpu[0][g]
    mean, ls, q, o, sh = (x[g].double() for x in a.gpu)
    if fp16:
        o, sh = a.gpu[3][g].half().double(), a.gpu[4][g].half().double()
    m32 = M.float()[i, 2]
    z32 = ((m32[:, 0] * mean32[:, 0] + m32[:, 1] * mean32[:, 1]) + m32[:, 2] * mean32[:, 2]) + m32[:, 3]
    A = M[i]
    t = (A[:, :, :3] @ mean[:, :, None])[:, :, 0] + A[:, :, 3]
    x, y, z = t.unbind(1)
    limx, limy = 1.3 * cam.width / 2 / cam.fx, 1.3 * cam.height / 2 / cam.fy
    L = (A[:, :, :3] @ _rotation(q)) * torch.exp(ls)[:, None, :]
    cx, cy = (x / z).clamp(-limx, limx), (y / z).clamp(-limy, limy)
    tx = cam.fx / z[:, None] * (L[:, 0] - cx[:, None] * L[:, 2])
    ty = cam.fy / z[:, None] * (L[:, 1] - cy[:, None] * L[:, 2])
    ca, cb, cc = (tx * tx).sum(1), (tx * ty).sum(1), (ty * ty).sum(1)
    det = torch.cross(tx, ty, dim=1).square().sum(1)
    u, v = cam.fx * x / z + cam.cx, cam.fy * y / z + cam.cy
    kq = 2 * torch.log(255 * o)
    hx, hy = torch.sqrt((kq * ca).clamp_min(0)), torch.sqrt((kq * cc).clamp_min(0))
    x0, x1 = torch.ceil(u - hx - 0.5).clamp_min(0), torch.floor(u + hx - 0.5).clamp_max(cam.width - 1)
    y0, y1 = torch.ceil(v - hy - 0.5).clamp_min(0), torch.floor(v + hy - 0.5).clamp_max(cam.height - 1)
    vis = (z32 >= cam.near) & (o >= 1 / 255) & (det > 0) & (x0 <= x1) & (y0 <= y1)
    d = mean - cam_a[i]
    dx, dy, dz = (d / d.norm(dim=1, keepdim=True)).unbind(1)
    xx, yy, zz, r = dx * dx, dy * dy, dz * dz, lambda k: math.sqrt(k / math.pi)
    Y = torch.stack([torch.full_like(dx, 0.5 * r(1)), -r(0.75) * dy, r(0.75) * dz, -r(0.75) * dx,
                     0.5 * r(15) * dx * dy, -0.5 * r(15) * dy * dz, 0.25 * r(5) * (3 * zz - 1), -0.5 * r(15) * dx * dz, 0.25 * r(15) * (xx - yy),
                     -0.25 * r(17.5) * dy * (3 * xx - yy), 0.5 * r(105) * dx * dy * dz, -0.25 * r(10.5) * dy * (5 * zz - 1),
                     0.25 * r(7) * dz * (5 * zz - 3), -0.25 * r(10.5) * dx * (5 * zz - 1), 0.25 * r(105) * dz * (xx - yy),
                     -0.25 * r(17.5) * dx * (xx - 3 * yy)], 1)
    rgb = ((Y[:, :, None] * sh).sum(1) + 0.5).clamp_min(0)
    rec = torch.stack([u, v, cc / det, -cb / det, ca / det, o, rgb[:, 0], rgb[:, 1], rgb[:, 2], x0, x1, y0, y1], 1)
    return z32[vis], (gid0[i] + g)[vis], rec[vis]


def _blend(rec, width, height):
    """Front-to-back blending of depth-ordered Gaussians, a chunk of them at a time."""
    n_px = width * height
    C, T = torch.zeros(n_px, 3, dtype=torch.float64, device="cuda"), torch.ones(n_px, dtype=torch.float64, device="cuda")
    done = torch.zeros(n_px, dtype=torch.bool, device="cuda")
    box = rec[:, 9:13].long()
    w = box[:, 1] - box[:, 0] + 1
    ends = torch.cumsum(w * (box[:, 3] - box[:, 2] + 1), 0).cpu()
    a, n = 0, rec.shape[0]
    while a < n:
        start = int(ends[a - 1]) if a else 0
        b = max(a + 1, int(torch.searchsorted(ends, start + 40_000_000)))
        R, B, W = rec[a:b], box[a:b], w[a:b]
        area = W * (B[:, 3] - B[:, 2] + 1)
        owner = torch.repeat_interleave(torch.arange(b - a, device="cuda"), area)
        k = torch.arange(len(owner), device="cuda") - (torch.cumsum(area, 0) - area)[owner]
        px, py = B[:, 0][owner] + k % W[owner], B[:, 2][owner] + k // W[owner]
        pix = py * width + px
        live = ~done[pix]
        owner, px, py, pix = owner[live], px[live], py[live], pix[live]
        dx, dy = px + 0.5 - R[:, 0][owner], py + 0.5 - R[:, 1][owner]
        power = R[:, 2][owner] * dx * dx + 2 * R[:, 3][owner] * dx * dy + R[:, 4][owner] * dy * dy
        alpha = (R[:, 5][owner] * torch.exp(-0.5 * power)).clamp_max(0.999)
        hit = alpha >= 1 / 255
        owner, pix, alpha = owner[hit], pix[hit], alpha[hit]
        pix, order = torch.sort(pix, stable=True)
        owner, alpha = owner[order], alpha[order]
        if len(pix):
            logs = torch.log1p(-alpha)
            cum = torch.cumsum(logs, 0)
            new = torch.ones_like(pix, dtype=torch.bool)
            new[1:] = pix[1:] != pix[:-1]
            seg = torch.cumsum(new, 0) - 1
            base = (cum - logs)[new][seg]
            before = T[pix] * torch.exp(cum - logs - base)
            after = before * (1 - alpha)
            ok = after >= 1e-4
            C.index_add_(0, pix[ok], (alpha * before)[ok][:, None] * R[:, 6:9][owner[ok]])
            done[pix[~ok]] = True
            T.scatter_reduce_(0, pix[ok], after[ok], "amin")
        a = b
    return C.view(height, width, 3), T.view(height, width)


def _exact_view(c, inst, cam, library):
    W = cam.world_to_cam
    M = np.concatenate([inst.scale[:, None, None] * (W[:, :3] @ inst.rot), ((W[:, :3] @ inst.trans.T).T + W[:, 3])[:, :, None]], 2)
    eye = -W[:, :3].T @ W[:, 3]
    cam_a = np.einsum("nji,nj->ni", inst.rot, eye - inst.trans) / inst.scale[:, None]
    tau = float(np.float32(256 * c["tau"] * c["tau"]))
    parts = []
    for k, a in enumerate(library):
        mine = np.nonzero(inst.asset == k)[0]
        for block in np.array_split(mine, max(1, len(mine) // 32)) if len(mine) else []:
            Mb, sb = torch.from_numpy(M[block]).cuda(), torch.from_numpy(inst.scale[block]).cuda()
            node, i, index, valid = _cut_and_cull(a, Mb, sb, tau, cam)
            gid0 = torch.from_numpy(block).cuda() << 32
            for part in torch.split(torch.arange(len(node), device="cuda"), 8192):
                parts.append(_project(a, node[part], i[part], index, valid, Mb, torch.from_numpy(cam_a[block]).cuda(), cam, gid0, c["fp16"]))
    if not any(len(p[0]) for p in parts):
        return (torch.zeros(c["height"], c["width"], 3, dtype=torch.float64, device="cuda"),
                torch.ones(c["height"], c["width"], dtype=torch.float64, device="cuda"))
    key, gid, rec = (torch.cat(x) for x in zip(*parts))
    order = torch.argsort(gid, stable=True)
    order = order[torch.argsort(key[order], stable=True)]
    return _blend(rec[order], c["width"], c["height"])


def exact(case, seed):
    c = case
    if c["kind"] != "frame" or c["views"] * c["instances"] * c["leaves"] > 4e7 or c["width"] > 2000:
        return None   # whole numbers, or too long
    inst, cams = _scene(c, seed)
    library = [_asset(k, c["leaves"]) for k in range(c["assets"])]
    rgb, T = (torch.stack(x) if c["views"] > 1 else x[0] for x in zip(*(_exact_view(c, inst, cam, library) for cam in cams)))
    return {"rgb": rgb, "T": T} if c["trans"] else {"rgb": rgb}
