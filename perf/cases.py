"""What this framework's time is measured on: calls a user's program makes, over the sizes and options it
makes them with.

A case is a dict of plain values.  Its ``kind`` says which public entry points it goes through:

  frame    F.atlas_frame, one view, launched eagerly (the call of the README)
  path     one graph captured from F.atlas_frame_dev_matrix, replayed after the next camera was copied in
  batch    F.atlas_batch, many views on lanes
  plan     F.BatchPlan.launch, many views in one launch
  serve    F.Server: one request of every session submitted, polled until all are done
  pack     F.fa_pack on a set of boxes
  vis      F.fa_visibility alone
  charts   F.fa_chartify alone, on a caller's visible bits
  uv       F.fa_parameterize and F.fa_uv, on a caller's charts and placements

Scenes are the framework's workloads (heightfield patches, floors of instanced patches, displaced
icospheres), made on the GPU from the seed; cameras come from the framework's scene module.  Sizes depend on
the case alone, positions, noise and cameras on the seed.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2502_17712_gb300 import fastatlas as F
from paper_2502_17712_gb300 import scenes as S

RESOLUTIONS = ((640, 360), (1280, 720), (1920, 1080), (2560, 1440))
FIELDS = ("vt", "tri_chart", "vert_chart", "root", "bbox", "fa", "fb", "rot", "count", "order", "place", "result",
          "uv", "affine", "partial")


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # the smallest call: one 64 x 64 heightfield patch in a small view; launches and latency
        dict(name="frame_small", kind="frame", scene="floor", parts=1, detail=64, width=480, height=270, ratio=1.0,
             atlas_log2=10, mode=0, flags=0, extras=False),
        # the headline frame: 4.1M triangles of 200 icospheres, 1080p into a 2048^2 atlas
        dict(name="frame_spheres_4m", kind="frame", scene="spheres", parts=200, detail=5, width=1920, height=1080,
             ratio=1.0, atlas_log2=11, mode=0, flags=0, extras=False),
        # every option at once on a mid-size scene and an odd window: vertex charts, conservative marking,
        # frustum-clipped boxes, partial bits, vertex charts out
        dict(name="frame_options", kind="frame", scene="spheres", parts=31, detail=4, width=1367, height=769, ratio=2.0,
             atlas_log2=12, mode=1, flags=3, extras=True),
        # an ordinary view of an ordinary level: a floor of 60 overlapping patches at 1080p
        dict(name="frame_floor", kind="frame", scene="floor", parts=60, detail=64, width=1920, height=1080, ratio=1.0,
             atlas_log2=11, mode=0, flags=0, extras=False),
        # a frame of a camera path: the heightfield at 1080p, one captured graph, the camera copied in
        dict(name="path_1080p", kind="path", detail=64, width=1920, height=1080, ratio=1.0, atlas_log2=11),
        # many clients' views in one call, 50 to 400 patches, mixed windows and atlases
        dict(name="batch_16_views", kind="batch", views=16, least=50, most=400, detail=64, lanes=8),
        # the same kind of batch as one launch of the persistent kernel
        dict(name="plan_8_views", kind="plan", views=8, least=20, most=120, detail=64, lanes=8),
        # serving: eight sessions ask for a view at once
        dict(name="serve_8_sessions", kind="serve", sessions=8, least=25, most=100, detail=5, slots=4),
        # the packer alone: a few boxes, and more boxes than any frame here has
        dict(name="pack_1k", kind="pack", boxes=1000, capacity=16384, atlas_log2=12, scales=64, mean=12.0),
        dict(name="pack_100k", kind="pack", boxes=100000, capacity=131072, atlas_log2=12, scales=64, mean=6.0),
        # charts of a caller's visible set (vertex mode), on a mesh of a million triangles
        dict(name="charts_vertex_1m", kind="charts", parts=128, detail=64, mode=1),
        # boxes and texture coordinates of a caller's charts
        dict(name="uv_300k", kind="uv", parts=37, detail=64, rows=9, width=1920, height=1080, ratio=1.0, atlas_log2=11),
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(("frame", "frame", "frame", "frame", "path", "batch", "plan", "serve", "pack", "pack", "vis",
                       "charts", "uv"))
    c = dict(kind=kind)
    if kind in ("frame", "vis", "path", "uv"):
        c.update(width=_log(rng, 320, 2560), height=_log(rng, 200, 1440))
    if kind in ("frame", "vis"):
        if rng.random() < 0.5:
            detail = rng.choice((3, 4, 5))
            c.update(scene="spheres", parts=_log(rng, 4, {3: 800, 4: 400, 5: 200}[detail]), detail=detail)
        else:
            detail = rng.choice((17, 33, 64, 100))
            c.update(scene="floor", parts=_log(rng, 1, 200 * 63 * 63 // (detail * detail)), detail=detail)
    if kind == "frame":
        opt = rng.random() < 0.3
        c.update(ratio=rng.choice((0.5, 1.0, 2.0)), atlas_log2=rng.choice((11, 12)), mode=1 if rng.random() < 0.3 else 0,
                 flags=rng.choice((1, 2, 3)) if opt else 0, extras=opt)
    elif kind == "path":
        c.update(detail=rng.randint(24, 160), ratio=rng.choice((0.5, 1.0)), atlas_log2=rng.choice((11, 12)))
    elif kind == "batch":
        c.update(views=rng.randint(2, 16), least=rng.randint(5, 50), most=rng.randint(60, 300), detail=64,
                 lanes=rng.choice((2, 4, 8)))
    elif kind == "plan":
        c.update(views=rng.randint(2, 8), least=rng.randint(2, 20), most=rng.randint(30, 120), detail=64,
                 lanes=rng.choice((2, 4, 8)))
    elif kind == "serve":
        c.update(sessions=rng.randint(2, 8), least=rng.randint(4, 25), most=rng.randint(30, 100), detail=5,
                 slots=rng.choice((1, 2, 4)))
    elif kind == "pack":
        n = _log(rng, 16, 100000)
        log2 = rng.choice((11, 12))
        c.update(boxes=n, capacity=max(1024, 1 << (n - 1).bit_length()), atlas_log2=log2, scales=rng.choice((16, 64)),
                 mean=round(min(24.0, max(2.0, 0.45 * 2 ** log2 / math.sqrt(n))), 2))
    elif kind == "vis":
        c.update(flags=rng.choice((0, 2)))
    elif kind == "charts":
        c.update(parts=_log(rng, 1, 256), detail=rng.choice((33, 64)), mode=rng.randint(0, 1))
    elif kind == "uv":
        c.update(parts=_log(rng, 1, 128), detail=rng.choice((33, 64)), rows=rng.randint(1, 20),
                 ratio=rng.choice((0.5, 1.0, 2.0)), atlas_log2=rng.choice((11, 12)))
    return c


# ------------------------------------------------------------------ scenes, on the GPU

def _gen(*key):
    s = 0
    for k in key:
        s = (s * 1000003 + int(k) + 12345) % (1 << 62)
    return torch.Generator(device="cuda").manual_seed(s)


@functools.lru_cache(maxsize=None)
def _grid(n):
    """The n x n patch's plane coordinates and index triples (host)."""
    sc = S.grid_scene(0, n)
    return sc.pos[:, :2].copy(), sc.idx.astype(np.int64)


@functools.lru_cache(maxsize=None)
def _sphere(level):
    v, f = S.icosphere(level)
    return v, f


def _instances(f, parts, nv):
    """Index triples of `parts` copies of a mesh of nv vertices, one after the other."""
    f = torch.as_tensor(f, device="cuda")
    step = torch.arange(parts, device="cuda").view(-1, 1, 1) * nv
    return (f.unsqueeze(0) + step).reshape(-1, 3).to(torch.int32).contiguous()


def _floor(seed, parts, n, half=6.0):
    """`parts` heightfield patches, rotated about z, scaled 0.5 to 1.5 and spread over a floor (one: as it is)."""
    xy, f = _grid(n)
    g = _gen(seed, 1)
    xy = torch.as_tensor(xy, device="cuda", dtype=torch.float64)
    u = lambda *s: torch.rand(*s, generator=g, device="cuda", dtype=torch.float64)  # noqa: E731
    z = 0.2 * torch.sin(3.0 * xy[:, 0]) * torch.cos(2.0 * xy[:, 1]) + (u(parts, xy.shape[0]) * 0.04 - 0.02)
    p = torch.cat([xy.unsqueeze(0).expand(parts, -1, -1), z.unsqueeze(2)], 2)
    if parts > 1:
        a, scale = u(parts, 1) * 2 * math.pi, (0.5 + u(parts, 1, 1))
        c, s = torch.cos(a), torch.sin(a)
        move = (u(parts, 1, 3) * 2 - 1) * torch.tensor([half, half, 0.3], device="cuda", dtype=torch.float64)
        p = torch.stack([c * p[..., 0] - s * p[..., 1], s * p[..., 0] + c * p[..., 1], p[..., 2]], 2) * scale + move
    return p.reshape(-1, 3).float().contiguous(), _instances(f, parts, xy.shape[0])


def _half(parts):
    """Half the side of the box the spheres are placed in: 200 of them in a 50^3 box, fewer in a smaller one."""
    return max(6.0, 25.0 * (parts / 200) ** (1 / 3))


def _spheres(seed, parts, level):
    """`parts` icospheres displaced by four octaves of lattice value noise, rotated, scaled 0.5 to 2 and placed
    in a box."""
    half = _half(parts)
    v, f = _sphere(level)
    g = _gen(seed, 2)
    v = torch.as_tensor(v, device="cuda", dtype=torch.float64)
    u = lambda *s: torch.rand(*s, generator=g, device="cuda", dtype=torch.float64)  # noqa: E731
    table, side = u(1 << 18) * 2 - 1, 64
    off = u(parts, 1, 3) * side
    disp = torch.ones(parts, v.shape[0], device="cuda", dtype=torch.float64)
    amp, freq = 0.1, 3.0
    for _ in range(4):
        q = v.unsqueeze(0) * freq + off
        i = torch.floor(q)
        w = q - i
        w = w * w * (3 - 2 * w)
        i = i.to(torch.int64)
        for corner in range(8):
            d = [(corner >> k) & 1 for k in range(3)]
            at = [(i[..., k] + d[k]) % side for k in range(3)]
            wt = [w[..., k] if d[k] else 1 - w[..., k] for k in range(3)]
            disp += amp * wt[0] * wt[1] * wt[2] * table[(at[0] * side + at[1]) * side + at[2]]
        amp, freq = amp * 0.5, freq * 2
    q = torch.randn(parts, 4, generator=g, device="cuda", dtype=torch.float64)
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    R = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
                     2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
                     2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    p = (v.unsqueeze(0) * disp.unsqueeze(2)) @ R.transpose(1, 2) * (0.5 + 1.5 * u(parts, 1, 1))
    p = p + (u(parts, 1, 3) * 2 - 1) * 0.96 * half
    return p.reshape(-1, 3).float().contiguous(), _instances(f, parts, v.shape[0])


def _scene(case, seed):
    if case["scene"] == "floor":
        return _floor(seed, case["parts"], case["detail"])
    return _spheres(seed, case["parts"], case["detail"])


def _camera(case, seed):
    W, H = case["width"], case["height"]
    if case["scene"] == "spheres":
        return S.box_camera(seed, W, H, half=_half(case["parts"]))
    return S.hemisphere_camera(seed, W, H, radius=3.0 if case["parts"] == 1 else 10.0)


def _sizes(scene, parts, detail):
    """(T, V) of a scene."""
    if scene == "floor":
        return 2 * (detail - 1) ** 2 * parts, detail * detail * parts
    return 20 * 4 ** detail * parts, (10 * 4 ** detail + 2) * parts


def _frame_buffers(sizes, max_charts, vert_chart=False, partial=False):
    """Output buffers of several views, the views' parts of one field one after the other in one tensor, each at
    a 256-byte boundary: (one FrameBuffers per view, {field: tensor})."""
    shapes = [F.FrameBuffers.allocate(32, 32, 1, vert_chart=True, partial=True)]
    lens = dict(vt=lambda T, V: (T + 31) // 32, tri_chart=lambda T, V: T, vert_chart=lambda T, V: V,
                uv=lambda T, V: T * 6, partial=lambda T, V: (T + 31) // 32, count=lambda T, V: 1, result=lambda T, V: 5)
    tail = dict(bbox=4, place=4, affine=6)
    whole, views = {}, [dict() for _ in sizes]
    for name in FIELDS:
        if (name == "vert_chart" and not vert_chart) or (name == "partial" and not partial):
            for v in views:
                v[name] = None
            continue
        n = [lens[name](T, V) if name in lens else max_charts * tail.get(name, 1) for T, V in sizes]
        at = np.concatenate([[0], np.cumsum([(x + 255) // 256 * 256 for x in n])])
        dtype = getattr(shapes[0], name).dtype
        whole[name] = torch.zeros(int(at[-1]), dtype=dtype, device="cuda")
        if name == "uv":
            whole[name].fill_(float("nan"))
        for v, x, a, (T, V) in zip(views, n, at, sizes):
            t = whole[name][int(a):int(a) + x]
            v[name] = t.view(T, 3, 2) if name == "uv" else t.view(-1, tail[name]) if name in tail else t
    return [F.FrameBuffers(**v) for v in views], whole


# ------------------------------------------------------------------ prepare and run, by kind

def _prepare_frame(case, seed):
    pos, idx = _scene(case, seed)
    T, V = idx.shape[0], pos.shape[0]
    charts = 1 << 17 if T > 200000 else 1 << 15
    ctx = F.Context(max_tris=T, max_verts=V, max_charts=charts, max_width=case["width"], max_height=case["height"],
                    max_atlas_log2=case["atlas_log2"])
    mesh = F.Mesh(ctx, pos, idx)
    (bufs,), out = _frame_buffers([(T, V)], charts, vert_chart=case["extras"], partial=case["extras"])
    return dict(ctx=ctx, mesh=mesh, bufs=bufs, M=_camera(case, seed), out=out)


def _run_frame(case, s):
    F.atlas_frame(s["ctx"], s["mesh"], s["bufs"], s["M"], case["width"], case["height"], case["ratio"],
                  case["atlas_log2"], chart_mode=case["mode"], flags=case["flags"])
    return s["out"]


def _prepare_path(case, seed):
    pos, idx = _floor(seed, 1, case["detail"])
    T, V = idx.shape[0], pos.shape[0]
    W, H = case["width"], case["height"]
    ctx = F.Context(max_tris=T, max_verts=V, max_charts=1 << 14, max_width=W, max_height=H,
                    max_atlas_log2=case["atlas_log2"])
    mesh = F.Mesh(ctx, pos, idx)
    (bufs,), out = _frame_buffers([(T, V)], 1 << 14)
    cams = np.stack([np.asarray(m, np.float32).reshape(16) for m in S.spline_cameras(seed, 8, W, H)])
    host = torch.from_numpy(cams[seed % 8].copy()).pin_memory()
    dm = torch.zeros(16, device="cuda")
    dm.copy_(host)

    def frame():
        F.atlas_frame_dev_matrix(ctx, mesh, bufs, dm, W, H, case["ratio"], case["atlas_log2"])

    frame()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        frame()
    return dict(graph=graph, dm=dm, host=host, out=out, keep=(ctx, mesh, bufs))


def _run_path(case, s):
    s["dm"].copy_(s["host"], non_blocking=True)
    s["graph"].replay()
    return s["out"]


def _views(case):
    """Patches, window and atlas of each view of a batch."""
    n = case["views"]
    for i in range(n):
        parts = case["least"] + (case["most"] - case["least"]) * i // max(1, n - 1)
        W, H = RESOLUTIONS[(i * 3 + 2) % 4]
        yield parts, W, H, (11, 12, 11)[i % 3]


def _prepare_batch(case, seed):
    views = list(_views(case))
    sizes = [_sizes("floor", parts, case["detail"]) for parts, _, _, _ in views]
    batch = F.Batch(case["lanes"], max_tris=max(t for t, _ in sizes), max_verts=max(v for _, v in sizes),
                    max_charts=1 << 16, max_width=2560, max_height=1440, max_atlas_log2=12)
    batch.set_schedule(case["lanes"], F.FA_BATCH_LONGEST_FIRST)
    meshes, params = [], []
    for i, (parts, W, H, log2) in enumerate(views):
        pos, idx = _floor(seed * 131 + i, parts, case["detail"])
        meshes.append(F.BatchMesh(batch, pos, idx))
        M = S.hemisphere_camera(seed * 131 + i, W, H, radius=3.0 if parts == 1 else 10.0)
        params.append(F.frame_params(M, W, H, 1.0, log2))
    bufs, out = _frame_buffers(sizes, 1 << 16)
    s = dict(batch=batch, meshes=meshes, params=params, bufs=bufs, out=out)
    if case["kind"] == "plan":
        s["plan"] = F.BatchPlan(batch, meshes, params, bufs)
    return s


def _run_batch(case, s):
    F.atlas_batch(s["batch"], s["meshes"], s["params"], s["bufs"])
    return s["out"]


def _run_plan(case, s):
    s["plan"].launch()
    return s["out"]


def _clients(case):
    """Spheres, window and atlas of each session."""
    n = case["sessions"]
    for i in range(n):
        parts = case["least"] + (case["most"] - case["least"]) * i // max(1, n - 1)
        W, H = RESOLUTIONS[1 + i % 3]
        yield parts, W, H, 11 + i % 2


def _prepare_serve(case, seed):
    clients = list(_clients(case))
    sizes = [_sizes("spheres", parts, case["detail"]) for parts, _, _, _ in clients]
    server = F.Server(case["slots"], 64 << 30, max_tris=max(t for t, _ in sizes), max_verts=max(v for _, v in sizes),
                      max_charts=1 << 17, max_width=2560, max_height=1440, max_atlas_log2=12)
    bufs, out = _frame_buffers(sizes, 1 << 17)
    asks = []
    for i, (parts, W, H, log2) in enumerate(clients):
        pos, idx = _spheres(seed * 131 + i, parts, case["detail"])
        sid = server.open_session(pos, idx, bufs[i])
        asks.append((sid, F.frame_params(S.box_camera(seed * 131 + i, W, H, half=_half(parts)), W, H, 1.0, log2)))
    torch.cuda.synchronize()  # the slots' streams are the server's own
    return dict(server=server, asks=asks, bufs=bufs, out=out)


def _run_serve(case, s):
    server, left = s["server"], len(s["asks"])
    for sid, params in s["asks"]:
        server.submit(sid, params)
    while left:
        left -= len(server.poll())
    return s["out"]


def _prepare_pack(case, seed):
    n = case["boxes"]
    g = _gen(seed, 3)
    side = torch.exp(torch.randn(n, 2, generator=g, device="cuda", dtype=torch.float64) + math.log(case["mean"]))
    q = torch.ceil(side.clamp(0.25, 1024.0) * 256.0).to(torch.int32)
    fa, fb = q.amin(1).contiguous(), q.amax(1).contiguous()
    ctx = F.Context(max_tris=1024, max_verts=1024, max_charts=case["capacity"], max_width=64, max_height=64,
                    max_atlas_log2=case["atlas_log2"])
    i32 = dict(dtype=torch.int32, device="cuda")
    return dict(ctx=ctx, fa=fa, fb=fb, count=torch.tensor([n], **i32), order=torch.zeros(n, **i32),
                place=torch.zeros(n, 4, **i32), res=torch.zeros(5, **i32))


def _run_pack(case, s):
    F.fa_pack(s["ctx"].handle, s["fa"], s["fb"], s["count"], case["atlas_log2"], case["scales"], F.FA_SELECT_EFFECTIVE,
              s["order"], s["place"], s["res"])
    return [s["order"], s["place"], s["res"]]


def _prepare_vis(case, seed):
    pos, idx = _scene(case, seed)
    ctx = F.Context(max_tris=idx.shape[0], max_verts=pos.shape[0], max_charts=1024, max_width=case["width"],
                    max_height=case["height"])
    return dict(ctx=ctx, mesh=F.Mesh(ctx, pos, idx), M=_camera(case, seed),
                vt=torch.zeros((idx.shape[0] + 31) // 32, dtype=torch.int32, device="cuda"))


def _run_vis(case, s):
    F.fa_visibility(s["ctx"].handle, s["mesh"].handle, s["M"], case["width"], case["height"], s["vt"],
                    flags=case["flags"])
    return s["vt"]


def _charts_struct(C, **more):
    i32 = dict(dtype=torch.int32, device="cuda")
    t = dict(root=torch.zeros(C, **i32), bbox=torch.zeros(C, 4, device="cuda"), fa=torch.zeros(C, **i32),
             fb=torch.zeros(C, **i32), rot=torch.zeros(C, dtype=torch.uint8, device="cuda"),
             count=torch.zeros(1, **i32))
    t.update(more)
    return t, F.fa_charts(*(t[k].data_ptr() for k in ("root", "bbox", "fa", "fb", "rot", "count")))


def _prepare_charts(case, seed):
    pos, idx = _floor(seed, case["parts"], case["detail"])
    T, V, n = idx.shape[0], pos.shape[0], case["detail"]
    # visible: blobs of a smooth field over each patch, minus some single triangles
    g = _gen(seed, 4)
    u = lambda *s: torch.rand(*s, generator=g, device="cuda")  # noqa: E731
    quad = torch.arange((n - 1) * (n - 1), device="cuda")
    x, y = (quad % (n - 1)).float() / n, (quad // (n - 1)).float() / n
    f = sum(torch.sin(x * (6 + 20 * u(case["parts"], 1)) + y * (6 + 20 * u(case["parts"], 1)) + 7 * u(case["parts"], 1))
            for _ in range(3))
    seen = (f > 0.6).repeat_interleave(2, dim=1).reshape(-1) & (u(T) > 0.03)
    bits = torch.zeros((T + 31) // 32 * 32, dtype=torch.int64, device="cuda")
    bits[:T] = seen
    words = (bits.view(-1, 32) << torch.arange(32, device="cuda")).sum(1)
    vt = torch.where(words >= 1 << 31, words - (1 << 32), words).to(torch.int32)
    ctx = F.Context(max_tris=T, max_verts=V, max_charts=T, max_width=64, max_height=64)
    t, charts = _charts_struct(T)
    i32 = dict(dtype=torch.int32, device="cuda")
    return dict(ctx=ctx, mesh=F.Mesh(ctx, pos, idx), vt=vt, t=t, charts=charts, tri=torch.zeros(T, **i32),
                vert=torch.zeros(V, **i32))


def _run_charts(case, s):
    F.fa_chartify(s["ctx"].handle, s["mesh"].handle, s["vt"], case["mode"], s["tri"], s["vert"], s["charts"])
    return [s["tri"], s["vert"], s["t"]["root"], s["t"]["count"]]


def _uv_inputs(case, seed):
    """A floor cut into charts of `rows` rows of quads; every tenth chart unseen; placements anywhere in the
    atlas.  The camera stands off the floor, so no triangle crosses the near plane."""
    n, parts = case["detail"], case["parts"]
    pos, idx = _floor(seed, parts, n)
    row = torch.arange(n - 1, device="cuda").repeat_interleave(2 * (n - 1)) // case["rows"]
    per = int(row[-1]) + 1
    label = (torch.arange(parts, device="cuda").view(-1, 1) * per + row.view(1, -1)).reshape(-1)
    seen = torch.arange(parts * per, device="cuda") % 10 != 9
    number = torch.cumsum(seen, 0) - 1
    tri = torch.where(seen[label], number[label], -1).to(torch.int32)
    C = int(seen.sum())
    om = 1 << case["atlas_log2"]
    place = torch.randint(0, om, (C, 4), generator=_gen(seed, 5), device="cuda", dtype=torch.int32)
    res = [48, om + 37, om, 0, C]
    M = S.hemisphere_camera(seed, case["width"], case["height"], radius=3.0 if parts == 1 else 14.0)
    return pos, idx, tri, C, place, res, M


def _prepare_uv(case, seed):
    pos, idx, tri, C, place, res, M = _uv_inputs(case, seed)
    T, V = idx.shape[0], pos.shape[0]
    ctx = F.Context(max_tris=T, max_verts=V, max_charts=C, max_width=case["width"], max_height=case["height"],
                    max_atlas_log2=case["atlas_log2"])
    i32 = dict(dtype=torch.int32, device="cuda")
    t, charts = _charts_struct(C, count=torch.tensor([C], **i32))
    return dict(ctx=ctx, mesh=F.Mesh(ctx, pos, idx), M=M, tri=tri, place=place, t=t, charts=charts,
                res=torch.tensor(res, **i32), uv=torch.full((T, 3, 2), float("nan"), device="cuda"),
                affine=torch.zeros(C, 6, device="cuda"))


def _run_uv(case, s):
    W, H, r = case["width"], case["height"], case["ratio"]
    F.fa_parameterize(s["ctx"].handle, s["mesh"].handle, s["M"], W, H, r, s["tri"], s["charts"])
    F.fa_uv(s["ctx"].handle, s["mesh"].handle, s["M"], W, H, r, s["tri"], s["charts"], s["place"], s["res"],
            case["atlas_log2"], 64, s["uv"], s["affine"])
    return dict(bbox=s["t"]["bbox"], fa=s["t"]["fa"], fb=s["t"]["fb"], rot=s["t"]["rot"], uv=s["uv"],
                affine=s["affine"])


def _exact_uv(case, seed):
    pos, idx, tri, C, place, res, M = _uv_inputs(case, seed)
    W, H, r = case["width"], case["height"], case["ratio"]
    M = torch.as_tensor(np.asarray(M, np.float32), device="cuda").double().view(4, 4)
    clip = pos.double() @ M[:, :3].T + M[:, 3]
    c = clip[idx.long()]  # [T, 3, 4]
    w = c[..., 3:4]
    ndc = c[..., :2] / w
    boxed = torch.maximum(torch.minimum(ndc, torch.ones_like(ndc)), -torch.ones_like(ndc))
    on = tri >= 0
    at = tri[on].long().view(-1, 1).expand(-1, 2)
    inf = torch.full((C, 2), float("inf"), device="cuda", dtype=torch.float64)
    lo = inf.scatter_reduce(0, at, boxed[on].amin(1), "amin")
    hi = (-inf).scatter_reduce(0, at, boxed[on].amax(1), "amax")
    half = torch.tensor([0.5 * W, 0.5 * H], device="cuda", dtype=torch.float64)
    size = (hi - lo) * half
    foot = torch.ceil(256.0 * r * size)
    rot = foot[:, 0] > foot[:, 1]
    alpha, s = float(1 << case["atlas_log2"]) / res[1], r * res[0] / 64.0
    t = tri[on].long()
    local = (ndc[on] - lo[t].unsqueeze(1)) * half
    turned = torch.stack([local[..., 1], size[t, 0].unsqueeze(1) - local[..., 0]], 2)
    local = torch.where(rot[t].view(-1, 1, 1), turned, local)
    uv = torch.full((idx.shape[0], 3, 2), float("nan"), device="cuda", dtype=torch.float64)
    uv[on] = alpha * (place[t, :2].double().unsqueeze(1) + s * local)
    g, z = s * half, torch.zeros(C, device="cuda", dtype=torch.float64)
    X, Y = place[:, 0].double(), place[:, 1].double()
    plain = torch.stack([alpha * g[0] + z, z, alpha * (X - g[0] * lo[:, 0]),
                         z, alpha * g[1] + z, alpha * (Y - g[1] * lo[:, 1])], 1)
    turned = torch.stack([z, alpha * g[1] + z, alpha * (X - g[1] * lo[:, 1]),
                          z - alpha * g[0], z, alpha * (Y + g[0] * hi[:, 0])], 1)
    return dict(bbox=torch.cat([lo, hi], 1), fa=None, fb=None, rot=None, uv=uv,
                affine=torch.where(rot.view(-1, 1), turned, plain))


_PREPARE = dict(frame=_prepare_frame, path=_prepare_path, batch=_prepare_batch, plan=_prepare_batch, serve=_prepare_serve,
                pack=_prepare_pack, vis=_prepare_vis, charts=_prepare_charts, uv=_prepare_uv)
_RUN = dict(frame=_run_frame, path=_run_path, batch=_run_batch, plan=_run_plan, serve=_run_serve, pack=_run_pack,
            vis=_run_vis, charts=_run_charts, uv=_run_uv)


def prepare(case, seed):
    s = _PREPARE[case["kind"]](case, int(seed))
    s["case"] = case
    return s


def run(state):
    return _RUN[state["case"]["kind"]](state["case"], state)


def exact(case, seed):
    """Boxes and texture coordinates have 64-bit values for given charts and placements; in a whole frame they
    follow from discrete steps (visible set, charts, packing) that plain arrays do not repeat in reasonable time."""
    return _exact_uv(case, int(seed)) if case["kind"] == "uv" else None


# ------------------------------------------------------------------ what a pass cannot do without

def _frame_work(T, V, W, H):
    """Positions and indices in; visible bits, chart ids and, for the triangles a window of this size can show
    (one per four pixels at most, half of them facing away), texture coordinates out."""
    shown = min(T // 2, W * H // 4)
    return 12 * V + 12 * T + T // 8 + 4 * T + 24 * shown, 100 * T + 200 * shown


def work(case):
    kind = case["kind"]
    if kind == "frame":
        T, V = _sizes(case["scene"], case["parts"], case["detail"])
        b, f = _frame_work(T, V, case["width"], case["height"])
    elif kind == "path":
        b, f = _frame_work(*_sizes("floor", 1, case["detail"]), case["width"], case["height"])
    elif kind in ("batch", "plan"):
        w = [_frame_work(*_sizes("floor", parts, case["detail"]), W, H) for parts, W, H, _ in _views(case)]
        b, f = (sum(x) for x in zip(*w))
    elif kind == "serve":
        w = [_frame_work(*_sizes("spheres", parts, case["detail"]), W, H) for parts, W, H, _ in _clients(case)]
        b, f = (sum(x) for x in zip(*w))
    elif kind == "pack":  # footprints in, order and placements out; every box at every scale
        b, f = case["boxes"] * (8 + 4 + 16), case["boxes"] * case["scales"] * 8
    elif kind == "vis":
        T, V = _sizes(case["scene"], case["parts"], case["detail"])
        b, f = 12 * V + 12 * T + T // 8, 100 * T
    elif kind == "charts":  # visible bits and neighbours in, chart ids out
        T, V = _sizes("floor", case["parts"], case["detail"])
        b, f = T // 8 + 12 * T // 2 + 4 * T + 4 * V, 10 * T
    else:  # uv: positions, indices and chart ids in, texture coordinates out
        T, V = _sizes("floor", case["parts"], case["detail"])
        b, f = 12 * V + 12 * T + 4 * T + 24 * T, 300 * T
    return {"bytes": int(b), "flops": int(f)}
