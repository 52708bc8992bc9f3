"""The calls whose time matters: listed cases and a generator of more of the same ranges.

Every case goes through the public entry points of the package
(paper_2604_21749_gb300.api) on seeded inputs made on the GPU.  The meshes
have the structure of the scans and terrains a brute-force rasterizer is used
for: dense, opaque, indexed, locally ordered triangles with FP32 positions,
uint32 indices and RGBA8 vertex colours.  Their heights are fractal noise;
the seed decides the heights, the placement and the camera's pose.

Paths ("path" of a case):
  render       one frame into a visibility buffer, as a viewer or a depth /
               id pass does it each time the camera moves
  view         a frame and its RGBA8 image, the loop of an interactive viewer
  batch        many instances of many meshes into several views at once, by
               the graph-replayed batched call
  static       the context-free call that allocates nothing
  resolve      the image of a rendered buffer, FP32 and RGBA8
  textured     the image with textures and the mip level of every pixel
  supersample  the box-filtered image of a buffer with ss x ss samples a pixel
  interpolate  the differentiable step: forward and backward of a per-vertex
               attribute, gradients of the attribute and of the positions
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2604_21749_gb300 import api


# ------------------------------------------------------------------ cases --
def _terrain(path, n, tx, tz, W, H, camera, dist=1.0, order="rows", **more):
    c = {"path": path, "scene": "terrain", "n": n, "tx": tx, "tz": tz, "W": W, "H": H, "camera": camera,
         "dist": dist, "order": order}
    c.update(more)
    return c


def listed():
    cases = [
        # The smallest call: a preview-sized frame of a small heightfield that stands on two ground
        # triangles reaching behind the camera.  Launches and latency are what it takes.
        dict(_terrain("render", 256, 1, 1, 512, 512, "small"), name="small_frame"),
        # Indoors: the camera inside a closed box, twelve triangles that cross the near plane and
        # fill a 4K screen between them (clipping, tiles, large spans).
        dict(path="render", scene="room", W=3840, H=2160, raycast=False, name="room_4k"),
        # The interactive viewer: a scan of some millions of triangles close up at full HD, frame and
        # RGBA8 image each pass.
        dict(_terrain("view", 1448, 1, 1, 1920, 1080, "close", 0.35), name="viewer_hd"),
        # One 100-million-triangle scan, close up at 4K.
        dict(_terrain("render", 7072, 1, 1, 3840, 2160, "close", 0.1), name="scan_100m"),
        # A terrain of a billion triangles (30 tiles) seen as a whole at 4K: the largest call.
        dict(_terrain("render", 4096, 6, 5, 3840, 2160, "overview"), name="terrain_billion"),
        # Geometry kept compressed to fit more of it: nine tiles of 8.4 M triangles.
        dict(_terrain("render", 2048, 3, 3, 3840, 2160, "overview", compressed=True), name="terrain_compressed"),
        # A populated scene into four views at once: 64 meshes of 1e4 to 2e6 triangles, 1000 instances
        # (half of them closed surfaces, so half of their triangles face away).
        dict(path="batch", scene="crowd", meshes=64, instances=1000, tmin=1e4, tmax=2e6, W=3840, H=2160, views=4,
             name="crowd_views"),
        # A plug-in that may not allocate: one million-triangle mesh, four instances, HD ready.
        dict(path="static", scene="copies", n=724, instances=4, W=1280, H=720, order="rows", name="static_copies"),
        # The image of a 4K frame of a 33 M-triangle terrain (an FP32 one for further processing and
        # an RGBA8 one for the screen).
        dict(_terrain("resolve", 1024, 4, 4, 3840, 2160, "overview"), name="resolve_4k"),
        # The same step with textures (a 2048 x 2048 chain for each of four tiles).
        dict(_terrain("textured", 512, 2, 2, 3840, 2160, "overview", log2_size=11), name="textured_4k"),
        # Anti-aliased output: 2 x 2 samples for each pixel of a full-HD image.
        dict(_terrain("supersample", 1024, 2, 2, 1920, 1080, "overview", ss=2), name="supersample_hd"),
        # One optimisation step on vertex colours and positions (4.2 M triangles, 1024 x 1024 image).
        dict(_terrain("interpolate", 1448, 1, 1, 1024, 1024, "overview", channels=3), name="interpolate_step"),
    ]
    return cases


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _size(rng, lo, hi):
    """An image size: usual ones and odd ones, W and H drawn apart."""
    W = int(round(_log(rng, lo, hi)))
    H = max(1, int(round(W * rng.uniform(0.5, 1.0))))
    return W, H


def draw(rng):
    path = rng.choice(["render", "render", "render", "room", "compressed", "view", "batch", "static", "resolve",
                       "textured", "supersample", "interpolate"])
    order = rng.choice(["rows", "rows", "mirrored", "scattered"])
    camera = rng.choice(["overview", "close"])
    dist = round(_log(rng, 0.02, 1.0), 4)
    if path == "room":
        W, H = _size(rng, 200, 3840)
        return dict(path="render", scene="room", W=W, H=H, raycast=rng.random() < 0.5)
    if path == "compressed":
        W, H = _size(rng, 200, 3840)
        tx, tz = rng.randint(1, 3), rng.randint(1, 3)
        return _terrain("render", int(_log(rng, 100, 2048)), tx, tz, W, H, camera, dist, order, compressed=True)
    if path == "batch":
        W, H = _size(rng, 320, 3840)
        return dict(path="batch", scene="crowd", meshes=rng.randint(2, 64), instances=int(_log(rng, 64, 1000)),
                    tmin=1e3, tmax=round(_log(rng, 1e4, 2e6)), W=W, H=H, views=rng.randint(1, 4))
    if path == "static":
        W, H = _size(rng, 128, 2560)
        return dict(path="static", scene="copies", n=int(_log(rng, 64, 1448)), instances=rng.randint(1, 8), W=W, H=H,
                    order=order)
    if path == "interpolate":
        W, H = _size(rng, 200, 2048)
        return _terrain("interpolate", int(_log(rng, 64, 2048)), 1, 1, W, H, camera, max(dist, 0.1), order,
                        channels=rng.choice([1, 3, 3, 4, 8, 16]))
    if path == "supersample":
        ss = rng.choice([2, 2, 3, 4])
        W, H = _size(rng, 100, 3840 // ss)
        return _terrain("supersample", int(_log(rng, 64, 1024)), rng.randint(1, 2), rng.randint(1, 2), W, H, camera,
                        dist, order, ss=ss)
    if path == "textured":
        W, H = _size(rng, 200, 3840)
        return _terrain("textured", int(_log(rng, 64, 1024)), rng.randint(1, 3), rng.randint(1, 3), W, H, camera, dist,
                        order, log2_size=rng.randint(6, 11))
    W, H = _size(rng, 200, 3840)
    tx, tz = rng.randint(1, 4), rng.randint(1, 4)
    return _terrain(path, int(_log(rng, 64, 4096 if path == "render" else 1448)), tx, tz, W, H, camera, dist, order)


# ----------------------------------------------------------------- inputs --
def _gen(*words):
    h = 1469598103934665603
    for w in words:
        h = ((h ^ (int(w) & 0xFFFFFFFF)) * 1099511628211) & 0x7FFFFFFFFFFFFFFF
    return torch.Generator(device="cuda").manual_seed(h)


def _noise(g, nu, nv, amplitude=0.2, octaves=6, base=8):
    """Fractal noise on (nv + 1) x (nu + 1) vertices: bicubic lattices of doubling frequency and
    halving weight."""
    total = torch.zeros((nv + 1, nu + 1), device="cuda")
    wsum = 0.0
    for o in range(octaves):
        f = base << o
        lat = torch.rand((1, 1, f + 1, f + 1), device="cuda", generator=g)
        total.add_(F.interpolate(lat, size=(nv + 1, nu + 1), mode="bicubic", align_corners=True)[0, 0],
                   alpha=0.5 ** o)
        wsum += 0.5 ** o
    return total.mul_(amplitude / wsum)


def _grid_indices(nu, nv, order, g):
    """Two triangles a cell, row by row; 'mirrored' splits the cells along the other diagonal, and
    'scattered' lists the triangles in random order (a mesh nobody sorted)."""
    i = torch.arange(nu, device="cuda", dtype=torch.int32)
    j = torch.arange(nv, device="cuda", dtype=torch.int32)
    v00 = (j[:, None] * (nu + 1) + i[None, :]).reshape(-1)
    v10, v01, v11 = v00 + 1, v00 + (nu + 1), v00 + (nu + 2)
    if order == "mirrored":
        tri = torch.stack([v00, v01, v11, v00, v11, v10], dim=1)
    else:
        tri = torch.stack([v00, v01, v10, v10, v01, v11], dim=1)
    tri = tri.reshape(-1, 3)
    if order == "scattered":
        tri = tri[torch.randperm(tri.shape[0], device="cuda", generator=g)]
    return tri.contiguous()


def _colours(h, amplitude=0.2):
    t = (h / amplitude).clamp(0, 1)
    return torch.stack([t * 255, (1 - t) * 180 + 40, (1 - t) * 90 + t * 160, torch.full_like(t, 255.0)],
                       dim=1).round().to(torch.uint8)


def _heightfield(n, g, idx, colours=True):
    h = _noise(g, n, n).reshape(-1)
    k = torch.arange(n + 1, device="cuda", dtype=torch.float32) / n
    pos = torch.empty(((n + 1) * (n + 1), 3), device="cuda")
    pos[:, 0] = k.repeat(n + 1)
    pos[:, 1] = h
    pos[:, 2] = k.repeat_interleave(n + 1)
    return pos, idx, _colours(h) if colours else None


def _sphere(n, g):
    """A closed displaced sphere of n x 2n cells, triangles facing outwards."""
    r = 1.0 + _noise(g, 2 * n, n, octaves=5)
    r[:, -1] = r[:, 0]
    r[0, :], r[-1, :] = r[0, 0], r[-1, 0]
    lat = torch.arange(n + 1, device="cuda", dtype=torch.float32)[:, None] * (math.pi / n)
    lon = (torch.arange(2 * n + 1, device="cuda") % (2 * n)).to(torch.float32)[None, :] * (math.pi / n)
    st = torch.sin(lat)
    st[0], st[-1] = 0.0, 0.0
    pos = torch.stack([r * st * torch.cos(lon), r * torch.cos(lat) * torch.ones_like(lon), r * st * torch.sin(lon)],
                      dim=2).reshape(-1, 3).contiguous()
    idx = _grid_indices(2 * n, n, "rows", None)[:, [0, 2, 1]].contiguous()
    return pos, idx, _colours((r - 1.0).reshape(-1))


def _look_at(eye, target):
    eye = np.asarray(eye, np.float64)
    f = np.asarray(target, np.float64) - eye
    f /= np.linalg.norm(f)
    s = np.cross(f, (0.0, 1.0, 0.0))
    s /= np.linalg.norm(s)
    u = np.cross(s, f)
    m = np.eye(4)
    m[0, :3], m[1, :3], m[2, :3] = s, u, -f
    m[0, 3], m[1, 3], m[2, 3] = -s @ eye, -u @ eye, f @ eye
    return m.astype(np.float32)


def _perspective(fovy, aspect, near, far):
    f = 1.0 / math.tan(math.radians(fovy) / 2.0)
    p = np.zeros((4, 4))
    p[0, 0], p[1, 1] = f / aspect, f
    p[2, 2], p[2, 3] = (far + near) / (near - far), 2.0 * far * near / (near - far)
    p[3, 2] = -1.0
    return p.astype(np.float32)


def _translate(x, y, z):
    m = np.eye(4, dtype=np.float32)
    m[:3, 3] = (x, y, z)
    return m


def _camera(case, rng, W, H, pos):
    """The pose: an overview of all tiles from above their near edge, a close-up of one spot, or the
    small scene's fixed distance; the seed turns and shifts it."""
    kind = case["camera"]
    if kind == "close":
        x, z = rng.uniform(0.3, 0.7, size=2)
        n = case["n"]
        y = float(pos[int(z * n) * (n + 1) + int(x * n), 1])
        dist, pitch, yaw = case["dist"], math.radians(rng.uniform(35, 55)), rng.uniform(0, 2 * math.pi)
        tgt = np.array([x, y, z])
        eye = tgt + dist * np.array([math.cos(pitch) * math.sin(yaw), math.sin(pitch), math.cos(pitch) * math.cos(yaw)])
        return _look_at(eye, tgt), _perspective(60.0, W / H, max(1e-4, 1e-3 * dist), 100.0)
    if kind == "small":
        eye = (0.5 + rng.uniform(-0.05, 0.05), 0.8, -0.3)
        return _look_at(eye, (0.5, 0.0, 0.5)), _perspective(60.0, W / H, 1e-3, 1000.0)
    tx, tz = case["tx"], case["tz"]
    s = max(tx, tz)
    eye = (tx / 2 + rng.uniform(-0.02, 0.02) * s, 0.2 + 0.45 * s, -0.15 * s)
    return (_look_at(eye, (tx / 2 + rng.uniform(-0.02, 0.02) * s, 0.0, tz / 2)),
            _perspective(55.0, W / H, 1e-2, 100.0 * s))


def _rotation(rng):
    w, x, y, z = (lambda q: q / np.linalg.norm(q))(rng.normal(size=4))
    return np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w)],
                     [2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w)],
                     [2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)]])


def _room():
    p = np.array([[x, y, z] for x in (-3, 3) for y in (-2, 2) for z in (-4, 4)], np.float32)
    idx = []
    for a, b, c, d in [(0, 1, 3, 2), (4, 6, 7, 5), (0, 4, 5, 1), (2, 3, 7, 6), (0, 2, 6, 4), (1, 5, 7, 3)]:
        idx += [[a, c, b], [a, d, c]]
    return p, np.array(idx, np.int32)


def _mip_chain(log2_size, g):
    side = 1 << log2_size
    lev = torch.randint(0, 256, (max(side >> 3, 1), max(side >> 3, 1), 4), device="cuda", generator=g)
    lev = lev.repeat_interleave(min(side, 8), 0).repeat_interleave(min(side, 8), 1)
    lev = (lev * 3 + torch.randint(0, 256, (side, side, 4), device="cuda", generator=g)) >> 2
    lev[..., 3] = 255
    out = [lev.reshape(-1).to(torch.uint8)]
    while lev.shape[0] > 1:
        lev = (lev[0::2, 0::2] + lev[0::2, 1::2] + lev[1::2, 0::2] + lev[1::2, 1::2] + 2) >> 2
        out.append(lev.reshape(-1).to(torch.uint8))
    return torch.cat(out)


def prepare(case, seed):
    rng = np.random.default_rng([seed, 77])
    path, W, H = case["path"], case["W"], case["H"]
    st = {"path": path, "W": W, "H": H}
    if case["scene"] == "copies":
        g = _gen(seed, 1)
        pos, idx, _ = _heightfield(case["n"], g, _grid_indices(case["n"], case["n"], case["order"], g), False)
        k = case["instances"]
        side = math.ceil(math.sqrt(k))
        models = [_translate(i % side, 0, i // side) for i in range(k)]
        eye = (side / 2 + rng.uniform(-0.1, 0.1), 0.2 + 0.45 * side, -0.15 * side)
        st.update(pos=pos, idx=idx, models=models, view=_look_at(eye, (side / 2, 0, side / 2)),
                  proj=_perspective(55.0, W / H, 1e-2, 100.0 * side),
                  vis=torch.empty((H, W), dtype=torch.int64, device="cuda"))
        return st

    r = api.Renderer()
    st["r"] = r
    if case["scene"] == "room":
        p, i = _room()
        m = r.upload_mesh(torch.from_numpy(p).cuda(), torch.from_numpy(i).cuda())
        r.add_instance(m)
        if case["raycast"]:
            r.set_config(stage3_raycast=1)
        eye = np.array([0.3, 0.1, 0.2]) + rng.uniform(-0.2, 0.2, size=3)
        st.update(view=_look_at(eye, (1.0, -0.4, -2.0)), proj=_perspective(80.0, W / H, 0.05, 100.0), vis=r.new_vis(W, H))
        return st

    if case["scene"] == "crowd":
        t = np.exp(rng.uniform(math.log(case["tmin"]), math.log(case["tmax"]), size=case["meshes"]))
        for m in range(case["meshes"]):
            g = _gen(seed, 2, m)
            if m % 2 == 0:
                n = max(8, int(round(math.sqrt(t[m] / 2))))
                pos, idx, col = _heightfield(n, g, _grid_indices(n, n, "rows", g))
            else:
                pos, idx, col = _sphere(max(8, int(round(math.sqrt(t[m] / 4)))), g)
            r.upload_mesh(pos, idx, col)
        area = 200.0
        for k in range(case["instances"]):
            m4 = np.eye(4)
            m4[:3, :3] = _rotation(rng) * rng.uniform(0.1, 10.0)
            m4[:3, 3] = (rng.uniform(-area / 2, area / 2), 0.0, rng.uniform(-area / 2, area / 2))
            r.add_instance(k if k < case["meshes"] else int(rng.integers(0, case["meshes"])), m4.astype(np.float32))
        views = []
        for v in range(case["views"]):
            w, h = (W, H) if v < 2 else (max(1, W // 2), max(1, H // 2))
            a = 2 * math.pi * v / case["views"] + 0.3
            eye = (0.7 * area * math.cos(a), 0.35 * area, 0.7 * area * math.sin(a))
            tgt = (0.1 * area * math.cos(a + 1), 0.0, 0.1 * area * math.sin(a + 1))
            views.append((_look_at(eye, tgt), _perspective(60.0, w / h, 0.05, 2000.0), w, h, r.new_vis(w, h)))
        st["views"] = views
        return st

    n, tx, tz = case["n"], case["tx"], case["tz"]
    shade = path in ("view", "resolve", "textured", "supersample")
    idx0 = _grid_indices(n, n, case["order"], _gen(seed, 3))
    mid, first, ids = (tz // 2) * tx + tx // 2, None, []
    for k in range(tx * tz):
        # every tile has buffers of its own, as separately loaded meshes have
        pos, idx, col = _heightfield(n, _gen(seed, 4, k), idx0 if k == tx * tz - 1 else idx0.clone(), shade)
        ids.append(r.upload_mesh(pos, idx, col, compressed=bool(case.get("compressed"))))
        at = (k % tx, k // tx) if case["camera"] != "close" else (k % tx - mid % tx, k // tx - mid // tx)
        r.add_instance(ids[-1], _translate(float(at[0]), 0.0, float(at[1])))
        if k == mid:
            first = pos
        if path == "interpolate":
            st["pos"], st["idx"] = pos, idx
        if path in ("resolve", "textured", "supersample"):
            st.setdefault("meshes", []).append((pos, idx, col, at))
    if case["camera"] == "small":
        q = 100.0
        ground = torch.tensor([[-q, -0.05, -q], [q, -0.05, -q], [-q, -0.05, q], [q, -0.05, q]], device="cuda")
        r.add_instance(r.upload_mesh(ground, torch.tensor([[0, 2, 1], [1, 2, 3]], dtype=torch.int32, device="cuda")))
    ss = case.get("ss", 1)
    st["view"], st["proj"] = _camera(case, rng, W, H, first)
    st["vis"] = r.new_vis(W * ss, H * ss)
    if path == "textured":
        k = torch.arange(n + 1, device="cuda", dtype=torch.float32) / n
        uv = torch.stack([k.repeat(n + 1), k.repeat_interleave(n + 1)], dim=1).contiguous()
        st["uv"], st["tex"] = uv, []
        for m in ids:
            st["tex"].append(_mip_chain(case["log2_size"], _gen(seed, 5, m)))
            r.set_mesh_texture(m, uv.clone(), st["tex"][-1], case["log2_size"])
    if path in ("resolve", "textured", "supersample", "interpolate"):
        r.render(st["view"], st["proj"], W * ss, H * ss, st["vis"])
        st["ss"] = ss
    if path == "interpolate":
        C = case["channels"]
        g = _gen(seed, 6)
        st["mesh"] = ids[0]
        st["pos"] = st["pos"].requires_grad_()
        st["attr"] = torch.rand((st["pos"].shape[0], C), device="cuda", generator=g).requires_grad_()
        # the gradient of an image loss: the residual of a render against its target
        st["grad"] = torch.randn((H, W, C), device="cuda", generator=g) * 0.05
    torch.cuda.synchronize()
    return st


# -------------------------------------------------------------------- run --
def run(st):
    path = st["path"]
    if path == "static":
        return api.render_static(st["pos"], st["idx"], st["models"], st["view"], st["proj"], st["W"], st["H"],
                                 vis=st["vis"])
    r = st["r"]
    if path == "render":
        return r.render(st["view"], st["proj"], st["W"], st["H"], st["vis"])
    if path == "view":
        vis = r.render(st["view"], st["proj"], st["W"], st["H"], st["vis"])
        return vis, r.resolve(st["view"], st["proj"], vis, want_f32=False)[1]
    if path == "batch":
        return r.render_batch(st["views"], use_graph=True)
    if path == "resolve":
        return r.resolve(st["view"], st["proj"], st["vis"])
    if path == "textured":
        return r.resolve_textured(st["view"], st["proj"], st["vis"])
    if path == "supersample":
        return r.resolve_ss(st["view"], st["proj"], st["vis"], st["ss"])
    out = api.InterpolateFn.apply(r, st["mesh"], st["pos"], st["attr"], st["vis"], st["view"], st["proj"])
    gp, ga = torch.autograd.grad(out, (st["pos"], st["attr"]), st["grad"])
    return out.detach(), gp, ga


# ------------------------------------------------------------------- work --
def work(case):
    """What a pass cannot do without.  Rendering reads the indices (12 B a triangle) and positions
    (12 B a vertex; compressed: the packed indices and 6 B) once, transforms each vertex once a view
    (18 flops) and writes 8 B a pixel.  The screen passes read 8 B a pixel and write the image; the
    triangles under the pixels are read once each (indices, positions and attributes of at most one
    triangle a pixel)."""
    path, W, H = case["path"], case["W"], case["H"]
    px = W * H
    if case["scene"] == "room":
        return {"bytes": 8 * px + 36 * 12, "flops": 20 * px}
    if case["scene"] == "crowd":
        t = math.exp((math.log(case["tmin"]) + math.log(case["tmax"])) / 2) if case["meshes"] < 8 else \
            (case["tmax"] - case["tmin"]) / math.log(case["tmax"] / case["tmin"])
        px = sum(px if v < 2 else px // 4 for v in range(case["views"]))
        return {"bytes": 18 * t * case["meshes"] + 8 * px, "flops": 9 * t * case["instances"] * case["views"]}
    n = case["n"]
    if case["scene"] == "copies":
        T, V = 2 * n * n, (n + 1) ** 2
        return {"bytes": 12 * T + 12 * V + 8 * px, "flops": 18 * V * case["instances"]}
    T, V = 2 * n * n * case["tx"] * case["tz"], (n + 1) ** 2 * case["tx"] * case["tz"]
    if path in ("render", "view"):
        bits = math.ceil(math.log2((n + 1) ** 2)) if case.get("compressed") else 32
        geo = 3 * T * bits / 8 + V * (6 if case.get("compressed") else 12)
        return {"bytes": geo + 8 * px + (4 * px + min(4 * V, 12 * px) if path == "view" else 0),
                "flops": 18 * V + (60 * px if path == "view" else 0)}
    if path == "resolve":
        return {"bytes": 28 * px + min(60 * px, 12 * T + 16 * V), "flops": 80 * px}
    if path == "textured":
        return {"bytes": 29 * px + min(76 * px, 12 * T + 20 * V + 4 * px), "flops": 250 * px}
    if path == "supersample":
        s = case["ss"] ** 2 * px
        return {"bytes": 8 * s + 20 * px + min(60 * s, 12 * T + 16 * V), "flops": 80 * s}
    C = case["channels"]
    # forward: buffer, triangles, image; backward: buffer, triangles, image gradient, both gradients out
    return {"bytes": 2 * (8 * px + min((48 + 12 * C) * px, 12 * T + (12 + 4 * C) * V)) + 8 * C * px + (12 + 4 * C) * V,
            "flops": (200 + 12 * C) * px}


# ------------------------------------------------------------------ exact --
def _rays(x, y, W, H, proj):
    rx = ((2 * x + 1).double() / W - 1) / float(proj[0, 0])
    ry = ((2 * y + 1).double() / H - 1) / float(proj[1, 1])
    return torch.stack([rx, ry, -torch.ones_like(rx)], dim=-1)


def _bary(r, v):
    """Barycentrics of the hit of each ray with its triangle's plane; v: (..., 3, 3) view space."""
    D = torch.stack([(r * torch.linalg.cross(v[..., (k + 1) % 3, :], v[..., (k + 2) % 3, :])).sum(-1)
                     for k in range(3)], dim=-1)
    return D / D.sum(-1, keepdim=True)


def _view_space(p, view, at):
    M = torch.from_numpy(np.asarray(view, np.float64)).cuda()
    w = p + torch.tensor([float(at[0]), 0.0, float(at[1])], dtype=torch.float64, device="cuda")
    return w @ M[:3, :3].T + M[:3, 3]


def _covered(st, W, H, base, T):
    """(pixel, x, y, triangle) of the pixels that show triangles base .. base + T - 1."""
    ids = (st["vis"].reshape(-1) & ((1 << 36) - 1)) - base
    ok = (st["vis"].reshape(-1) != -1) & (ids >= 0) & (ids < T)
    pix = ok.nonzero()[:, 0]
    return pix, pix % W, pix // W, ids[pix]


def exact(case, seed):
    path = case["path"]
    if path in ("render", "view", "batch", "static"):
        return None                      # visibility words and bytes: whole numbers
    st = prepare(case, seed)
    ss = st["ss"]
    W, H = st["W"] * ss, st["H"] * ss
    view, proj = st["view"], np.asarray(st["proj"], np.float64)
    if path == "interpolate":
        C = case["channels"]
        pix, x, y, t = _covered(st, W, H, 0, st["idx"].shape[0])
        tri = st["idx"][t].long()
        pos = st["pos"].detach().double().requires_grad_()
        attr = st["attr"].detach().double().requires_grad_()
        b = _bary(_rays(x, y, W, H, proj), _view_space(pos[tri], view, (0, 0)))
        vals = (b[..., None] * attr[tri]).sum(1)
        out = torch.zeros((H * W, C), dtype=torch.float64, device="cuda").index_copy(0, pix, vals)
        gp, ga = torch.autograd.grad(out, (pos, attr), st["grad"].double().reshape(-1, C))
        return out.detach().reshape(H, W, C), gp, ga
    img = torch.zeros((H * W, 4), dtype=torch.float64, device="cuda")
    base = 0
    for k, (pos, idx, col, at) in enumerate(st["meshes"]):
        T = idx.shape[0]
        for lo in range(0, H * W, 1 << 22):
            part = {"vis": st["vis"].reshape(-1)[lo:lo + (1 << 22)]}
            pix, _, _, t = _covered(part, W, H, base, T)
            if pix.numel() == 0:
                continue
            pix = pix + lo
            x, y = pix % W, pix // W
            tri = idx[t].long()
            v = _view_space(pos[tri].double(), view, at)
            if path != "textured":
                b = _bary(_rays(x, y, W, H, proj), v)
                img[pix] = (b[..., None] * (col[tri].double() / 255)).sum(1)
                continue
            uv = st["uv"][tri].double()
            s = torch.stack([(_bary(_rays(x + (q & 1), y + (q >> 1), W, H, proj), v)[..., None] * uv).sum(1)
                             for q in range(4)])
            L = case["log2_size"]
            foot = (s.amax(0) - s.amin(0)).amax(-1) * (1 << L)
            lev = torch.floor(torch.log2(foot.clamp(min=1e-300))).clamp(0, L).long()
            side = torch.ones_like(lev) << (L - lev)
            start = ((1 << (2 * L + 2)) - (torch.ones_like(lev) << (2 * (L - lev) + 2))) // 3
            cell = torch.minimum(torch.floor(s[0] * side[:, None]).clamp(min=0).long(), side[:, None] - 1)
            img[pix] = st["tex"][k].reshape(-1, 4)[start + cell[:, 1] * side + cell[:, 0]].double() / 255
        base += T
    img = img.reshape(H, W, 4)
    if path == "textured":
        return img, None, None
    if ss > 1:
        img = img.reshape(H // ss, ss, W // ss, ss, 4).mean(dim=(1, 3))
    return img, None
