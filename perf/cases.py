"""The work this framework is measured by: frames of resident clouds, multi-view
launches, level of detail, shading, images to the host, serving and the opening
of a cloud, each through the public entry points of the package.

A case is a dict of plain values:

* ``kind``: ``frame`` (Context.render), ``host`` (pc_render_host), ``shards``
  (Context.render_range, merge_min, resolve), ``serve`` (pc_submit, pc_poll),
  ``open`` (Context.upload of raw points, then the first frame);
* ``scene``, ``points``, ``extent``, ``buildings``: the cloud (see ``_scene``);
* ``camera``, ``w``, ``h``, ``views``: what is drawn of it (see ``_cameras``);
* options: ``k`` (forced precision, 0 adaptive), ``cull``, ``shade`` (0 plain,
  1 two-word sums, 2 packed sums), ``lod`` (threshold in pixels; the cloud is
  then a layered octree), ``lod_far``, ``dilate``, ``graph`` (captured replay).

Every output is a whole buffer of integers: visibility keys (depth bits and
point index), RGBA8 images. They are unique for given inputs (binary32 operations
in a fixed order, ties settled by index, integer colour sums), so every case
compares exactly and none has a 64-bit value to be near to.
"""
import math

import numpy as np
import torch

import paper_2204_01287_gb300 as pcr

BATCH = 10240


# ---- cases ------------------------------------------------------------------

def _case(kind, scene, points, camera, w, h, **more):
    c = {"kind": kind, "scene": scene, "points": points, "extent": 10000.0, "buildings": 0.0,
         "camera": camera, "w": w, "h": h, "views": 1, "k": 0, "cull": True, "shade": 0,
         "lod": 0.0, "lod_far": 0.0, "dilate": False, "graph": False}
    c.update(more)
    return c


def listed():
    return [
        # A small cloud in a viewer's window: four short passes, where latency counts.
        _case("frame", "cube", 1_000_000, "orbit", 512, 512, extent=1.0, k=3, cull=False,
              name="cube_1m_512"),
        # The same cloud from 16 directions in one call (thumbnails, turntables), replayed
        # as a captured graph on a stream of the program's own.
        _case("frame", "cube", 1_000_003, "orbit", 512, 512, extent=1.0, views=16, graph=True,
              name="cube_1m_orbit16_graph"),
        # One request's view of a mid-size survey, an odd window size.
        _case("frame", "terrain", 10_000_000, "random", 1283, 721, name="survey_10m_view"),
        # A frame of a fly-through: culling and adaptive precision at work.
        _case("frame", "terrain", 100_000_000, "fly", 1920, 1080, name="fly_100m_1080p"),
        # The whole of a very large cloud in view, about a thousand points per pixel.
        _case("frame", "terrain", 2_000_000_000, "overview", 1920, 1080, extent=40000.0,
              buildings=0.2, name="overview_2b_1080p"),
        # A headset's stereo pair over a large cloud, both eyes in one launch.
        _case("frame", "terrain", 200_000_000, "stereo", 2016, 2240, extent=40000.0,
              buildings=0.2, views=2, name="stereo_200m"),
        # High-quality shading of a dense overview (two-word sums).
        _case("frame", "terrain", 200_000_000, "overview", 1920, 1080, extent=40000.0,
              buildings=0.2, shade=1, name="shaded_overview_200m"),
        # Level of detail along a fly-through.
        _case("frame", "terrain", 32_000_000, "fly", 1920, 1080, lod=300.0, name="lod_fly_32m"),
        # A headset over a level-of-detail cloud: foveated thresholds, dilation, shading.
        _case("frame", "terrain", 24_000_000, "stereo", 2016, 2240, views=2, lod=100.0,
              lod_far=300.0, dilate=True, shade=2, name="lod_foveated_stereo"),
        # A rendered image for the host (export, a network client), 4K.
        _case("host", "terrain", 10_000_000, "random", 3840, 2160, name="host_image_4k"),
        # A burst of 32 requests to the serving loop, drawn into the clients' framebuffers.
        _case("serve", "terrain", 10_000_000, "random", 1280, 720, views=32,
              name="serve_burst_32"),
        # Opening a cloud: raw points to the encoded cloud on the device, and its first frame.
        _case("open", "terrain", 4_000_000, "overview", 1280, 720, name="open_4m"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame"] * 10 + ["host", "shards", "serve", "open"])
    scene = rng.choice(["terrain", "terrain", "terrain", "terrain", "cube", "scan"])
    if scene == "cube":
        extent, camera = 1.0, rng.choice(["orbit", "inside"])
    else:
        extent = float(_log(rng, 2000, 40000))
        camera = rng.choice(["fly", "random", "overview", "stereo"])
    w, h = _log(rng, 160, 3840), _log(rng, 120, 2160)
    points = _log(rng, 100_000, 300_000_000)
    more = {"extent": extent, "buildings": rng.choice([0.0, 0.2]) if scene == "terrain" else 0.0,
            "cull": rng.random() < 0.85, "k": rng.choice([0] * 8 + [1, 2, 3])}
    if kind == "open":
        points = _log(rng, 100_000, 8_000_000)
    if kind == "serve":
        points = _log(rng, 100_000, 20_000_000)
        more["views"] = rng.randint(4, 48)
        w, h = min(w, 1920), min(h, 1080)
    if kind == "host":
        points = _log(rng, 100_000, 40_000_000)
    if kind == "frame":
        if camera == "stereo":
            more["views"] = 2
        elif camera != "overview" and points < 50_000_000 and rng.random() < 0.4:
            more["views"] = rng.randint(2, 24)
            w, h = min(w, 1280), min(h, 720)
        more["shade"] = rng.choice([0, 0, 0, 1, 2])
        more["dilate"] = rng.random() < 0.15
        more["graph"] = rng.random() < 0.2
        if scene != "scan" and rng.random() < 0.25:
            points = _log(rng, 100_000, 24_000_000)
            more["lod"] = float(_log(rng, 50, 600))
            more["lod_far"] = rng.choice([0.0, 2.0]) * more["lod"]
        # no more to do than the largest listed cases
        points = min(points, int(4e8 / more.get("views", 1) / (2.5 if more["shade"] else 1.0)))
    return _case(kind, scene, points, camera, w, h, **more)


def work(case):
    """What one pass has to move and compute. A view reads each visible point's words once
    (k = 1: 4 bytes, the usual precision; the cube's 30-bit points 12) and one colour per covered
    pixel, or with shading every visible point's colour, and writes 8 bytes of key and 4 of colour
    per pixel. The visible share is what these cameras see: everything from outside, about a
    fifth along a fly-through. A point costs its three clip rows, a divide and the pixel (30)."""
    n, px = case["points"], case["w"] * case["h"] * case["views"]
    outside = case["camera"] in ("orbit", "overview", "stereo")
    seen = n * (1.0 if outside else 0.2)
    if case["lod"]:
        seen = min(seen, 2_400_000 * max(1.0, (300.0 / case["lod"]) ** 2))
    shared = seen   # views of one launch share a cloud that is read once
    words = {1: 4, 2: 8, 3: 12}[case["k"] or 1]
    b = shared * words + 16 * px + (4 * seen if case["shade"] else 0)
    f = 30.0 * seen * case["views"]
    if case["kind"] == "host":
        b += 4 * px
    if case["kind"] == "open":
        b += n * (16 + 16)   # raw points and colours in, words and colours out
    return {"bytes": b, "flops": f}


def tolerance(case):
    return "exact"


def exact(case, seed):
    # Keys are binary32 bit patterns with indices, images are bytes: no 64-bit value exists.
    return None


# ---- inputs -------------------------------------------------------------------

def _rng(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + stream * 7919) & 0x7FFFFFFFFFFF)
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float32)


class _Terrain:
    """Value-noise heights (2 km base wavelength, 300 m amplitude, six octaves), as a
    bilinear height map."""

    def __init__(self, seed, extent):
        n = int(min(4096, max(256, extent / 10.0)))
        g = _rng(seed, 1)
        acc = torch.zeros(1, 1, n, n, device="cuda")
        amp, cells = 150.0, max(1.0, extent / 2000.0)
        for _ in range(6):
            lattice = _rand(g, 1, 1, int(cells) + 2, int(cells) + 2) * 2 - 1
            acc += amp * torch.nn.functional.interpolate(lattice, size=(n, n), mode="bicubic",
                                                         align_corners=True)
            amp, cells = amp * 0.5, cells * 2
        self.map, self.extent, self.n = acc[0, 0].contiguous().reshape(-1), extent, n

    def height(self, x, y):
        u = ((x / self.extent + 0.5) * (self.n - 1)).clamp(0, self.n - 1.001)
        v = ((y / self.extent + 0.5) * (self.n - 1)).clamp(0, self.n - 1.001)
        i, j = u.long(), v.long()
        fu, fv = u - i, v - j
        p = j * self.n + i
        m = self.map
        a = m[p] * (1 - fu) + m[p + 1] * fu
        b = m[p + self.n] * (1 - fu) + m[p + self.n + 1] * fu
        return a * (1 - fv) + b * fv

    def at(self, x, y):
        return float(self.height(torch.tensor([x], device="cuda"), torch.tensor([y], device="cuda")))


def _scene(case, seed, first, count, terrain):
    """Points [first, first + count) and their colours: uniform in a cube, a terrain (part of
    the points on box buildings), or a terrain in a scanner's order along rays."""
    g = _rng(seed, 100 + first % 1000003)
    n, e = count, case["extent"]
    if case["scene"] == "cube":
        xyz = _rand(g, n, 3)
        rgba = torch.randint(-2**31, 2**31 - 1, (n,), generator=g, device="cuda", dtype=torch.int32)
        return xyz, rgba
    if case["scene"] == "scan":
        per_line = 20000
        i = torch.arange(first, first + n, device="cuda", dtype=torch.float64)
        lines = max(1, (case["points"] + per_line - 1) // per_line)
        yaw = 2 * math.pi * (torch.floor(i / per_line) + 0.5 * _rand(g, n).double()) / lines
        dist = 5.0 + (0.3 * e - 5.0) * (torch.remainder(i, per_line) + _rand(g, n).double()) / per_line
        x, y = (dist * torch.cos(yaw)).float(), (dist * torch.sin(yaw)).float()
    else:
        x, y = (_rand(g, n) - 0.5) * e, (_rand(g, n) - 0.5) * e
    z = terrain.height(x, y)
    t = ((z / 300.0) + 0.5).clamp(0, 1)
    rgb = torch.stack([50 + 190 * t, 100 + 100 * t * t, 40 + 180 * t * t * t], 1)
    z = z + (_rand(g, n) * 2 - 1) * 0.01
    if case["buildings"] > 0:
        nb = int(max(20, 20000 * (e / 40000.0) ** 2))
        gb = _rng(seed, 2)
        bx, by = (_rand(gb, nb) - 0.5) * e * 0.98, (_rand(gb, nb) - 0.5) * e * 0.98
        wx, wy, hz = 10 + 50 * _rand(gb, nb), 10 + 50 * _rand(gb, nb), 5 + 75 * _rand(gb, nb)
        z0 = terrain.height(bx, by) - 2.0
        on = (_rand(g, n) < case["buildings"]).nonzero().squeeze(1)
        b = torch.randint(0, nb, (on.numel(),), generator=g, device="cuda")
        fu, fv, face = _rand(g, on.numel()), _rand(g, on.numel()), _rand(g, on.numel())
        ax, ay, az = wx[b], wy[b], hz[b]
        top, wall_x, wall_y = ax * ay, ax * az, ay * az
        pick = face * (top + 2 * wall_x + 2 * wall_y)
        roof = pick < top
        along_x = pick < top + 2 * wall_x
        far = torch.where(along_x, pick >= top + wall_x, pick >= top + 2 * wall_x + wall_y).float()
        x[on] = bx[b] + ax * (torch.where(roof | along_x, fu, far) - 0.5)
        y[on] = by[b] + ay * (torch.where(roof, fv, torch.where(along_x, far, fu)) - 0.5)
        z[on] = z0[b] + az * torch.where(roof, torch.ones_like(fv), fv)
        rgb[on] = 150.0
    rgb = (rgb + (_rand(g, n, 1) - 0.5) * 24).clamp(0, 255).int()
    rgba = rgb[:, 0] | (rgb[:, 1] << 8) | (rgb[:, 2] << 16) | (-1 << 24)
    return torch.stack([x, y, z], 1), rgba


def _spread3(v):
    for shift, mask in ((32, 0x001F00000000FFFF), (16, 0x001F0000FF0000FF), (8, 0x100F00F00F00F00F),
                        (4, 0x10C30C30C30C30C3), (2, 0x1249249249249249)):
        v = (v | (v << shift)) & mask
    return v


def _points(case, seed, terrain):
    n, step = case["points"], 40_000_000
    xyz = torch.empty(n, 3, device="cuda")
    rgba = torch.empty(n, device="cuda", dtype=torch.int32)
    for a in range(0, n, step):
        m = min(step, n - a)
        xyz[a:a + m], rgba[a:a + m] = _scene(case, seed, a, m, terrain)
    return xyz, rgba


def _encoded(xyz, rgba, sort):
    """The cloud in the layout of pc_upload_encoded (Morton order, batches of 10,240 points, 30-bit
    fixed point in three words), made on the GPU and handed over in pinned host arrays."""
    n, step = xyz.shape[0], 40_000_000
    if sort:
        lo, hi = xyz.amin(0).double(), xyz.amax(0).double()
        size = (hi - lo).clamp(min=1e-30)
        key = torch.empty(n, device="cuda", dtype=torch.int64)
        for a in range(0, n, step):
            q = torch.floor((xyz[a:a + step].double() - lo) / size * 2097152).clamp(0, 2097151).long()
            key[a:a + step] = _spread3(q[:, 0]) | (_spread3(q[:, 1]) << 1) | (_spread3(q[:, 2]) << 2)
            del q
        order = torch.sort(key, stable=True)[1]
        del key
        rgba = rgba[order]
        xyz = xyz[order]
        del order
    nb = (n + BATCH - 1) // BATCH
    batches = np.zeros(nb, pcr.BATCH_DTYPE)
    host = [torch.empty(n, dtype=torch.int32, pin_memory=True) for _ in range(4)]
    host[3].copy_(rgba)
    mins, sizes = [], []
    for a in range(0, n, BATCH * 4096):
        p = xyz[a:a + BATCH * 4096]
        m = p.shape[0]
        pad = (-m) % BATCH
        if pad:
            p = torch.cat([p, p[-1:].expand(pad, 3)])
        p = p.reshape(-1, BATCH, 3)
        mn = p.amin(1)
        sz = p.amax(1) - mn
        d = sz.double().clamp(min=1e-30)[:, None]
        q = torch.floor((p.double() - mn.double()[:, None]) / d * 1073741824.0)
        q = q.clamp(0, 1073741823).int().reshape(-1, 3)[:m]
        q = torch.where((sz > 0).repeat_interleave(BATCH, 0)[:m], q, torch.zeros_like(q))
        for i, shift in enumerate((20, 10, 0)):
            f = (q >> shift) & 1023
            host[i][a:a + m].copy_(f[:, 0] | (f[:, 1] << 10) | (f[:, 2] << 20))
        mins.append(mn)
        sizes.append(sz)
        del p, d, q
    batches["min"], batches["size"] = torch.cat(mins).cpu().numpy(), torch.cat(sizes).cpu().numpy()
    batches["first"] = np.arange(nb, dtype=np.int64) * BATCH
    batches["count"] = np.minimum(BATCH, n - np.arange(nb, dtype=np.int64) * BATCH)
    return [batches] + [t.numpy().view(np.uint32) for t in host]


def _look_at(eye, target, up, fovy, aspect, near, far):
    """World to clip, column-major float32 (the layout of pc_view)."""
    eye, target = np.asarray(eye, np.float64), np.asarray(target, np.float64)
    f = (target - eye) / np.linalg.norm(target - eye)
    s = np.cross(f, up)
    s /= np.linalg.norm(s)
    view = np.eye(4)
    view[0, :3], view[1, :3], view[2, :3] = s, np.cross(s, f), -f
    view[:3, 3] = -view[:3, :3] @ eye
    t = 1.0 / math.tan(math.radians(fovy) / 2)
    proj = np.zeros((4, 4))
    proj[0, 0], proj[1, 1], proj[3, 2] = t / aspect, t, -1.0
    proj[2, 2], proj[2, 3] = (far + near) / (near - far), 2 * far * near / (near - far)
    return (proj @ view).astype(np.float32).T.reshape(16)


def _cameras(case, seed, terrain):
    """One matrix per view: around or inside the unit cube; along a loop at 50 to 500 m above
    the ground; anywhere at 50 to 3000 m; the whole area from outside; its stereo pair."""
    r = np.random.RandomState(seed % (1 << 31))
    e, asp, out = case["extent"], case["w"] / case["h"], []
    z = (0, 0, 1)
    turn = r.uniform(-0.25, 0.25)   # where the viewer of an overview stands
    for v in range(case["views"]):
        a = r.uniform(0, 2 * math.pi)
        if case["camera"] == "orbit":
            eye = 0.5 + 2.0 * np.array([math.sin(a), 0.2 * math.sin(3 * a), math.cos(a)])
            m = _look_at(eye, (0.5, 0.5, 0.5), (0, 1, 0), 60.0, asp, 0.1, 100.0)
        elif case["camera"] == "inside":
            m = _look_at(r.uniform(0.2, 0.8, 3), r.uniform(0, 1, 3) + (0, 0, 2), (0, 1, 0), 60.0, asp,
                         0.01, 100.0)
        elif case["camera"] == "fly":
            x, y = 0.33 * e * math.cos(a), 0.22 * e * math.sin(a)
            tx, ty = 0.33 * e * math.cos(a + 0.19), 0.22 * e * math.sin(a + 0.19)
            m = _look_at((x, y, terrain.at(x, y) + r.uniform(50, 500)), (tx, ty, terrain.at(tx, ty)), z,
                         60.0, asp, 1.0, 4 * e)
        elif case["camera"] == "random":
            x, y, tx, ty = (float(t) for t in r.uniform(-0.5 * e, 0.5 * e, 4))
            m = _look_at((x, y, terrain.at(x, y) + r.uniform(50, 3000)), (tx + 10.0, ty, terrain.at(tx, ty)),
                         z, r.uniform(45, 90), asp, 1.0, 4 * e)
        else:
            stereo = case["camera"] == "stereo"
            d, up = (0.8, 0.45) if stereo else (0.95, 0.62)
            eye = np.array([d * e * math.sin(turn), -d * e * math.cos(turn), up * e])
            tgt = np.array([0.0, -0.05 * e if stereo else -0.02 * e, 0.0])
            if stereo:   # 65 mm between the eyes
                side = np.array([math.cos(turn), math.sin(turn), 0.0]) * (0.0325 if v else -0.0325)
                eye, tgt = eye + side, tgt + side
            m = _look_at(eye, tgt, z, 90.0 if stereo else 55.0, asp, 0.01 * e, 4 * e)
        out.append(m)
    return out


# ---- a program's state and one pass -------------------------------------------

def prepare(case, seed):
    terrain = None if case["scene"] == "cube" else _Terrain(seed, case["extent"])
    xyz, rgba = _points(case, seed, terrain)
    flags = ((pcr.PC_VIEW_CULL if case["cull"] else 0) | pcr.PC_VIEW_FORCE_K(case["k"]) |
             (0, pcr.PC_VIEW_HQS, pcr.PC_VIEW_HQS_PACKED)[case["shade"]] |
             (pcr.PC_VIEW_DILATE if case["dilate"] else 0))
    if case["kind"] == "shards":
        flags |= pcr.PC_VIEW_SIGNED_EMPTY
    views = [pcr.make_view(m, case["w"], case["h"], flags, case["lod"], case["lod_far"])
             for m in _cameras(case, seed, terrain)]
    ctx = pcr.Context(0, flags=pcr.PC_CFG_GRAPHS if case["graph"] else 0)
    state = {"kind": case["kind"], "ctx": ctx, "views": views, "stream": None}
    if case["kind"] == "open":
        state["xyz"], state["rgba"] = xyz.cpu().numpy(), rgba.cpu().numpy().view(np.uint32)
    else:
        state["cloud"] = ctx.upload_encoded(*_encoded(xyz, rgba, case["scene"] != "scan"))
        if case["lod"]:
            plain = state["cloud"]
            state["cloud"] = pcr.pc_build_lod(ctx.h, plain, 12, BATCH, 0)
            pcr.pc_release_cloud(ctx.h, plain)
        info = pcr.pc_cloud_get_info(ctx.h, state["cloud"])
        state["batches"] = info.n_batches
    del xyz, rgba
    if case["kind"] == "host":
        state["images"] = [torch.empty(v.width * v.height, dtype=torch.int32, pin_memory=True).numpy()
                           for v in views]
    else:
        state["fbs"] = ctx.framebuffers(views)
    if case["kind"] == "shards":
        state["part"] = ctx.framebuffers(views)
    if case["graph"]:
        state["stream"] = torch.cuda.Stream()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return state


def run(state):
    ctx, views, kind = state["ctx"], state["views"], state["kind"]
    if kind == "host":
        pcr.pc_render_host(ctx.h, state["cloud"], views, state["images"])
        return state["images"]
    fbs = state["fbs"]
    if kind == "frame":
        ctx.render(state["cloud"], views, fbs, state["stream"])
    elif kind == "shards":
        # the frame as two batch ranges, merged and resolved
        half = state["batches"] // 2
        ctx.render_range(state["cloud"], half, state["batches"] - half, views, state["part"])
        if half:
            ctx.render_range(state["cloud"], 0, half, views, fbs)
            for (a, _), (b, _) in zip(fbs, state["part"]):
                ctx.merge_min(a, b)
            ctx.resolve(state["cloud"], views, fbs)
        else:
            return [list(fb) for fb in state["part"]]
    elif kind == "serve":
        # one request per view, every request submitted before the first is waited for
        tickets = [pcr.pc_submit(ctx.h, state["cloud"], [v], [(a.data_ptr(), b.data_ptr())])
                   for v, (a, b) in zip(views, fbs)]
        for t in tickets:
            pcr.pc_poll(ctx.h, t)
            pcr.pc_release_ticket(ctx.h, t)
        return [b for _, b in fbs]
    elif kind == "open":
        cloud = ctx.upload(state["xyz"], state["rgba"])
        ctx.render(cloud, views, fbs)
        pcr.pc_release_cloud(ctx.h, cloud)
    return [list(fb) for fb in fbs]
