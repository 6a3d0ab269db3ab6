"""What this renderer's users have it do, as cases that can be timed and compared.

Most cases are frames of a walk through a level-of-detail scene, rendered one
after another by a view that keeps its cut from frame to frame: a small object
viewer, a million-leaf model and the 18-million-leaf city, at image sizes from a
thumbnail to 1440p, as plain launches and as captured frames, in both storage
precisions, with the options a program picks.  The others are the rest of the
package's calls: frames whose images go to host memory, a teleport (no previous
cut to start from), many views in one call, the frame server and the standalone
pair sort.  Scenes are the weights of such a program: they are generated once,
loaded once and shared by every view; the seed of a case chooses where in the
scene the camera walks.
"""
from __future__ import annotations

import gc
import math

import numpy as np
import torch

import paper_2506_02774_gb300 as vgr
import scenegen

# Focal length in pixels per pixel of image width, tau in pixels (the workloads' own).
FOCAL = 1100.0 / 1920.0
BOX_M = 200.0  # side of the box scenes in metres (the million-leaf box; smaller ones have larger Gaussians)


def listed():
    return [
        # an object viewer's thumbnail: 4,096 leaves, 128 x 128, where launches and latency are the whole cost
        dict(name="thumbnail", kind="walk", scene="tiny", leaves=4096, width=128, height=128, tau=3.0, graph=False),
        # a small model in an odd-sized window, captured frames
        dict(name="window_60k", kind="walk", scene="box", leaves=60_000, width=801, height=603, tau=3.0, graph=True),
        # the million-leaf box at 1080p: ordinary use
        dict(name="box1m_1080p", kind="walk", scene="box", leaves=1_000_000, width=1920, height=1080, tau=3.0,
             graph=True),
        # the same scene after a jump: every frame finds its cut from the root
        dict(name="box1m_teleport", kind="walk", scene="box", leaves=1_000_000, width=1280, height=720, tau=3.0,
             graph=True, teleport=True),
        # plain launches with parent-child interpolation and the frustum-aware cut on small tiles
        dict(name="box1m_interp_frustum", kind="walk", scene="box", leaves=1_000_000, width=1366, height=768, tau=6.0,
             graph=False, interp=True, frustum=True, tile=8),
        # the city street walk at 1080p, the headline workload
        dict(name="city_1080p", kind="walk", scene="city", leaves=18_000_000, width=1920, height=1080, tau=3.0,
             graph=True),
        # the same walk in reduced storage at 1440p, coarser detail, 32-pixel tiles
        dict(name="city_half_1440p", kind="walk", scene="city", leaves=6_000_000, width=2560, height=1440, tau=4.0,
             graph=True, half=True, tile=32),
        # without the preemptive filter (3DGS-style footprints), for comparisons with other renderers
        dict(name="city_canonical_540p", kind="walk", scene="city", leaves=6_000_000, width=960, height=540, tau=6.0,
             graph=True, half=True, canonical=True),
        # a walk whose frames are all wanted in host memory
        dict(name="city_to_host", kind="host", scene="city", leaves=18_000_000, width=1920, height=1080, tau=3.0,
             frames=4),
        # eight users' views of mixed sizes in one call
        dict(name="batch_8_views", kind="batch", scene="city", leaves=6_000_000, width=1280, height=720, tau=3.0,
             views=8, half=True),
        # the frame server under full load: twelve clients, eight frames each
        dict(name="serve_12_clients", kind="serve", scene="city", leaves=6_000_000, width=640, height=360, tau=3.0,
             views=12, frames=8, half=True),
        # the pair sort as a call of its own
        dict(name="sort_4m", kind="sort", n=4_000_000, bits=32),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["small", "small", "box", "box", "city", "city", "host", "batch", "sort"])
    if kind == "sort":
        return dict(kind="sort", n=int(_log(rng, 1_000, 4_000_000)), bits=rng.randint(6, 32))
    if kind == "small":
        width = int(_log(rng, 64, 1200))
        return dict(kind="walk", scene="box", leaves=int(_log(rng, 2_000, 200_000)), width=width,
                    height=max(16, int(width * rng.uniform(0.5, 1.3))), tau=round(rng.uniform(1.0, 8.0), 2),
                    graph=rng.random() < 0.5, half=rng.random() < 0.3, tile=rng.choice([8, 16, 16, 32]),
                    interp=rng.random() < 0.2, lut=rng.random() < 0.1)
    if kind == "box":
        width = int(_log(rng, 320, 2560))
        return dict(kind="walk", scene="box", leaves=1_000_000, width=width, height=int(width * rng.uniform(0.5, 0.8)),
                    tau=round(rng.uniform(1.5, 8.0), 2), graph=rng.random() < 0.8, half=rng.random() < 0.3,
                    tile=rng.choice([8, 16, 16, 16, 32]), interp=rng.random() < 0.2, frustum=rng.random() < 0.2,
                    teleport=rng.random() < 0.2)
    width = int(_log(rng, 480, 1920))
    size = dict(width=width, height=int(width * 0.5625) + rng.randint(0, 3), tau=round(rng.uniform(3.0, 9.0), 2))
    if kind == "city":
        return dict(kind="walk", scene="city", leaves=6_000_000, graph=rng.random() < 0.8, half=rng.random() < 0.5,
                    tile=rng.choice([16, 16, 32]), interp=rng.random() < 0.15, lut=rng.random() < 0.1, **size)
    if kind == "host":
        return dict(kind="host", scene="city", leaves=6_000_000, frames=rng.randint(2, 4), half=rng.random() < 0.5,
                    **size)
    return dict(kind="batch", scene="city", leaves=6_000_000, views=rng.randint(2, 8), half=rng.random() < 0.5, **size)


# ------------------------------------------------------------- scenes and cameras
_scenes: dict = {}
_hiers: dict = {}


def _kept(store, key, most, make):
    """store[key], made on first use; the least recently used beyond `most` are dropped."""
    if key in store:
        store[key] = store.pop(key)
    else:
        while len(store) >= most:
            store.pop(next(iter(store)))
            gc.collect()
        store[key] = make()
    return store[key]


def _scene(case):
    """The host arrays of a scene, which its name and size alone decide."""
    def make():
        if case["scene"] != "box":
            return scenegen.make_scene(case["scene"], case["leaves"])
        return scenegen.build_tree(scenegen.gen_leaves(
            case["leaves"], 2, kind="box", sh_degree=3, box=(0.0, BOX_M, 0.0, BOX_M, 0.0, 0.15 * BOX_M),
            logscale=(-3.0 - math.log(case["leaves"] / 1e6) / 3.0, 0.5)))
    return _kept(_scenes, (case["scene"], case["leaves"]), 8, make)


def _hierarchy(case):
    """A program loads its scene once and keeps the handle (a view keeps its own reference)."""
    half = bool(case.get("half"))
    return _kept(_hiers, (case["scene"], case["leaves"], half), 12,
                 lambda: vgr.Hierarchy(_scene(case), vgr.STORE_HALF if half else vgr.STORE_FP32))


def _size(case, i):
    """Image size of view i: views of one call have uneven sizes."""
    if case["kind"] not in ("batch", "serve"):
        return case["width"], case["height"]
    k = (0.5, 1.0, 0.75, 1.5)[i % 4]
    return int(case["width"] * k) // 2 * 2, int(case["height"] * k) // 2 * 2


def _camera(case, seed, frame, i=0):
    """Frame `frame` of the walk of view i that `seed` chooses."""
    w, h = _size(case, i)
    seed = 1000 * seed + i
    if case["scene"] == "city":
        return scenegen.street_trajectory("city", seed, 30 + frame, w, h)
    rng = np.random.default_rng(seed)
    side = 20.0 if case["scene"] == "tiny" else BOX_M
    yaw = rng.uniform(0.0, 2.0 * math.pi)
    ahead = np.array([math.cos(yaw), math.sin(yaw), 0.0])
    # start towards the side that the camera looks away from
    start = side * (0.5 - 0.35 * ahead + np.append(rng.uniform(-0.05, 0.05, 2), 0.0))
    start[2] = side * (0.125 if case["scene"] == "tiny" else 0.05)
    return scenegen.camera(start + 0.04 * frame * ahead, yaw + 0.003 * frame, w, h, max(FOCAL * w, 40.0))


def _view(case):
    return vgr.View(_hierarchy(case), use_graph=case.get("graph", True), tile_size=case.get("tile", 16),
                    lod_interp=case.get("interp", False), lod_frustum=case.get("frustum", False),
                    filter=vgr.FILTER_CANONICAL if case.get("canonical") else vgr.FILTER_PREEMPTIVE,
                    exp_mode=vgr.EXP_LUT if case.get("lut") else vgr.EXP_EXACT, lut_size=64)


# ------------------------------------------------------------- the calls
def prepare(case, seed):
    if case["kind"] == "sort":
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        # depth-like keys: the bits of positive floats over four decades, cut to the sorted bits
        z = torch.exp(torch.rand(case["n"], generator=g, device="cuda") * math.log(1e4) + math.log(0.2))
        keys = (z.view(torch.int32) >> (32 - case["bits"])) if case["bits"] < 31 else z.view(torch.int32)
        vals = torch.randint(0, 1 << 31, (case["n"],), generator=g, device="cuda", dtype=torch.int64).to(torch.int32)
        return dict(case=case, keys=keys.contiguous(), vals=vals)
    n, frames = case.get("views", 1), case.get("frames", 2)
    state = dict(case=case, hier=_hierarchy(case), tau=case["tau"],
                 cams=[[_camera(case, seed, f, i) for f in range(frames)] for i in range(n)])
    if case["kind"] == "serve":
        state["server"] = vgr.Server(state["hier"], n, host_images=True)
        state["requests"] = [dict(client=i, arrival_s=0.0, cam=state["cams"][i][f], tau=case["tau"])
                             for f in range(frames) for i in range(n)]
        # a running server has its clients admitted
        state["server"].serve([dict(client=i, arrival_s=0.0, cam=state["cams"][i][0], tau=case["tau"])
                               for i in range(n)])
        return state
    state["views"] = [_view(case) for _ in range(n)]
    if case["kind"] == "host":
        w, h = _size(case, 0)
        # zeroed: the copies must be what fills them
        state["pinned"] = [torch.zeros((h, w, 3), dtype=torch.float32, pin_memory=True) for _ in range(frames)]
        state["host"] = [p.numpy() for p in state["pinned"]]
        state["views"][0].render(_camera(case, seed, -1), case["tau"])
        return state
    if case["kind"] == "batch":
        for f in (-2, -1):
            vgr.render_batch(state["views"], [_camera(case, seed, f, i) for i in range(n)], [case["tau"]] * n)
        return state
    for f in (-3, -2, -1):  # a walk under way: the frames before this pass's
        if case.get("teleport"):
            state["views"][0].reset()
        state["views"][0].render(_camera(case, seed, f), case["tau"])
    return state


def _held(t, state):
    """A frame's image is the view's own buffer: whoever holds it holds the view."""
    t.views = state["views"]
    return t


def run(state):
    case = state["case"]
    if case["kind"] == "sort":
        return vgr.sort_pairs(state["keys"], state["vals"], case["bits"])
    tau = state["tau"]
    if case["kind"] == "serve":
        res = state["server"].serve(state["requests"])
        return dict(images=[state["server"].client_host_image(i, c[0]["height"], c[0]["width"])
                            for i, c in enumerate(state["cams"])],
                    status=res["status"].astype(np.int64), cut_count=res["cut_count"].astype(np.int64),
                    visible_count=res["visible_count"].astype(np.int64), pair_count=res["pair_count"].astype(np.int64))
    if case["kind"] == "batch":
        n = len(state["views"])
        for f in range(2):
            res = vgr.render_batch(state["views"], [state["cams"][i][f] for i in range(n)], [tau] * n)
        return dict(images=[_held(r.image(), state) for r in res], cut=[r.cut_count for r in res],
                    visible=[r.stats["visible_count"] for r in res], pairs=[r.stats["pair_count"] for r in res])
    view = state["views"][0]
    if case["kind"] == "host":
        for cam, img in zip(state["cams"][0], state["host"]):
            r = view.render_pipelined(cam, tau, img)
        view.wait_host_images()
        return dict(images=state["host"], cut=r.cut_count)
    for cam in state["cams"][0]:  # two frames of the walk; the second is looked at
        if case.get("teleport"):
            view.reset()
        r = view.render(cam, tau)
    return dict(image=_held(r.image(), state), cut=r.cut_count, visible=r.stats["visible_count"],
                pairs=r.stats["pair_count"])


# ------------------------------------------------------------- what a pass cannot do without
def work(case):
    """Bytes: the sorted pairs in and out; or, per frame, the cut's nodes (centre,
    radius, parent's, previous and new list entry), the visible Gaussians'
    attributes and the image.  Operations: the projection and colour of the
    visible Gaussians and the blending of some twenty of them per pixel.  The
    shares of the leaves in the cut and in view are those of the scenes at
    their usual detail."""
    if case["kind"] == "sort":
        return dict(bytes=16 * case["n"], flops=0)
    cut = case["leaves"] * (0.57 if case["scene"] == "city" else 0.8) * min(1.0, 3.0 / case["tau"])
    seen = cut * (0.48 if case["scene"] == "city" else 0.35)
    sh = 12 if case["scene"] == "tiny" else 192
    per_seen = 48 + sh if not case.get("half") else 40 + sh // 2
    total = dict(bytes=0.0, flops=0.0)
    n, frames = case.get("views", 1), case.get("frames", 2)
    for i in range(n):
        w, h = _size(case, i)
        total["bytes"] += frames * (44.0 * cut + per_seen * seen + 12.0 * w * h)
        total["flops"] += frames * (400.0 * seen + 20.0 * 20.0 * w * h)
    return total


# ------------------------------------------------------------- the same in 64 bits
def _cut64(sc, cam, tau, boxes):
    """The cut's node ids, ascending: the granularity test is defined in
    single-rounded FP32, so the cut is an integer result."""
    dev = "cuda"
    f32 = torch.float32
    mean = torch.from_numpy(sc["mean"]).to(dev)
    rad2 = torch.from_numpy(sc["radius2"]).to(dev)
    first = torch.from_numpy(sc["first_child"].view(np.int32)).to(dev).long()
    nchild = torch.from_numpy(sc["n_child"]).to(dev).long()
    pos = torch.tensor(np.asarray(cam["pos"], np.float32), device=dev)
    t = np.float32(tau) / max(np.float32(cam["fx"]), np.float32(cam["fy"]))
    k = torch.tensor(np.float32(t * t), device=dev, dtype=f32)
    planes = _planes(cam) if boxes else None
    box = torch.from_numpy(sc["bbox"]).to(dev) if boxes else None
    front = torch.zeros(1, dtype=torch.long, device=dev)
    out = []
    while front.numel():
        d = pos - mean[front]
        d2 = (d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]) + d[:, 2] * d[:, 2]
        expand = (nchild[front] > 0) & (d2 * k < rad2[front])
        if boxes:
            b = box[front]
            for w0, w1, w2, o in planes:
                x = b[:, 3] if w0 >= 0 else b[:, 0]
                y = b[:, 4] if w1 >= 0 else b[:, 1]
                z = b[:, 5] if w2 >= 0 else b[:, 2]
                expand &= ((float(w0) * x + float(w1) * y) + float(w2) * z) - float(o) >= 0
        out.append(front[~expand])
        p = front[expand]
        c = nchild[p]
        at = torch.repeat_interleave(first[p] - (torch.cumsum(c, 0) - c), c)
        front = at + torch.arange(at.numel(), device=dev)
    return torch.sort(torch.cat(out))[0]


def _planes(cam, guard=2.0):
    """World planes of the frustum-aware cut: near, and the image edges moved out by the guard."""
    R, pos = np.asarray(cam["R"], np.float64), np.asarray(cam["pos"], np.float64)
    fx, fy, cx, cy = (float(cam[k]) for k in ("fx", "fy", "cx", "cy"))
    w, h = cam["width"], cam["height"]
    out = []
    for a, o in (((0, 0, 1), float(cam["z_near"])), ((fx, 0, cx + guard), 0), ((-fx, 0, w - cx + guard), 0),
                 ((0, fy, cy + guard), 0), ((0, -fy, h - cy + guard), 0)):
        n = (R.T @ np.asarray(a, np.float64)).astype(np.float32)
        out.append((n[0], n[1], n[2], np.float32(n.astype(np.float64) @ pos + o)))
    return out


def _sh64(d, sh):
    """Real spherical harmonics (orthonormal, Condon-Shortley phase) times coefficients, + 1/2, clamped at 0."""
    x, y, z = d.unbind(1)
    pi = math.pi
    Y = [torch.full_like(x, 0.5 / math.sqrt(pi))]
    if sh.shape[1] > 1:
        c = math.sqrt(3 / (4 * pi))
        Y += [-c * y, c * z, -c * x]
    if sh.shape[1] > 4:
        c, e, g = math.sqrt(15 / (4 * pi)), math.sqrt(5 / (16 * pi)), math.sqrt(15 / (16 * pi))
        Y += [c * x * y, -c * y * z, e * (3 * z * z - 1), -c * x * z, g * (x * x - y * y)]
    if sh.shape[1] > 9:
        a, b = math.sqrt(35 / (32 * pi)), math.sqrt(105 / (4 * pi))
        c, e, g = math.sqrt(21 / (32 * pi)), math.sqrt(7 / (16 * pi)), math.sqrt(105 / (16 * pi))
        Y += [-a * y * (3 * x * x - y * y), b * x * y * z, -c * y * (5 * z * z - 1), e * z * (5 * z * z - 3),
              -c * x * (5 * z * z - 1), g * z * (x * x - y * y), -a * x * (x * x - 3 * y * y)]
    return torch.clamp(torch.einsum("nk,nkc->nc", torch.stack(Y, 1), sh) + 0.5, min=0.0)


def _image64(sc, cam, tau, half, boxes):
    """One frame as the method defines it: cut, EWA projection, depth order, front-to-back blending, in 64 bits."""
    dev, f64 = "cuda", torch.float64
    W, H = cam["width"], cam["height"]
    cut = _cut64(sc, cam, tau, boxes)
    R32 = torch.tensor(np.asarray(cam["R"], np.float32).reshape(9), device=dev)
    C32 = torch.tensor(np.asarray(cam["pos"], np.float32), device=dev)
    mean = torch.from_numpy(sc["mean"]).to(dev)[cut]
    d = mean - C32
    key = (R32[6] * d[:, 0] + R32[7] * d[:, 1]) + R32[8] * d[:, 2]  # FP32: it decides the order
    theta = torch.from_numpy(sc["opacity"]).to(dev)[cut]
    keep = (key > float(cam["z_near"])) & (theta >= 1.0 / 255.0)
    cut, mean, key, theta = cut[keep], mean[keep], key[keep], theta[keep].to(f64)
    ids = cut.cpu().numpy()
    cov = torch.from_numpy(sc["cov6"][ids]).to(dev)
    if half:
        cov = cov.to(torch.bfloat16)
    cov = cov.to(f64)
    R, C = R32.to(f64).reshape(3, 3), C32.to(f64)
    p = (mean.to(f64) - C) @ R.T
    z = p[:, 2]
    fx, fy, cx, cy = (float(cam[k]) for k in ("fx", "fy", "cx", "cy"))
    xz, yz = p[:, 0] / z, p[:, 1] / z
    u, v = fx * xz + cx, fy * yz + cy
    lx, ly = 1.3 * (0.5 * W / fx), 1.3 * (0.5 * H / fy)
    M0 = (fx / z)[:, None] * (R[0] - torch.clamp(xz, -lx, lx)[:, None] * R[2])
    M1 = (fy / z)[:, None] * (R[1] - torch.clamp(yz, -ly, ly)[:, None] * R[2])
    S = cov[:, [0, 1, 2, 1, 3, 4, 2, 4, 5]].reshape(-1, 3, 3)
    s00 = torch.einsum("ni,nij,nj->n", M0, S, M0) + 0.3
    s01 = torch.einsum("ni,nij,nj->n", M0, S, M1)
    s11 = torch.einsum("ni,nij,nj->n", M1, S, M1) + 0.3
    det = s00 * s11 - s01 * s01
    r2 = 2.0 * torch.log(theta * 255.0)
    bx, by = torch.sqrt(r2 * s00), torch.sqrt(r2 * s11)
    x0 = torch.clamp(torch.ceil(u - bx - 0.5), min=0).long()
    x1 = torch.clamp(torch.floor(u + bx - 0.5), max=W - 1).long()
    y0 = torch.clamp(torch.ceil(v - by - 0.5), min=0).long()
    y1 = torch.clamp(torch.floor(v + by - 0.5), max=H - 1).long()
    sel = torch.nonzero((x0 <= x1) & (y0 <= y1) & (det > 0)).flatten()
    sel = sel[torch.sort(key[sel], stable=True)[1]]  # ascending id within equal keys
    sh = torch.from_numpy(sc["sh"][ids[sel.cpu().numpy()]]).to(dev)
    if half:
        sh = sh.to(torch.float16)
    rgb = torch.empty((sel.numel(), 3), device=dev, dtype=f64)
    for b in range(0, sel.numel(), 1 << 20):
        q = sel[b:b + (1 << 20)]
        dv = mean[q].to(f64) - C
        rgb[b:b + (1 << 20)] = _sh64(dv / dv.norm(dim=1, keepdim=True), sh[b:b + (1 << 20)].to(f64))
    u, v, x0, x1, y0, y1, theta = (a[sel] for a in (u, v, x0, x1, y0, y1, theta))
    A, B, Cc = s11[sel] / det[sel], -s01[sel] / det[sel], s00[sel] / det[sel]
    img = torch.zeros((H * W, 3), device=dev, dtype=f64)
    rows = max(1, (1 << 16) // W)
    for r0 in range(0, H, rows):  # a band of rows at a time
        r1 = min(H, r0 + rows) - 1
        g = torch.nonzero((y0 <= r1) & (y1 >= r0)).flatten()
        ya, yb = torch.clamp(y0[g], min=r0), torch.clamp(y1[g], max=r1)
        nx = x1[g] - x0[g] + 1
        cnt = nx * (yb - ya + 1)
        if not g.numel():
            continue
        own = torch.repeat_interleave(torch.arange(g.numel(), device=dev), cnt)
        loc = torch.arange(own.numel(), device=dev) - (torch.cumsum(cnt, 0) - cnt)[own]
        py = ya[own] + loc // nx[own]
        px = x0[g][own] + loc % nx[own]
        gi = g[own]
        dx, dy = u[gi] - (px + 0.5), v[gi] - (py + 0.5)
        alpha = theta[gi] * torch.exp(-0.5 * (A[gi] * dx * dx + Cc[gi] * dy * dy) - B[gi] * dx * dy)
        hit = alpha >= 1.0 / 255.0
        pix, gi, alpha = (py * W + px)[hit], gi[hit], torch.clamp(alpha[hit], max=0.99)
        del own, loc, py, px, dx, dy, hit
        pix, at = torch.sort(pix, stable=True)  # front to back within a pixel
        gi, alpha = gi[at], alpha[at]
        if not pix.numel():
            continue
        lg = torch.log1p(-alpha)
        inc = torch.cumsum(lg, 0)
        start = torch.cat([torch.ones(1, dtype=torch.bool, device=dev), pix[1:] != pix[:-1]])
        head = torch.cummax(torch.where(start, torch.arange(pix.numel(), device=dev), 0), 0)[0]
        before = inc - lg
        T = torch.exp(before - before[head])
        go = T * (1.0 - alpha) >= 1e-4  # the first that falls below stops its pixel
        img.index_add_(0, pix[go], (alpha * T)[go, None] * rgb[gi[go]])
    return img.reshape(H, W, 3)


def exact(case, seed):
    # whole numbers have no other value; an interpolated Gaussian, the unfiltered
    # footprint and the table are variants of their own, without a value in 64 bits here
    if case["kind"] == "sort" or case.get("interp") or case.get("canonical") or case.get("lut"):
        return None
    sc = _scene(case)
    half, boxes = bool(case.get("half")), bool(case.get("frustum"))

    def image(f, i=0):
        return _image64(sc, _camera(case, seed, f, i), case["tau"], half, boxes)

    if case["kind"] == "host":
        n = case.get("frames", 2)
        return dict(images=[image(f).cpu() if f == n - 1 else None for f in range(n)], cut=None)
    if case["kind"] == "batch":
        n = case["views"]
        return dict(images=[image(1, i) if i < 2 else None for i in range(n)], cut=[None] * n, visible=[None] * n,
                    pairs=[None] * n)
    if case["kind"] == "serve":
        n = case["views"]
        return dict(images=[image(case["frames"] - 1, i).cpu() if i < 2 else None for i in range(n)], status=None,
                    cut_count=None, visible_count=None, pair_count=None)
    return dict(image=image(1), cut=None, visible=None, pairs=None)
