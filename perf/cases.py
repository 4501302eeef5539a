"""The work this framework does for its users, as measurable cases.

A mapping backend renders per-pixel surfels of indoor keyframes, refines them
against the keyframes (forward + backward), attributes errors, gates and
voxelizes new primitives, and moves maps by Sim(3) transforms.  Each case is
one such call sequence through the package's public entry points, on seeded
synthetic rooms: piecewise-planar walls and boxes seen from a camera walking
through them, one surfel per keyframe pixel (the shapes of scenes.py, built
on the GPU so that inputs are quick to make).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2604_03092_gb300.mapping import sim3_apply, voxelize
from paper_2604_03092_gb300.rasterizer import RasterConfig, Rasterizer, accum_gate, render
from paper_2604_03092_gb300.scenes import View

DEV = "cuda"
ALPHA_MIN, ALPHA_MAX, T_MIN, Z_NEAR, LOWPASS = 1.0 / 255.0, 0.99, 1e-4, 0.01, math.sqrt(0.5)


def listed():
    return [
        # a small scene of random surfels seen by one small camera: the smallest differentiable render
        dict(name="random_small", kind="random", n=4096, views=1, width=128, height=96, dist=False, ray=False),
        # all maps at once, the depth-distortion regulariser and per-pixel depth on, odd image size
        dict(name="random_dist_odd", kind="random", n=20011, views=2, width=333, height=251, dist=True, ray=True),
        # one keyframe's surfels rendered at one pose (preview, residuals): forward only
        dict(name="render_keyframe", kind="render", keyframes=1, views=1, width=512, height=384, vw=512, vh=384),
        # refinement of a single keyframe over the views around it
        dict(name="refine_keyframe8", kind="refine", keyframes=1, views=8, width=512, height=384, vw=512, vh=384,
             normals=False),
        # refinement with a normal loss, a few keyframes, odd sizes throughout
        dict(name="refine_odd_normals", kind="refine", keyframes=3, views=5, width=401, height=301, vw=347, vh=259,
             normals=True),
        # refinement of the latest keyframes' submap
        dict(name="refine_submap8", kind="refine", keyframes=8, views=8, width=512, height=384, vw=512, vh=384,
             normals=False),
        # refinement of a long submap: the largest step
        dict(name="refine_submap24", kind="refine", keyframes=24, views=24, width=512, height=384, vw=512, vh=384,
             normals=False),
        # independent submaps of uneven size refined in one batch
        dict(name="refine_uneven12", kind="uneven", submaps=12, n_min=50000, n_max=500000, layout=7),
        # map fusion at a new keyframe: render the map, attribute its errors, gate the insertion
        dict(name="fuse_map48", kind="fuse", keyframes=48, width=512, height=384, vw=640, vh=480),
        # a new keyframe's per-pixel map voxelized and moved into the world
        dict(name="insert_keyframe", kind="insert", width=512, height=384),
        # loop correction: every keyframe's surfels moved by its pose change
        dict(name="correct_map", kind="correct", n=6291456, keyframes=32),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["random", "render", "refine", "refine", "uneven", "fuse", "insert", "correct"])
    if kind == "random":
        w = _logint(rng, 64, 400)
        return dict(kind=kind, n=_logint(rng, 1000, 24000), views=rng.randint(1, 3), width=w,
                    height=max(48, int(w * rng.uniform(0.6, 0.9))), dist=rng.random() < 0.5, ray=rng.random() < 0.5)
    w = rng.randint(256, 512)
    vw = rng.randint(256, 640)
    size = dict(width=w, height=int(w * 0.75), vw=vw, vh=int(vw * rng.uniform(0.7, 0.8)))
    if kind == "render":
        return dict(kind=kind, keyframes=_logint(rng, 1, 8), views=rng.randint(1, 3), **size)
    if kind == "refine":
        k = _logint(rng, 1, 14)
        return dict(kind=kind, keyframes=k, views=rng.randint(1, min(2 * k + 4, 14)), normals=rng.random() < 0.3,
                    **size)
    if kind == "uneven":
        return dict(kind=kind, submaps=rng.randint(3, 12), n_min=rng.randint(20000, 60000),
                    n_max=rng.randint(100000, 500000), layout=rng.randint(0, 10 ** 6))
    if kind == "fuse":
        return dict(kind=kind, keyframes=_logint(rng, 4, 48), **size)
    if kind == "insert":
        return dict(kind=kind, width=rng.randint(200, 640), height=rng.randint(150, 480))
    return dict(kind="correct", n=_logint(rng, 50000, 6291456), keyframes=rng.randint(1, 64))


# ---------------------------------------------------------------------------
# scenes
# ---------------------------------------------------------------------------
class _Room:
    """Rooms side by side along x, joined by doorways, with boxes in them."""

    W, D, H = 5.0, 6.0, 2.8

    def __init__(self, rooms: int, rng: np.random.Generator, boxes: int = 10):
        rect = []  # axis, position, bounds of the two other axes
        X = rooms * self.W
        for y in (0.0, self.H):
            rect.append((1, y, 0.0, X, 0.0, self.D))
        for z in (0.0, self.D):
            rect.append((2, z, 0.0, X, 0.0, self.H))
        for r in range(rooms + 1):
            x = r * self.W
            if r in (0, rooms):
                rect.append((0, x, 0.0, self.H, 0.0, self.D))
            else:
                rect += [(0, x, 0.0, self.H, 0.0, 2.5), (0, x, 0.0, self.H, 3.5, self.D), (0, x, 2.1, self.H, 2.5, 3.5)]
        self.rect = rect
        lo, hi = [], []
        for r in range(rooms):
            for _ in range(boxes):
                s = np.array([rng.uniform(0.2, 1.0), rng.uniform(0.2, 1.4), rng.uniform(0.2, 1.0)])
                a = np.array([rng.uniform(r * self.W + 0.3, (r + 1) * self.W - 0.3 - s[0]), 0.0,
                              rng.uniform(0.3, self.D - 0.3 - s[2])])
                if rng.uniform() < 0.3:
                    a[1] = rng.uniform(0.5, max(0.6, self.H - s[1] - 0.1))
                lo.append(a)
                hi.append(a + s)
        self.lo = torch.tensor(np.array(lo), device=DEV)
        self.hi = torch.tensor(np.array(hi), device=DEV)
        t = lambda a: torch.tensor(a, device=DEV)
        self.freq = t(rng.uniform(0.8, 4.0, (3, 3, 3)) * rng.choice([-1, 1], (3, 3, 3)))
        self.phase, self.amp = t(rng.uniform(0, 2 * np.pi, (3, 3))), t(rng.uniform(0.1, 0.25, (3, 3)))
        self.base = t(rng.uniform(0.3, 0.7, (1 + rooms * boxes, 3)))

    def cast(self, eye, dirs):
        """Distance (in units of dirs) and object id of the nearest hit."""
        o = torch.tensor(eye, device=DEV)
        best = torch.full((dirs.shape[0],), 8.0, device=DEV, dtype=torch.float64)
        hit = torch.zeros(dirs.shape[0], dtype=torch.int64, device=DEV)
        for a, p, l1, h1, l2, h2 in self.rect:
            b, c = [k for k in range(3) if k != a]
            t = (p - o[a]) / dirs[:, a]
            u, v = o[b] + t * dirs[:, b], o[c] + t * dirs[:, c]
            ok = (t > 1e-6) & (t < best) & (u >= l1) & (u <= h1) & (v >= l2) & (v <= h2)
            best = torch.where(ok, t, best)
        for b in range(self.lo.shape[0]):
            t0, t1 = (self.lo[b] - o) / dirs, (self.hi[b] - o) / dirs
            tn, tf = torch.minimum(t0, t1).amax(1), torch.maximum(t0, t1).amin(1)
            ok = (tf >= tn) & (tn > 1e-6) & (tn < best)
            best = torch.where(ok, tn, best)
            hit = torch.where(ok, b + 1, hit)
        return best.clamp(0.5, 8.0), hit

    def colour(self, X, hit):
        col = self.base[hit]
        for k in range(3):
            col = col + self.amp[:, k] * torch.sin(X @ self.freq[:, k].T + self.phase[:, k])
        chk = torch.floor(X * 2).sum(1) % 2
        return (col * (0.8 + 0.4 * chk[:, None])).clamp(0.0, 1.0)


def _look(eye, yaw, pitch):
    f = np.array([math.sin(yaw), pitch, math.cos(yaw)])
    f /= np.linalg.norm(f)
    r = np.cross(f, [0.0, -1.0, 0.0])
    r /= np.linalg.norm(r)
    R = np.stack([r, np.cross(f, r), f])
    return np.concatenate([R, (-R @ eye)[:, None]], 1)


def _walk(rng, n, rooms, step=0.05, deg=2.0):
    """Camera poses of a walk: step metres and deg degrees per keyframe."""
    eye = np.array([rng.uniform(1.5, 3.5), rng.uniform(1.3, 1.6), rng.uniform(1.0, 2.0)])
    yaw, turn = rng.uniform(-0.3, 0.3), math.radians(deg) * rng.choice([-1.0, 1.0])
    out = []
    for k in range(n):
        out.append(_look(eye, yaw, 0.08 * math.sin(0.3 * k)))
        nxt = eye + step * np.array([math.sin(yaw), 0.0, math.cos(yaw)])
        if 0.6 < nxt[0] < rooms * _Room.W - 0.6 and 0.6 < nxt[2] < _Room.D - 0.6:
            eye = nxt
        else:
            yaw += 6 * turn
        yaw += turn
    return out


def _jitter(rng, Rt, deg=5.0, trans=0.2):
    a = rng.normal(size=3)
    a *= math.radians(rng.uniform(0, deg)) / np.linalg.norm(a)
    K = np.array([[0, -a[2], a[1]], [a[2], 0, -a[0]], [-a[1], a[0], 0]])
    th = np.linalg.norm(a)
    dR = np.eye(3) + math.sin(th) / th * K + (1 - math.cos(th)) / th ** 2 * (K @ K)
    d = rng.normal(size=3)
    C = -Rt[:, :3].T @ Rt[:, 3] + d / np.linalg.norm(d) * rng.uniform(0, trans)
    R = dR @ Rt[:, :3]
    return np.concatenate([R, (-R @ C)[:, None]], 1)


def _quat(R):
    """Rotation matrices [n, 3, 3] -> unit quaternions (w, x, y, z)."""
    m = [[R[:, i, j] for j in range(3)] for i in range(3)]
    four = torch.stack([1 + m[0][0] + m[1][1] + m[2][2], 1 + m[0][0] - m[1][1] - m[2][2],
                        1 - m[0][0] + m[1][1] - m[2][2], 1 - m[0][0] - m[1][1] + m[2][2]], 1)
    rows = [torch.stack([four[:, 0], m[2][1] - m[1][2], m[0][2] - m[2][0], m[1][0] - m[0][1]], 1),
            torch.stack([m[2][1] - m[1][2], four[:, 1], m[1][0] + m[0][1], m[0][2] + m[2][0]], 1),
            torch.stack([m[0][2] - m[2][0], m[1][0] + m[0][1], four[:, 2], m[2][1] + m[1][2]], 1),
            torch.stack([m[1][0] - m[0][1], m[0][2] + m[2][0], m[2][1] + m[1][2], four[:, 3]], 1)]
    pick = four.argmax(1)
    q = torch.stack(rows, 1)[torch.arange(R.shape[0], device=R.device), pick]
    return q / q.norm(dim=1, keepdim=True)


def _keyframe(room, Rt, w, h, f, gen, world=True):
    """The per-pixel surfels of one keyframe: means, scales, quats, opacity,
    rgb (float32), in the world or the keyframe's camera frame."""
    R = torch.tensor(Rt[:, :3], device=DEV)
    eye = -Rt[:, :3].T @ Rt[:, 3]
    jj, ii = torch.meshgrid(torch.arange(h, device=DEV), torch.arange(w, device=DEV), indexing="ij")
    dc = torch.stack([(ii + 0.5 - w / 2) / f, (jj + 0.5 - h / 2) / f, torch.ones_like(ii, dtype=torch.float64)], -1)
    depth, hit = room.cast(eye, dc.reshape(-1, 3).double() @ R)
    P = dc.double() * depth.view(h, w, 1)
    n = torch.linalg.cross(torch.gradient(P, dim=1)[0], torch.gradient(P, dim=0)[0])
    n = n / n.norm(dim=-1, keepdim=True).clamp_min(1e-12)
    n = torch.where(((n * P).sum(-1, keepdim=True) > 0), -n, n)
    n = torch.where(n.norm(dim=-1, keepdim=True) < 0.5, torch.tensor([0.0, 0.0, -1.0], device=DEV).double(), n)
    ex = torch.tensor([1.0, 0.0, 0.0], device=DEV).double()
    tu = ex - n[..., :1] * n
    tu = tu / tu.norm(dim=-1, keepdim=True).clamp_min(1e-9)
    cam = torch.stack([tu, torch.linalg.cross(n, tu), n], -1).reshape(-1, 3, 3)
    X = P.reshape(-1, 3)
    Xw = X @ R + torch.tensor(eye, device=DEV)
    u = torch.rand(w * h, 3, device=DEV, generator=gen, dtype=torch.float64)
    scales = (depth / f)[:, None] * (0.8 + 0.7 * u[:, :2])
    parts = (Xw if world else X, scales, _quat(R.T @ cam if world else cam), 0.5 + 0.5 * u[:, 2],
             room.colour(Xw, hit))
    return [p.float().contiguous() for p in parts]


def _view(Rt, w, h, f, off=0, cnt=-1):
    return View(w, h, f, f, w / 2.0, h / 2.0, Rt.astype(np.float32), off, cnt)


def _scene(case, seed):
    """(params, views) of a rendering case, from the seed alone."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    if case["kind"] == "random":
        n, w, h = case["n"], case["width"], case["height"]
        u = lambda *s: torch.rand(*s, device=DEV, generator=gen)
        z = lambda *s: torch.randn(*s, device=DEV, generator=gen)
        means = torch.cat([2 * u(n, 2) - 1, 2 + 2 * u(n, 1)], 1)
        prm = [means, torch.exp(math.log(0.01) + math.log(10.0) * u(n, 2)), z(n, 4), torch.sigmoid(z(n)), u(n, 3)]
        eye = np.concatenate([np.eye(3), np.zeros((3, 1))], 1)
        views = [_view(eye if v == 0 else _jitter(rng, eye, 5.0, 0.1), w, h, 100.0 * w / 128)
                 for v in range(case["views"])]
        return prm, views
    if case["kind"] == "uneven":
        prm, views, off = [], [], 0
        shapes = np.random.default_rng(case["layout"])  # the submaps' sizes belong to the case
        for _ in range(case["submaps"]):
            n = int(round(math.exp(shapes.uniform(math.log(case["n_min"]), math.log(case["n_max"])))))
            w, h = [(320, 240), (512, 384), (640, 480)][int(shapes.integers(3))]
            f = 400.0 * w / 512
            room = _Room(1, rng, 6)
            base = _walk(rng, 1, 1)[0]
            kfs = [_keyframe(room, _jitter(rng, base, 10.0, 0.3), w, h, f, gen) for _ in range(-(-n // (w * h)))]
            pick = torch.randperm(len(kfs) * w * h, device=DEV, generator=gen)[:n].sort().values
            prm.append([torch.cat([k[i] for k in kfs])[pick] for i in range(5)])
            views += [_view(_jitter(rng, base), w, h, f, off, n) for _ in range(4)]
            off += n
        return [torch.cat([p[i] for p in prm]) for i in range(5)], views
    k, w, h = case["keyframes"], case["width"], case["height"]
    vw, vh = case["vw"], case["vh"]
    rooms = 1 if k <= 3 else 3
    room = _Room(rooms, rng)
    poses = _walk(rng, k, rooms, *((0.05, 2.0) if case["kind"] != "fuse" else (0.12, 2.5)))
    kfs = [_keyframe(room, P, w, h, 400.0 * w / 512, gen) for P in poses]
    prm = [torch.cat([f[i] for f in kfs]) for i in range(5)]
    nv = case.get("views", 1)
    vp = [poses[i] if k == nv else _jitter(rng, poses[i * k // nv]) for i in range(nv)] \
        if case["kind"] != "fuse" else [_jitter(rng, poses[-1])]
    return prm, [_view(P, vw, vh, 400.0 * vw / 512) for P in vp]


def _upstream(case, views, seed):
    """Upstream gradients of the rendered maps: those of a mean L1 loss on
    colour and 0.1 of it on depth, and, where the case has them, of normal,
    alpha and distortion terms."""
    gen = torch.Generator(device=DEV).manual_seed(seed + 1)
    sizes = {(v.height, v.width) for v in views}
    P = sum(v.height * v.width for v in views)
    shp = (lambda c: ((len(views), 3) if c else (len(views),)) + next(iter(sizes))) if len(sizes) == 1 else \
        (lambda c: ((3 * P) if c else P,))
    sign = lambda s: torch.sign(torch.randn(s, device=DEV, generator=gen))
    g = [sign(shp(1)) / (3 * P), 0.1 * sign(shp(0)) / P, None, None]
    if case.get("normals") or case["kind"] == "random":
        g[2] = 0.05 * torch.randn(shp(1), device=DEV, generator=gen) / (3 * P)
    if case["kind"] == "random":
        g[3] = 0.1 * torch.randn(shp(0), device=DEV, generator=gen) / P
        if case["dist"]:
            g.append(0.05 * torch.rand(shp(0), device=DEV, generator=gen) / P)
    return g


# ---------------------------------------------------------------------------
# prepare / run
# ---------------------------------------------------------------------------
def _insert_inputs(case, seed):
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    w, h = case["width"], case["height"]
    room = _Room(1, rng)
    pose = _walk(rng, 1, 1)[0]
    m, s, q, o, c = _keyframe(room, pose, w, h, 400.0 * w / 512, gen, world=False)
    R = torch.tensor(pose[:, :3].T.copy(), device=DEV)[None]
    eye = -pose[:, :3].T @ pose[:, 3]
    row = torch.cat([_quat(R)[0], torch.tensor(eye, device=DEV), torch.tensor([rng.uniform(0.9, 1.1)], device=DEV)])
    return (m, q, s, o, c), row.float()[None].contiguous()


def _correct_inputs(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    n, k = case["n"], case["keyframes"]
    means = torch.rand(n, 3, device=DEV, generator=gen) * torch.tensor([15.0, 2.8, 6.0], device=DEV)
    quats = torch.nn.functional.normalize(torch.randn(n, 4, device=DEV, generator=gen), dim=1)
    scales = 0.001 + 0.02 * torch.rand(n, 2, device=DEV, generator=gen)
    rows = torch.cat([torch.tensor([1.0, 0.0, 0.0, 0.0], device=DEV) + 0.02 * torch.randn(k, 4, device=DEV,
                                                                                        generator=gen),
                      0.05 * torch.randn(k, 3, device=DEV, generator=gen),
                      1 + 0.02 * torch.randn(k, 1, device=DEV, generator=gen)], 1).contiguous()
    index = (torch.arange(n, device=DEV) * k // n).to(torch.int32)
    return means, quats, scales, rows, index


def prepare(case, seed):
    if case["kind"] == "insert":
        maps, row = _insert_inputs(case, seed)
        # the map's arrays, with room for all of the keyframe's primitives
        return dict(case=case, maps=maps, sim3=row, world=[torch.zeros_like(a) for a in maps],
                    block=torch.zeros(maps[3].shape[0], dtype=torch.int32, device=DEV))
    if case["kind"] == "correct":
        return dict(case=case, inputs=_correct_inputs(case, seed))
    prm, views = _scene(case, seed)
    cfg = RasterConfig.for_problem(views, prm[0].shape[0], depth_ray=bool(case.get("ray")))
    rast = Rasterizer(views, prm[0].shape[0], cfg)
    rast.forward(*prm)  # sizes the instance capacity, with room for it to grow as surfels move
    rast.set_capacity(int(rast.stats()["needed_capacity"] * 1.1) + 4096)
    st = dict(case=case, rast=rast, params=prm)
    if case["kind"] in ("random", "refine", "uneven"):
        st["params"] = [p.requires_grad_(True) for p in prm]
        st["pose"] = torch.zeros(len(views), 6, device=DEV, requires_grad=True)
        st["upstream"] = _upstream(case, views, seed)
    if case["kind"] == "fuse":
        st["keep"] = torch.zeros(rast.n_pixels, dtype=torch.int32, device=DEV)
        st["target"] = torch.rand(1, 3, views[0].height, views[0].width, device=DEV,
                                  generator=torch.Generator(device=DEV).manual_seed(seed + 2))
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "insert":
        w, h = case["width"], case["height"]
        (m, q, s, o, c), block, n_out = voxelize(*state["maps"], w, h, 0.05)
        n = int(n_out)  # the map grows by this many primitives
        sim3_apply(m[:n], q[:n], s[:n], state["sim3"])
        for dst, new in zip([*state["world"], state["block"]], (m, q, s, o, c, block)):
            dst[:n] = new[:n]
        return (*state["world"], state["block"], n)
    if kind == "correct":
        means, quats, scales, rows, index = state["inputs"]
        m, q, s = means.clone(), quats.clone(), scales.clone()  # the old map is drawn until this one is whole
        sim3_apply(m, q, s, rows, index)
        return m, q, s
    rast, prm = state["rast"], state["params"]
    if kind == "render":
        with torch.no_grad():
            return tuple(render(rast, *prm))
    if kind == "fuse":
        with torch.no_grad():
            rgb, depth, normal, alpha = render(rast, *prm)
            err = (rgb - state["target"]).abs().mean(1)
            worst = rast.max_error(err)
            keep, n_keep = accum_gate(alpha, 0.5)
            n = int(n_keep)  # primitives to insert
            state["keep"][:n] = keep[:n]
            return rgb, depth, normal, alpha, worst, state["keep"], n
    g = state["upstream"]
    out = render(rast, *prm, pose_tangent=state["pose"], check=kind == "random",
                 distortion=bool(case.get("dist")))
    live = [(o, x) for o, x in zip(out, g) if x is not None]
    grads = torch.autograd.grad([o for o, _ in live], [*prm, state["pose"]], [x for _, x in live])
    return tuple(o.detach() for o in out) + tuple(grads)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind == "insert":
        n = case["width"] * case["height"]
        return {"bytes": n * 52 + n * 56 // 3, "flops": n * 40}
    if kind == "correct":
        return {"bytes": case["n"] * (36 * 2 + 4), "flops": case["n"] * 60}
    if kind == "uneven":
        n = int(case["submaps"] * (case["n_max"] - case["n_min"]) / math.log(case["n_max"] / case["n_min"]))
        P, layers = case["submaps"] * 4 * 196608, 6 * n / (case["submaps"] * 196608)
    elif kind == "random":
        n, P = case["n"], case["views"] * case["width"] * case["height"]
        layers = 40 * n / 4096
    else:
        n = case["keyframes"] * case["width"] * case["height"]
        P, layers = case.get("views", 1) * case["vw"] * case["vh"], 6 * case["keyframes"]
    pairs = int(P * min(max(layers, 5), 150))  # blended surfels per pixel, until the pixel is opaque
    if kind in ("render", "fuse"):
        extra = n * 4 + P * 20 if kind == "fuse" else 0
        return {"bytes": n * 52 + P * 32 + extra, "flops": pairs * 45}
    maps = 4 + (3 if case.get("normals") else 0) + (4 if kind == "random" else 0) + (1 if case.get("dist") else 0)
    return {"bytes": n * 52 * 2 + P * 4 * (8 + maps + (1 if case.get("dist") else 0)), "flops": pairs * 180}


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------
def _rot(q):
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    return torch.stack([torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)], 1),
                        torch.stack([2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)], 1),
                        torch.stack([2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1)], 1)


def _depth_key(R, t, m32):
    """The single-precision camera depth surfels are sorted by: t + R20 x +
    R21 y + R22 z, each product and sum rounded once."""
    k = t[2].float().expand(m32.shape[0])
    for j in range(3):
        k = (R[2, j].double() * m32[:, j].double() + k.double()).float()
    return k


def _exact_view(view, prm, pose, ray, dist):
    """One view's (rgb, depth, normal, alpha, distortion), differentiable."""
    means, scales, quats, opacity, rgb = prm
    Rt = torch.tensor(np.asarray(view.Rt), device=DEV).double()
    R, t = Rt[:, :3], Rt[:, 3]
    W, H = view.width, view.height
    fx, fy, cx, cy = view.fx, view.fy, view.cx, view.cy

    def moved(a):  # a + phi x a
        return a + torch.linalg.cross(pose[3:].expand_as(a), a)

    with torch.no_grad():
        zkey = _depth_key(R, t, means.float())
    Rs = _rot(quats)
    mu = moved(means @ R.T + t) + pose[:3]
    U = moved(Rs[:, :, 0] @ R.T) * scales[:, :1]
    V = moved(Rs[:, :, 1] @ R.T) * scales[:, 1:]
    n = moved(Rs[:, :, 2] @ R.T)
    n = torch.where((n * mu).sum(1, keepdim=True) > 0, -n, n)
    a, b, c = torch.linalg.cross(V, mu), torch.linalg.cross(mu, U), torch.linalg.cross(U, V)
    det = (c * mu).sum(1)
    z = mu[:, 2]
    px, py = fx * mu[:, 0] / z + cx, fy * mu[:, 1] / z + cy
    with torch.no_grad():
        k2 = 2 * torch.log(opacity / np.float32(ALPHA_MIN).astype(np.float64))
        k = k2.clamp_min(0).sqrt()
        vis = (opacity >= np.float32(ALPHA_MIN).astype(np.float64)) & \
            (z - k * (U[:, 2] ** 2 + V[:, 2] ** 2).sqrt() > Z_NEAR)
        M = torch.stack([U, V, mu], 2)  # camera-frame columns; the conic of the disk u^2 + v^2 <= k^2
        K = torch.tensor([[fx, 0, cx], [0, fy, cy], [0, 0, 1.0]], device=DEV).double()
        M = K @ M
        d = torch.stack([k2, k2, -torch.ones_like(k2)], 1)
        C = lambda i, j: (M[:, i] * M[:, j] * d).sum(1)
        ex, ey = C(0, 2) / C(2, 2), C(1, 2) / C(2, 2)
        hx = (ex * ex - C(0, 0) / C(2, 2)).clamp_min(0).sqrt()
        hy = (ey * ey - C(1, 1) / C(2, 2)).clamp_min(0).sqrt()
        lp = LOWPASS * k
        x0 = torch.ceil(torch.minimum(ex - hx, px - lp) - 0.5 - 1e-3).clamp(0, W).nan_to_num(0)
        x1 = torch.floor(torch.maximum(ex + hx, px + lp) - 0.5 + 1e-3).clamp(-1, W - 1).nan_to_num(-1)
        y0 = torch.ceil(torch.minimum(ey - hy, py - lp) - 0.5 - 1e-3).clamp(0, H).nan_to_num(0)
        y1 = torch.floor(torch.maximum(ey + hy, py + lp) - 0.5 + 1e-3).clamp(-1, H - 1).nan_to_num(-1)
        w_ = torch.where(vis, (x1 - x0 + 1).clamp_min(0), 0.0).long()
        cnt = w_ * (y1 - y0 + 1).clamp_min(0).long()
        s = torch.repeat_interleave(torch.arange(cnt.shape[0], device=DEV), cnt)
        k_in = torch.arange(s.shape[0], device=DEV) - (cnt.cumsum(0) - cnt)[s]
        ix, iy = x0.long()[s] + k_in % w_[s], y0.long()[s] + k_in // w_[s]

    def weight(s, ix, iy):
        qx, qy = ix + 0.5, iy + 0.5
        rx, ry = (qx - cx) / fx, (qy - cy) / fy
        den = c[s, 0] * rx + c[s, 1] * ry + c[s, 2]
        u = (a[s, 0] * rx + a[s, 1] * ry + a[s, 2]) / den
        v = (b[s, 0] * rx + b[s, 1] * ry + b[s, 2]) / den
        ro = (u * u + v * v) / 2
        rl = ((qx - px[s]) ** 2 + (qy - py[s]) ** 2) / (2 * LOWPASS ** 2)
        obj = ro <= rl
        raw = opacity[s] * torch.exp(-torch.where(obj, ro, rl))
        return raw.clamp(max=float(np.float32(ALPHA_MAX))), obj, det[s] / den

    with torch.no_grad():
        al = weight(s, ix, iy)[0]
        keep = al >= float(np.float32(ALPHA_MIN))
        s, pix, al = s[keep], (iy * W + ix)[keep], al[keep]
        order = torch.sort(zkey[s], stable=True).indices  # ties stay in surfel order
        order = order[torch.sort(pix[order], stable=True).indices]
        s, pix, al = s[order], pix[order], al[order]
        first = torch.searchsorted(pix, torch.arange(H * W, device=DEV))
        lg = torch.log1p(-al)
        cs = lg.cumsum(0)
        before = torch.cat([cs.new_zeros(1), cs])[first[pix]]
        on = cs - before >= math.log(float(np.float32(T_MIN)))
        s, pix = s[on], pix[on]
        first = torch.searchsorted(pix, torch.arange(H * W, device=DEV))
    al, obj, zr = weight(s, pix % W, pix // W)
    cs = torch.log1p(-al).cumsum(0)
    ext = torch.cat([cs.new_zeros(1), cs])
    T = torch.exp(torch.cat([cs.new_zeros(1), cs[:-1]]) - ext[first[pix]])
    w = al * T
    zz = torch.where(obj, zr, z[s]) if ray else z[s]
    feat = torch.cat([rgb[s], zz[:, None], n[s], torch.ones_like(zz)[:, None]], 1) * w[:, None]
    img = torch.zeros(H * W, 8, device=DEV, dtype=torch.float64).index_add(0, pix, feat)
    ds = None
    if dist:
        wz = w * zz
        cz = wz.cumsum(0)
        B = torch.cat([cz.new_zeros(1), cz[:-1]]) - torch.cat([cz.new_zeros(1), cz])[first[pix]]
        ds = torch.zeros(H * W, device=DEV, dtype=torch.float64).index_add(0, pix, 2 * w * (zz * (1 - T) - B))
        ds = ds.view(H, W)
    img = img.T.reshape(8, H, W)
    return img[:3], img[3], img[4:7], img[7], ds


def _exact_render(case, seed):
    prm32, views = _scene(case, seed)
    want = case["kind"] != "render"
    prm = [p.double().requires_grad_(want) for p in prm32]
    pose = torch.zeros(len(views), 6, device=DEV, dtype=torch.float64, requires_grad=want)
    up = _upstream(case, views, seed) if want else []
    nout = 5 if case.get("dist") else 4
    outs, gsum = [[] for _ in range(nout)], None
    sizes = {(v.height, v.width) for v in views}
    off = 0
    for i, v in enumerate(views):
        lo = v.surfel_offset
        hi = prm[0].shape[0] if v.surfel_count < 0 else lo + v.surfel_count
        with torch.set_grad_enabled(want):
            im = _exact_view(v, [p[lo:hi] for p in prm], pose[i], bool(case.get("ray")), nout == 5)
        hw = v.height * v.width
        for k in range(nout):
            outs[k].append(im[k].detach())
        if want:
            loss = 0.0
            for k, g in enumerate(up):
                if g is None:
                    continue
                c = 3 if k in (0, 2) else 1
                gv = g[i] if len(sizes) == 1 else g[c * off:c * (off + hw)]
                loss = loss + (im[k].reshape(-1) * gv.double().reshape(-1)).sum()
            gr = torch.autograd.grad(loss, [*prm, pose])
            gsum = list(gr) if gsum is None else [a + b for a, b in zip(gsum, gr)]
        off += hw
    res = [torch.stack(o) if len(sizes) == 1 else torch.cat([x.reshape(-1) for x in o]) for o in outs]
    return tuple(res) + tuple(gsum or ())


def exact(case, seed):
    kind = case["kind"]
    if kind == "correct":
        means, quats, scales, rows, index = [t.double() if t.is_floating_point() else t.long()
                                             for t in _correct_inputs(case, seed)]
        return _exact_sim3(means, quats, scales, rows[index])
    if kind == "insert":
        return _exact_insert(case, seed)
    if kind == "fuse":
        return None
    if kind in ("refine", "render") and case["keyframes"] * case.get("views", 1) > 64:
        return None
    return _exact_render(case, seed)


def _exact_sim3(m, q, s, rows):
    g = rows[:, :4] / rows[:, :4].norm(dim=1, keepdim=True)
    R = _rot(g)
    m2 = rows[:, 7:] * torch.einsum("nij,nj->ni", R, m) + rows[:, 4:7]
    a, b = g.unbind(1), q.unbind(1)
    q2 = torch.stack([a[0] * b[0] - a[1] * b[1] - a[2] * b[2] - a[3] * b[3],
                      a[0] * b[1] + a[1] * b[0] + a[2] * b[3] - a[3] * b[2],
                      a[0] * b[2] - a[1] * b[3] + a[2] * b[0] + a[3] * b[1],
                      a[0] * b[3] + a[1] * b[2] - a[2] * b[1] + a[3] * b[0]], 1)
    return m2, q2, s * rows[:, 7:]


def _exact_insert(case, seed):
    (m, q, s, o, c), row = _insert_inputs(case, seed)
    w, h = case["width"], case["height"]
    bw, bh = (w + 1) // 2, (h + 1) // 2
    idx = torch.full((bh * 2, bw * 2), -1, dtype=torch.int64, device=DEV)
    idx[:h, :w] = torch.arange(w * h, device=DEV).view(h, w)
    idx = idx.view(bh, 2, bw, 2).permute(0, 2, 1, 3).reshape(-1, 4)  # block members, row-major
    has = idx >= 0
    g = idx.clamp_min(0)
    zs = m[g][..., 2]
    inf = torch.tensor(math.inf, device=DEV)
    spread = torch.where(has, zs, -inf).amax(1) - torch.where(has, zs, inf).amin(1)  # float32, as compared
    merge = ~(spread > torch.tensor(0.05, device=DEV))
    wgt = has.double()[..., None]
    mean = lambda a: (a.double()[g] * wgt).sum(1) / wgt.sum(1)
    qd = q.double()[g]
    q32 = q[g]
    sg = torch.where(((q32 * q32[:, :1]).sum(-1, keepdim=True)) >= 0, 1.0, -1.0).double()
    qs = (qd * sg * wgt).sum(1)
    qs = qs / qs.norm(dim=1, keepdim=True)
    emit = torch.where(merge[:, None], torch.tensor([True, False, False, False], device=DEV), has)
    blk = torch.arange(bw * bh, device=DEV)[:, None].expand(-1, 4)
    # a ragged block's members come first in row-major order
    out = []
    for a, merged in ((m, mean(m)), (q, qs), (s, mean(s)), (o[:, None], mean(o[:, None])), (c, mean(c))):
        v = torch.where(merge[:, None, None], merged[:, None, :], a.double()[g])
        out.append(v[emit])
    n = out[0].shape[0]
    out[:3] = _exact_sim3(out[0], out[1], out[2], row.double().expand(n, -1))
    world = [torch.cat([a, a.new_zeros(w * h - n, a.shape[1])]) for a in out]
    world[3] = world[3][:, 0]
    return (*world, torch.cat([blk[emit].int(), torch.zeros(w * h - n, dtype=torch.int32, device=DEV)]), n)
