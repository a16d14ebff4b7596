"""The performance cases: what a user of this library has it do, through its public
entry points, with inputs made on the spot from a seed.

Scenes
  unit   one 64x48 keyframe of random targets in a unit cube, no occupancy bitfield,
         8 levels of 2^14 entries (the plain one-step workload);
  room   a 6x4x3 m room of spheres and boxes, 20 keyframes of 640x480, 16 levels of
         2^19 entries up to N = 2048, a 128^3 bitfield of the cells at a surface;
  floor  a 20x20x3 m floor of 4x4 rooms, 8 keyframes of 1200x680, 16 levels of 2^22
         entries up to N = 8192, a 256^3 bitfield (a map whose tables do not fit the L2).
Kinds
  step    one mapping step with the optimiser (optionally after a keyframe is sent
          again from pinned host memory, as the tracking window does), loss read back;
  grad    the mapping loss through torch.autograd, value and gradient;
  pose    a step that also returns the gradient of every keyframe pose;
  render  one view into device buffers; group: several views of several maps at once;
  cov     the depth variances of a bundle adjustment window, host arrays in and out.
"""

from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2210_13641_gb300 import binding
from paper_2210_13641_gb300.autograd import mapping_loss

F32 = np.float32
MLP = 9408           # weights of the two MLPs (multiply-adds per sample of one forward)
# retained samples per ray, about: the room and the floor by their bitfields (at most
# 128), the unit cube by its 32 steps
PER_RAY = {"unit": 6, "room": 60, "floor": 76}


def dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


# ---------------------------------------------------------------- the cases

def listed():
    return [
        # the smallest training call: one small keyframe, FP32 (launches and latency)
        dict(name="step_unit_fp32", kind="step", scene="unit", precision="fp32", rays=4096, upload=False),
        # the same scene with the tensor-core MLP and an odd batch
        dict(name="step_unit_fp16", kind="step", scene="unit", precision="fp16", rays=1021, upload=False),
        # the mapping loop at its ordinary batch, a keyframe sent again before every step
        dict(name="step_room_fp16", kind="step", scene="room", precision="fp16", rays=262144, upload=True),
        # continuous mapping of a served scene: smaller steps between requests
        dict(name="step_room_bf16", kind="step", scene="room", precision="bf16", rays=65536, upload=False),
        # a user's own optimiser through autograd, ragged batch
        dict(name="grad_room_fp16", kind="grad", scene="room", precision="fp16", rays=100003),
        # the plain form, as the accuracy comparison trains it
        dict(name="grad_room_fp32", kind="grad", scene="room", precision="fp32", rays=65536),
        # joint refinement of the keyframe poses
        dict(name="pose_room_fp16", kind="pose", scene="room", precision="fp16", rays=65536),
        # a building-size map: tables in HBM, the largest batch
        dict(name="step_floor_bf16", kind="step", scene="floor", precision="bf16", rays=1048576, upload=False),
        # a preview and an ordinary view of a fitted map
        dict(name="render_room_small", kind="render", scene="room", precision="bf16", width=160, height=120),
        dict(name="render_room_vga", kind="render", scene="room", precision="fp16", width=640, height=480),
        # render queries of several served scenes answered together (one of them HD)
        dict(name="render_group_hd", kind="group", scene="room", precision="fp16", width=1280, height=720, maps=3),
        # depth variances of a 20-keyframe window of the tracking frontend
        dict(name="cov_window", kind="cov", keyframes=20, pixels=4800, links=3),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "grad", "pose", "render", "group", "cov"])
    if kind == "cov":
        return dict(kind="cov", keyframes=rng.randint(2, 24), pixels=_log(rng, 37, 12000), links=rng.randint(1, 5))
    if kind in ("render", "group"):
        w = _log(rng, 64, 1280)
        c = dict(kind=kind, scene="room", precision=rng.choice(["fp16", "bf16"]), width=w,
                 height=max(33, min(800, int(w * rng.uniform(0.5, 0.8)))))
        if kind == "group":
            c["maps"] = rng.randint(2, 4)
        elif rng.random() < 0.2:
            c["precision"] = "fp32"
        return c
    scene = rng.choice(["unit", "room", "room", "floor"]) if kind != "pose" else rng.choice(["unit", "room"])
    prec = rng.choice(["fp16", "bf16", "fp16", "bf16", "fp32"])
    top = {"unit": 1 << 16, "room": 1 << 18, "floor": 1 << 19}[scene]
    c = dict(kind=kind, scene=scene, precision=prec, rays=_log(rng, 500, top // 4 if prec == "fp32" else top))
    if kind == "step":
        c["upload"] = rng.random() < 0.5
    return c


# ---------------------------------------------------------------- configurations

def config(case):
    """The field and step configuration of the case's scene."""
    scene, diag = case["scene"], lambda e: math.sqrt(sum(v * v for v in e))
    common = dict(n_features=2, enc_width=32, density_hidden=64, geo_width=16, color_hidden=64, occ_every=0,
                  occ_decay=F32(0.95), occ_thresh=F32(0.01), lambda_d=F32(1.0), lr=F32(1e-2), beta1=F32(0.9),
                  beta2=F32(0.99), eps=F32(1e-8), render_t_min=F32(1e-4), precision=case["precision"], seed=0)
    if scene == "unit":
        return SimpleNamespace(n_levels=8, log2_table=14, n_min=16, growth=1.5, n_max=None, near=F32(0.1),
                               step=F32(2.9 / 32), n_steps=32, max_samples=32, occ_res=0,
                               grid_origin=np.zeros(3, F32), grid_inv_size=F32(1.0), box_max=np.ones(3, F32), **common)
    side, extent, steps, top, log2t, res = ((6.0, (6.0, 4.0, 3.0), 1024, 2048, 19, 128) if scene == "room" else
                                            (20.0, (20.0, 20.0, 3.0), 4096, 8192, 22, 256))
    return SimpleNamespace(n_levels=16, log2_table=log2t, n_min=16, growth=None, n_max=top, near=F32(0.05),
                           step=F32(diag(extent) / steps), n_steps=steps, max_samples=128, occ_res=res,
                           grid_origin=np.zeros(3, F32), grid_inv_size=F32(1.0 / side),
                           box_max=(np.array(extent) / side).astype(F32), **common)


SHAPES = [("W1", (64, 32)), ("W2", (16, 64)), ("W3", (64, 32)), ("W4", (64, 64)), ("W5", (3, 64))]


def parameters(cfg, gen, opaque):
    """Flat parameters with the spread of a fitted map: table values of a few tenths,
    He-scaled weights; opaque: the density row is positive, so that surfaces stop rays."""
    d = dev()
    tables = (torch.rand(cfg.n_levels * (1 << cfg.log2_table) * 2, generator=gen, device=d) * 2 - 1) * 0.7
    parts = [tables]
    for name, (a, b) in SHAPES:
        w = torch.randn((a, b), generator=gen, device=d) * (0.8 * math.sqrt(2.0 / b))
        if name == "W2" and opaque:
            w[0] = w[0].abs() * 4.5
        parts.append(w.reshape(-1))
    return torch.cat(parts).to(torch.float32)


# ---------------------------------------------------------------- scenes

def _scene(case, rng):
    """Spheres [n,4] and boxes [n,6] (centre, half size) of a room or a floor of rooms."""
    if case["scene"] == "room":
        E, cells, per = np.array([6.0, 4.0, 3.0]), (1, 1), 30
    else:
        E, cells, per = np.array([20.0, 20.0, 3.0]), (4, 4), 8
    cell = E / np.array([cells[0], cells[1], 1])
    sph, box = [], []
    for i in range(cells[0]):
        for j in range(cells[1]):
            lo = np.array([i * cell[0], j * cell[1], 0.0]) + 0.2 * np.array([1, 1, 0])
            hi = lo + cell - 0.4 * np.array([1, 1, 0])
            for k in range(per):
                if k % 2:
                    h = rng.uniform(0.1, 0.5, 3)
                    box.append(np.concatenate([rng.uniform(lo + h, hi - h), h]))
                else:
                    r = rng.uniform(0.1, 0.5)
                    sph.append(np.concatenate([rng.uniform(lo + r, hi - r), [r]]))
    for a, n in ((0, cells[0]), (1, cells[1])):  # inner walls 0.1 m thick, a 1 m doorway in each segment
        for i in range(1, n):
            for j in range(cells[1 - a]):
                door = rng.uniform(0.5, cell[1 - a] - 1.5)
                for s, e in ((0.0, door), (door + 1.0, cell[1 - a])):
                    c, h = np.zeros(3), np.zeros(3)
                    c[a], h[a] = i * cell[a], 0.05
                    c[1 - a], h[1 - a] = j * cell[1 - a] + (s + e) / 2, (e - s) / 2
                    c[2], h[2] = E[2] / 2, E[2] / 2
                    box.append(np.concatenate([c, h]))
    return SimpleNamespace(E=E, sph=np.array(sph), box=np.array(box), cell=cell, cells=cells)


def _inside(sc, p, margin):
    return bool(np.any(np.linalg.norm(p - sc.sph[:, :3], axis=1) < sc.sph[:, 3] + margin) or
                np.any(np.all(np.abs(p - sc.box[:, :3]) < sc.box[:, 3:] + margin, axis=1)))


def look_at(eye, target):
    f = (target - eye) / np.linalg.norm(target - eye)
    x = np.cross([0.0, 0.0, -1.0], f)
    x /= np.linalg.norm(x)
    return np.concatenate([np.stack([x, np.cross(f, x), f], 1), eye[:, None]], 1).astype(F32)


def pose(sc, rng):
    """A camera inside one room, clear of its objects, looking at a point of that room."""
    while True:
        lo = np.array([rng.integers(sc.cells[0]) * sc.cell[0], rng.integers(sc.cells[1]) * sc.cell[1], 0.0])
        eye, tgt = (lo + rng.uniform(0.4, sc.cell - 0.4) for _ in range(2))
        if not _inside(sc, eye, 0.15) and np.linalg.norm((tgt - eye)[:2]) > 1.0:
            return look_at(eye, tgt)


def view(sc, c2w, K, W, H):
    """z-depth [H,W] and colour [H,W,3] of the scene, exact ray intersections."""
    f = dict(dtype=torch.float32, device=dev())
    u = (torch.arange(W, **f) + 0.5 - K[2]) / K[0]
    v = (torch.arange(H, **f) + 0.5 - K[3]) / K[1]
    dc = torch.stack([u[None, :].expand(H, W), v[:, None].expand(H, W), torch.ones((H, W), **f)], -1).reshape(-1, 3)
    M = torch.tensor(c2w, **f)
    d, o = dc @ M[:, :3].T, M[:, 3]
    E = torch.tensor(sc.E, **f)
    t = torch.maximum(-o / d, (E - o) / d).amin(1)
    t = torch.where(torch.isfinite(t) & (t > 0), t, torch.full_like(t, 1.0))
    a = (d * d).sum(1)
    for s in torch.tensor(sc.sph, **f):
        oc = o - s[:3]
        b, c = d @ oc, (oc * oc).sum() - s[3] ** 2
        disc = b * b - a * c
        th = (-b - disc.clamp(min=0).sqrt()) / a
        t = torch.where((disc > 0) & (th > 1e-4) & (th < t), th, t)
    for s in torch.tensor(sc.box, **f):
        t0, t1 = (s[:3] - s[3:] - o) / d, (s[:3] + s[3:] - o) / d
        tn, tf = torch.minimum(t0, t1).amax(1), torch.maximum(t0, t1).amin(1)
        t = torch.where((tn <= tf) & (tn > 1e-4) & (tn < t), tn, t)
    p = o + t[:, None] * d
    w = torch.tensor([[3.1, 5.3, 2.2], [7.7, 2.9, 4.1], [2.3, 6.1, 8.9]], **f)
    return t.reshape(H, W), (0.5 + 0.45 * torch.sin(p @ w)).reshape(H, W, 3)


def occupancy(sc, cfg):
    """Bits of the cells within 1.5 cells of a surface (x fastest), as host bytes."""
    R, f = cfg.occ_res, dict(dtype=torch.float32, device=dev())
    cell = 1.0 / (float(cfg.grid_inv_size) * R)
    g = (torch.arange(R, **f) + 0.5) * cell
    E = torch.tensor(sc.E, **f)
    out = []
    for z in torch.split(g, 32):
        p = torch.stack(torch.meshgrid(z, g, g, indexing="ij")[::-1], -1).reshape(-1, 3)
        inside = ((p > 0) & (p < E)).all(1)
        dist = torch.minimum(p, E - p).amin(1).abs()
        for s in torch.tensor(sc.sph, **f):
            dist = torch.minimum(dist, ((p - s[:3]).norm(dim=1) - s[3]).abs())
        for s in torch.tensor(sc.box, **f):
            q = (p - s[:3]).abs() - s[3:]
            dist = torch.minimum(dist, (q.clamp(min=0).norm(dim=1) + q.amax(1).clamp(max=0)).abs())
        out.append((inside & (dist < 1.5 * cell)).cpu().numpy())
    return np.packbits(np.concatenate(out), bitorder="little")


def world(case, seed):
    """Configuration, parameters, keyframes and bitfield of a case, from the seed alone."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=dev()).manual_seed(seed)
    cfg = config(case)
    w = SimpleNamespace(cfg=cfg, rng=rng, kfs=[], bits=None)
    w.params = parameters(cfg, gen, case["kind"] in ("render", "group"))
    if case["scene"] == "unit":
        q, c = rng.normal(size=(3, 3)), rng.uniform(0.2, 0.8, 3)
        Q = np.linalg.qr(q)[0]
        Q *= np.sign(np.linalg.det(Q))
        rand = lambda *s: torch.rand(s, generator=gen, device=dev())  # noqa: E731
        w.kfs = [SimpleNamespace(kf_id=0, c2w=np.concatenate([Q, c[:, None]], 1).astype(F32),
                                 K=np.array([50, 50, 32, 24], F32), W=64, H=48, rgb=rand(48, 64, 3),
                                 depth=rand(48, 64) * 2 + 0.5, var=100.0 ** (rand(48, 64) * 2 - 2),
                                 depth_is_z=False)]
        return w
    sc = w.scene = _scene(case, rng)
    w.bits = occupancy(sc, cfg)
    if case["kind"] in ("render", "group"):
        return w
    n, W, H, fx = (20, 640, 480, 525.0) if case["scene"] == "room" else (8, 1200, 680, 600.0)
    K = np.array([fx, fx, W / 2, H / 2], F32)
    for i in range(n):
        c2w = pose(sc, rng)
        z, rgb = view(sc, c2w, K, W, H)
        # depth noise growing with the depth squared, known to the mapper per pixel
        s = (0.01 * z * z * (0.5 + 1.5 * torch.rand(z.shape, generator=gen, device=z.device))).clamp(min=0.05)
        w.kfs.append(SimpleNamespace(kf_id=i, c2w=c2w, K=K, W=W, H=H, rgb=rgb.contiguous(),
                                     depth=z + s * torch.randn(z.shape, generator=gen, device=z.device), var=s * s,
                                     depth_is_z=True))
    return w


def hessian(case, seed):
    """Blocks of a bundle adjustment Hessian [[C, E], [E^T, P]]: every keyframe linked to
    `links` others, random Jacobians, a prior on the first pose."""
    rng = np.random.default_rng(seed)
    nk, n = case["keyframes"], case["pixels"]
    links = min(case["links"], nk - 1)
    C, P = np.zeros((6 * nk, 6 * nk)), np.zeros(nk * n)
    blk, e = -np.ones((nk * n, case["links"] + 1), np.int32), np.zeros((nk * n, case["links"] + 1, 6))
    for i in range(nk):
        rows = slice(i * n, (i + 1) * n)
        blk[rows, 0] = i
        for k, j in enumerate(rng.choice([x for x in range(nk) if x != i], size=links, replace=False)):
            blk[rows, k + 1] = j
            J = rng.normal(size=(n, 2, 13))
            J[..., 12] *= 3.0
            A = J * rng.uniform(0.2, 2.0, size=(n, 2, 1))
            G = A.reshape(-1, 13).T @ J.reshape(-1, 13)
            s = [slice(6 * i, 6 * i + 6), slice(6 * j, 6 * j + 6)]
            for a in range(2):
                for b in range(2):
                    C[s[a], s[b]] += G[6 * a:6 * a + 6, 6 * b:6 * b + 6]
            P[rows] += np.einsum("nr,nr->n", A[..., 12], J[..., 12])
            e[rows, 0] += np.einsum("nrc,nr->nc", A[..., :6], J[..., 12])
            e[rows, k + 1] += np.einsum("nrc,nr->nc", A[..., 6:12], J[..., 12])
    C[:6, :6] += 1e4 * np.eye(6)
    return dict(C=(C + C.T) / 2, P=P, blk=blk, e=e)


# ---------------------------------------------------------------- prepare and run

def make_map(w):
    m = binding.NerfMap(w.cfg)
    m.set_params(w.params)
    if w.bits is not None:
        m.set_occupancy(w.bits)
    for kf in w.kfs:
        m.add_keyframe(kf, rgb=kf.rgb, depth=kf.depth, var=kf.var)
    return m


def cameras(case, w, n):
    """n views of the room: the case's size, then thumbnails and half sizes."""
    out = []
    for i in range(n):
        W, H = case["width"], case["height"]
        if i:
            W, H = (160, 120) if i % 2 else (max(1, W // 2), max(1, H // 2))
        out.append((pose(w.scene, w.rng), np.array([0.82 * W, 0.82 * W, W / 2, H / 2], F32), W, H))
    return out


def prepare(case, seed):
    if case["kind"] == "cov":
        return dict(kind="cov", h=hessian(case, seed))
    w = world(case, seed)
    s = dict(kind=case["kind"], seed=seed)
    d = dev()
    if case["kind"] in ("render", "group"):
        n = 1 if case["kind"] == "render" else case["maps"]
        s["maps"] = [make_map(w)]
        for i in range(1, n):
            w.params = parameters(w.cfg, torch.Generator(device=d).manual_seed(seed + 1000 * i), True)
            s["maps"].append(make_map(w))
        s["views"] = cameras(case, w, n)
        s["outs"] = [tuple(torch.empty(sh, device=d) for sh in ((H, W, 3), (H, W), (H, W)))
                     for _, _, W, H in s["views"]]
        return s
    s["map"], s["rays"] = make_map(w), case["rays"]
    if case["kind"] == "grad":
        s["params"] = w.params.clone().requires_grad_(True)
    else:
        s["out"] = torch.empty_like(w.params)
    if case.get("upload"):
        kf = w.kfs[0]
        s["kf"] = kf
        s["host"] = {k: getattr(kf, k).cpu().contiguous().pin_memory() for k in ("rgb", "depth", "var")}
    return s


def run(s):
    kind = s["kind"]
    if kind == "cov":
        h = s["h"]
        return list(binding.marginal_covariances(h["C"], h["P"], h["blk"], h["e"]))
    if kind == "render":
        c2w, K, W, H = s["views"][0]
        s["maps"][0].render(c2w, K, W, H, *s["outs"][0])
        return list(s["outs"][0])
    if kind == "group":
        binding.render_group(s["maps"], s["views"], [o[:2] for o in s["outs"]])
        return [list(o[:2]) for o in s["outs"]]
    m = s["map"]
    if kind == "grad":
        loss = mapping_loss(s["params"], m, s["rays"], s["seed"])
        g, = torch.autograd.grad(loss, s["params"])
        return dict(loss=loss.detach(), grads=g)
    if kind == "pose":
        loss = m.step(s["rays"], s["seed"], no_update=True, pose_grad=True)
        return dict(loss=loss, pose=m.pose_grads(), grads=torch.from_numpy(m.get_grads()) if not s["out"].is_cuda
                    else m.get_grads(out=s["out"]))
    if "kf" in s:
        m.add_keyframe(s["kf"], **s["host"])
    loss = m.step(s["rays"], s["seed"])
    return dict(loss=loss, params=m.get_params(out=s["out"]))


def work(case):
    """Bytes: parameters (and for a step the two moments) read and written once, texels
    and outputs; a map larger than what the batch touches counts what it touches.
    Operations: encoding (8 corners, 2 features per level) and MLPs of every retained
    sample, three times over with the backward pass."""
    if case["kind"] == "cov":
        p, c, B = case["keyframes"] * case["pixels"], 6 * case["keyframes"], case["links"] + 1
        return dict(bytes=p * (8 + B * 52 + 8) + 16 * c * c, flops=p * B * B * 36 * 4 + c ** 3)
    cfg = config(case)
    n_param = cfg.n_levels * (2 << cfg.log2_table) + MLP
    if case["kind"] in ("render", "group"):
        views = [case["width"] * case["height"]]
        views += [19200 if i % 2 else views[0] // 4 for i in range(1, case.get("maps", 1))]
        s = sum(views) * 44  # evaluated samples: rays stop at opaque surfaces
        return dict(bytes=sum(min(4 * n_param, v * 44 * cfg.n_levels * 64) + 16 * v for v in views),
                    flops=s * (2 * MLP + cfg.n_levels * 48))
    s = case["rays"] * PER_RAY[case["scene"]]
    touched = min(n_param, s * cfg.n_levels * 16 + MLP)
    moved = 24 * n_param if case["kind"] == "step" else 4 * (touched + n_param)
    return dict(bytes=moved + 32 * case["rays"] + (20 * 307200 if case.get("upload") else 0),
                flops=3 * s * (2 * MLP + cfg.n_levels * 48))


# ---------------------------------------------------------------- the same in 64 bits
# Ray draw, ray casting and sampling decide in 32 bits, as the interface states (each
# operation rounded once); everything after those decisions is in 64 bits.

def _mix(z):
    """SplitMix64's output function on int64 tensors (wrapping products)."""
    lsr = lambda v, k: (v >> k) & ((1 << (64 - k)) - 1)  # noqa: E731
    z = z + (0x9E3779B97F4A7C15 - (1 << 64))
    z = (z ^ lsr(z, 30)) * (0xBF58476D1CE4E5B9 - (1 << 64))
    z = (z ^ lsr(z, 27)) * (0x94D049BB133111EB - (1 << 64))
    return z ^ lsr(z, 31)


def _umod(r, n):
    return ((((r >> 1) & ((1 << 63) - 1)) % n) * 2 + (r & 1)) % n


def _cast(c2w, K, u, v):
    """Origin and unit direction [n,3] of the pixels' rays; c2w [n,12] or [12], K likewise."""
    g = lambda M, i: M[..., i]  # noqa: E731
    dx = ((u.to(torch.float32) + 0.5) - g(K, 2)) / g(K, 0)
    dy = ((v.to(torch.float32) + 0.5) - g(K, 3)) / g(K, 1)
    w = [(g(c2w, 4 * a) * dx + g(c2w, 4 * a + 1) * dy) + g(c2w, 4 * a + 2) for a in range(3)]
    n = torch.sqrt((w[0] * w[0] + w[1] * w[1]) + w[2] * w[2])
    o = torch.stack([g(c2w, 4 * a + 3).expand_as(n) for a in range(3)], 1)
    return o, torch.stack([x / n for x in w], 1)


def _march(cfg, bits, o, d):
    """Retained (ray, t, grid position) of the rays, in ray order."""
    i = torch.arange(cfg.n_steps, device=o.device).to(torch.float32)
    t = float(cfg.near) + i * float(cfg.step)
    x = [((o[:, a, None] + t * d[:, a, None]) - float(cfg.grid_origin[a])) * float(cfg.grid_inv_size) for a in range(3)]
    keep = torch.ones_like(x[0], dtype=torch.bool)
    for a in range(3):
        keep &= (x[a] >= 0) & (x[a] < float(cfg.box_max[a]))
    if cfg.occ_res:
        c = [(v * float(cfg.occ_res)).floor().clamp(0, cfg.occ_res - 1).to(torch.int64) for v in x]
        keep &= bits[c[0] + cfg.occ_res * (c[1] + cfg.occ_res * c[2])]
    keep &= keep.cumsum(1) <= cfg.max_samples
    r, k = keep.nonzero(as_tuple=True)
    return r, t[k], torch.stack([v[r, k] for v in x], 1)


def _levels(cfg):
    b = cfg.growth or math.exp(math.log(cfg.n_max / cfg.n_min) / (cfg.n_levels - 1))
    return [int(math.floor(cfg.n_min * b ** l * (1.0 + 1e-9))) for l in range(cfg.n_levels)]


def _corners(cfg, N, l, x32, x64):
    """Slots [s,8] in the flat tables and weights [s,8] of a level."""
    q = x32 * float(N)
    c = q.floor().clamp(0, N - 1)
    w = (q - c).to(torch.float64)
    if x64 is not None:  # the derivative with respect to the position
        w = w + (x64 * N - (x64 * N).detach())
    c, T = c.to(torch.int64), 1 << cfg.log2_table
    slot, wt = [], []
    for k in range(8):
        b = [k & 1, (k >> 1) & 1, k >> 2]
        v = [c[:, a] + b[a] for a in range(3)]
        if (N + 1) ** 3 <= T:
            s = v[0] + (N + 1) * (v[1] + (N + 1) * v[2])
        else:
            s = (v[0] ^ (v[1] * 2654435761) ^ (v[2] * 805459861)) & (T - 1)
        slot.append(s + l * T)
        f = [w[:, a] if b[a] else 1 - w[:, a] for a in range(3)]
        wt.append(f[0] * f[1] * f[2])
    return torch.stack(slot, 1), torch.stack(wt, 1)


def _sh(d):
    x, y, z = d[:, 0], d[:, 1], d[:, 2]
    p, s = math.pi, math.sqrt
    c = [s(3 / (4 * p)), s(15 / p), s(5 / p), s(35 / (2 * p)), s(105 / p), s(21 / (2 * p)), s(7 / p)]
    return torch.stack([
        torch.full_like(x, 0.5 * s(1 / p)), -c[0] * y, c[0] * z, -c[0] * x, c[1] / 2 * x * y, -c[1] / 2 * y * z,
        c[2] / 4 * (3 * z * z - 1), -c[1] / 2 * x * z, c[1] / 4 * (x * x - y * y), -c[3] / 4 * y * (3 * x * x - y * y),
        c[4] / 2 * x * y * z, -c[5] / 4 * y * (5 * z * z - 1), c[6] / 4 * z * (5 * z * z - 3),
        -c[5] / 4 * x * (5 * z * z - 1), c[4] / 4 * z * (x * x - y * y), -c[3] / 4 * x * (x * x - 3 * y * y)], 1)


def _field(W, feat, sh):
    h = torch.relu(feat @ W[0].T) @ W[1].T
    sigma = torch.exp(h[:, 0].clamp(max=15.0))
    z = torch.relu(torch.relu(torch.cat([h, sh], 1) @ W[2].T) @ W[3].T) @ W[4].T
    return sigma, torch.sigmoid(z)


def _composite(cfg, n, r, t, sigma, rgb, t_min=0.0):
    """Colour [n,3], depth [n], opacity [n] of n rays from their samples (ray order)."""
    first = torch.searchsorted(r, torch.arange(n, device=r.device))
    k = torch.arange(r.shape[0], device=r.device) - first[r]
    tau = torch.zeros((n, cfg.max_samples), dtype=torch.float64, device=r.device)
    tau = tau.index_put((r, k), sigma * float(cfg.step))
    T = torch.exp(-(tau.cumsum(1) - tau))
    w = T * -torch.expm1(-tau)
    if t_min:
        w = torch.where((T < t_min).cumsum(1) == 0, w, torch.zeros_like(w))
    w = w[r, k]
    out = torch.zeros((n, 5), dtype=torch.float64, device=r.device)
    return out.index_add(0, r, torch.cat([w[:, None] * rgb, (w * t)[:, None], w[:, None]], 1))


def _unpack(cfg, params):
    nt = cfg.n_levels * (2 << cfg.log2_table)
    W, at = [], nt
    for _, (a, b) in SHAPES:
        W.append(params[at:at + a * b].reshape(a, b).to(torch.float64).clone())
        at += a * b
    return params[:nt].reshape(-1, 2).to(torch.float64), W


def _encode(cfg, tables, x32):
    f = torch.zeros((x32.shape[0], 32), dtype=torch.float64, device=x32.device)
    for l, N in enumerate(_levels(cfg)):
        slot, wt = _corners(cfg, N, l, x32, None)
        f[:, 2 * l:2 * l + 2] = (tables[slot] * wt[..., None]).sum(1)
    return f


def _occupied(cfg, w):
    return torch.from_numpy(np.unpackbits(w.bits, bitorder="little").astype(bool)).to(dev()) if cfg.occ_res else None


def _exact_view(cfg, w, params, cam):
    c2w, K, W, H = cam
    d = dev()
    tables, mlp = _unpack(cfg, params)
    bits, out = _occupied(cfg, w), []
    M, Kt = torch.tensor(c2w.reshape(12), device=d), torch.tensor(K, device=d)
    for pix in torch.split(torch.arange(W * H, device=d), 1 << 14):
        o, dr = _cast(M, Kt, pix % W, pix // W)
        r, t, x = _march(cfg, bits, o, dr)
        sigma, rgb = _field(mlp, _encode(cfg, tables, x), _sh(dr.to(torch.float64)[r]))
        out.append(_composite(cfg, pix.shape[0], r, t.to(torch.float64), sigma, rgb, float(cfg.render_t_min)))
    out = torch.cat(out)
    return [out[:, :3].reshape(H, W, 3), out[:, 3].reshape(H, W), out[:, 4].reshape(H, W)]


def _exact_loss(case, cfg, w, seed):
    """Loss, flat gradient and, for a pose case, the gradient of every keyframe pose."""
    d, n = dev(), case["rays"]
    want_pose = case["kind"] == "pose"
    tables, W = _unpack(cfg, w.params)
    W = [v.requires_grad_(True) for v in W]
    bits = _occupied(cfg, w)
    g_tab, g_W = torch.zeros_like(tables), [torch.zeros_like(v) for v in W]
    kf = [(k.W, k.H) for k in w.kfs]
    M = torch.tensor(np.stack([k.c2w.reshape(12) for k in w.kfs]), device=d)
    K = torch.tensor(np.stack([k.K for k in w.kfs]), device=d)
    xi = torch.zeros((len(kf), 6), dtype=torch.float64, device=d, requires_grad=True)
    g_xi, loss = torch.zeros_like(xi), 0.0
    for ray in torch.split(torch.arange(n, dtype=torch.int64, device=d), 1 << (11 if want_pose else 12)):
        slot = _umod(_mix((ray << 1) ^ seed), len(kf))
        r1 = _mix(((ray << 1) | 1) ^ seed)
        px = torch.tensor(kf, device=d)[slot]
        pix = _umod(r1, px[:, 0] * px[:, 1])
        u, v = pix % px[:, 0], pix // px[:, 0]
        o, dr = _cast(M[slot], K[slot], u, v)
        tgt, dep, var = (torch.zeros((ray.shape[0],) + s, dtype=torch.float64, device=d) for s in ((3,), (), ()))
        for j, k in enumerate(w.kfs):
            at = slot == j
            p = pix[at]
            s2 = torch.ones(p.shape[0], dtype=torch.float64, device=d)
            if k.depth_is_z:
                sx = ((p % k.W).double() + 0.5 - float(k.K[2])) / float(k.K[0])
                sy = ((p // k.W).double() + 0.5 - float(k.K[3])) / float(k.K[1])
                s2 = sx * sx + sy * sy + 1
            tgt[at] = k.rgb.reshape(-1, 3)[p].double()
            dep[at] = k.depth.reshape(-1)[p].double() * s2.sqrt()
            var[at] = k.var.reshape(-1)[p].double() * s2
        r, t, x = _march(cfg, bits, o, dr)
        x64, d64 = None, dr.to(torch.float64)
        if want_pose:
            # the pose moved by exp(xi): p -> p + rho + phi x p, d -> d + phi x d
            e = xi[slot]
            d64 = d64 + torch.linalg.cross(e[:, 3:], d64)
            o64 = o.double()
            o64 = o64 + e[:, :3] + torch.linalg.cross(e[:, 3:], o64)
            x64 = (o64[r] + t.double()[:, None] * d64[r]) * float(cfg.grid_inv_size)
        if x64 is None:
            feat = _encode(cfg, tables, x).requires_grad_(True)
        else:
            cols = []
            for l, N in enumerate(_levels(cfg)):
                sl, wt = _corners(cfg, N, l, x, x64)
                cols.append((tables[sl] * wt[..., None]).sum(1))
            feat = torch.cat(cols + [x64.new_zeros((x.shape[0], 32 - 2 * cfg.n_levels))], 1)
        sigma, rgb = _field(W, feat, _sh(d64)[r])
        out = _composite(cfg, ray.shape[0], r, t.double(), sigma, rgb)
        part = (((out[:, :3] - tgt) ** 2).sum(1) + float(cfg.lambda_d) * (out[:, 3] - dep) ** 2 / var).sum() / n
        wanted = [feat] + W + ([xi] if want_pose else [])
        grads = torch.autograd.grad(part, wanted)
        loss += float(part.detach())
        for a, b in zip(g_W, grads[1:6]):
            a += b
        if want_pose:
            g_xi += grads[6]
        for l, N in enumerate(_levels(cfg)):
            sl, wt = _corners(cfg, N, l, x, None)
            g_tab.index_add_(0, sl.reshape(-1), (wt[..., None] * grads[0][:, None, 2 * l:2 * l + 2]).reshape(-1, 2))
    return loss, torch.cat([g_tab.reshape(-1)] + [v.reshape(-1) for v in g_W]), g_xi


def exact(case, seed):
    if case["kind"] == "cov":
        h = hessian(case, seed)
        C, P, blk, e = h["C"], h["P"], h["blk"], h["e"]
        E = np.zeros((C.shape[0], P.shape[0]))
        for b in range(blk.shape[1]):
            at = np.nonzero(blk[:, b] >= 0)[0]
            for k in range(6):
                E[6 * blk[at, b] + k, at] += e[at, b, k]
        S = np.linalg.inv(C - (E / P) @ E.T)
        S = (S + S.T) / 2
        F = E / P
        return [S, 1.0 / P + np.einsum("cp,cp->p", F, S @ F)]
    if case.get("rays", 0) * (2.0 if case["kind"] == "pose" else 1.0) > 140000 and case["scene"] != "unit":
        return None  # tens of seconds in 64 bits
    if case["kind"] in ("step", "grad", "pose") and case["scene"] == "floor" and case["rays"] > 30000:
        return None
    w = world(case, seed)
    cfg = w.cfg
    if case["kind"] in ("render", "group"):
        n = 1 if case["kind"] == "render" else case["maps"]
        params = [w.params] + [parameters(cfg, torch.Generator(device=dev()).manual_seed(seed + 1000 * i), True)
                               for i in range(1, n)]
        out = [_exact_view(cfg, w, p, cam) for p, cam in zip(params, cameras(case, w, n))]
        return out[0] if case["kind"] == "render" else [v[:2] for v in out]
    loss, g, g_xi = _exact_loss(case, cfg, w, seed)
    if case["kind"] == "grad":
        return dict(loss=torch.tensor(loss, dtype=torch.float64), grads=g)
    if case["kind"] == "pose":
        return dict(loss=torch.tensor(loss, dtype=torch.float64), pose=g_xi, grads=g)
    # the first optimiser step: both moments' bias corrections cancel their (1 - beta)
    p = w.params.to(torch.float64) - float(cfg.lr) * g / (g.abs() + float(cfg.eps))
    return dict(loss=torch.tensor(loss, dtype=torch.float64), params=p)
