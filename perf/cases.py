"""The work a user of the renderer has it do, as cases that can be timed and compared.

Each kind of case is one call (or one step) of a user's program through the
package's public entry points; the inputs are seeded synthetic stand-ins of
the shapes in `paper_2205_14330_gb300.scenes` (surface points of random
spheres and boxes, SH coefficients around a grey DC term, log-uniform
radii), made on the GPU.

  view    render views, forward only: a novel-view viewer, an evaluation pass
  step    forward and backward through torch.autograd (`pbr.render`)
  graph   one captured training step: forward, image loss, backward
  train   one captured training iteration: forward, Eq. 8, backward, Adam
  serve   a burst of requests to the serving loop over resident scenes
  refine  one coarse-to-fine update of a point cloud (Algorithm 1)
  frame   initialisation of the next video frame (Chamfer descent, transfer)
  hull    visual-hull initialisation from silhouettes
"""
import math

import numpy as np
import torch

DEV = "cuda"


# ------------------------------------------------------------------- cases
def listed():
    return [
        # the smallest training call: 4,096 points in a box, one 128 x 128 view
        dict(name="tiny_step", kind="step", n=4096, deg=2, cloud="box", rmin=0.02, rmax=0.02,
             sizes="128x128", views=1, orbit=2.5),
        # the paper's video setting at inference: 45k points a frame, at most
        # 15 points per pixel, one camera
        dict(name="paper_view", kind="view", n=45_000, deg=2, cloud="surface", rmin=0.003,
             rmax=0.01, sizes="1024x768", views=1, orbit=4.0, cap=15),
        # a viewer's frame of a large static scene, white background
        dict(name="view_1m", kind="view", n=1_000_000, deg=3, cloud="surface", rmin=0.003,
             rmax=0.01, sizes="1920x1080", views=1, orbit=4.0, bg=1.0),
        # evaluation of a trained scene on views of odd sizes, SH directions in
        # the world frame
        dict(name="eval_ragged", kind="view", n=300_000, deg=1, cloud="surface", rmin=0.003,
             rmax=0.01, sizes="401x399,799x601,1279x719,257x1023", views=16, orbit=3.6,
             world=True),
        # a static scene's training step through autograd, default options
        dict(name="static_step", kind="step", n=500_000, deg=2, cloud="surface", rmin=0.003,
             rmax=0.01, sizes="800x800", views=4, orbit=4.0),
        # the same scene's whole training iteration, captured, default options
        dict(name="train_iter", kind="train", n=500_000, deg=2, cloud="surface", rmin=0.003,
             rmax=0.01, sizes="800x800", views=4, orbit=4.0),
        # the batched multi-view training step of the benchmark, captured, on
        # the schedule the autotuner takes for it
        dict(name="batch_step", kind="graph", n=1_000_000, deg=3, cloud="surface", rmin=0.003,
             rmax=0.01, sizes="400x400,800x800,1280x720,1920x1080", views=64, orbit=4.0,
             tile="16x32", persistent=True),
        # multi-view video: 10 frames of 200k points, 16 cameras each
        dict(name="video_step", kind="graph", n=200_000, deg=2, cloud="surface", rmin=0.003,
             rmax=0.01, sizes="1024x768", views=16, orbit=4.0, frames=10, tile="16x32",
             persistent=True),
        # a burst of requests for random cameras over four resident scenes
        dict(name="serve_burst", kind="serve", n=400_000, deg=2, cloud="surface", rmin=0.003,
             rmax=0.01, sizes="256x256,1024x768,640x480,1920x1072,480x1088,1280x720", views=16,
             orbit=4.0, frames=4),
        # the coarse-to-fine update of a trained scene
        dict(name="refine_1m", kind="refine", n=1_000_000, deg=3, vox=256, k=8),
        # the next frame of a video from the trained one
        dict(name="frame_200k", kind="frame", n=200_000, deg=2, iters=20, k=4),
        # the initial cloud of a scene from 16 silhouettes
        dict(name="hull_200k", kind="hull", n=200_000, deg=2, sizes="1024x768", views=16),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["view", "view", "step", "step", "graph", "graph", "train", "serve",
                       "refine", "frame", "hull"])
    deg = rng.randrange(4)
    if kind == "refine":
        return dict(kind=kind, n=_log_int(rng, 20_000, 1_000_000), deg=deg,
                    vox=rng.choice([64, 100, 128, 200, 256]), k=rng.randrange(4, 13))
    if kind == "frame":
        return dict(kind=kind, n=_log_int(rng, 5_000, 200_000), deg=deg,
                    iters=rng.randrange(5, 21), k=rng.randrange(1, 9))
    if kind == "hull":
        return dict(kind=kind, n=_log_int(rng, 20_000, 300_000), deg=deg,
                    sizes="%dx%d" % (_log_int(rng, 200, 1024), _log_int(rng, 200, 768)),
                    views=rng.randrange(4, 21))
    n = _log_int(rng, 4_000, 1_000_000)
    most = {"view": 16, "step": 8, "graph": 48, "train": 8, "serve": 16}[kind]
    views = max(1, min(_log_int(rng, 1, most), 30_000_000 // n))
    sizes = ",".join("%dx%d" % (_log_int(rng, 96, 1920), _log_int(rng, 96, 1080))
                     for _ in range(min(views, 4)))
    c = dict(kind=kind, n=n, deg=deg, cloud="surface", sizes=sizes, views=views,
             orbit=round(rng.uniform(3.0, 5.0), 3), rmin=0.003, rmax=0.01)
    if n < 60_000:  # fewer points are larger, as a scene is covered
        c.update(rmin=0.008, rmax=0.03)
    if kind == "serve":
        c["frames"] = rng.randrange(1, 5)
        return c
    if kind == "graph" and views <= 16 and n <= 100_000:
        c["frames"] = rng.randrange(1, 4)
    c["tile"] = rng.choice(["16x16", "16x16", "8x8", "16x32"])
    c["persistent"] = rng.random() < (0.7 if kind in ("graph", "train") else 0.3)
    if rng.random() < 0.3:
        c["world"] = True
    if rng.random() < 0.3:
        c["bg"] = 1.0
    if rng.random() < 0.2:
        c["cap"] = 15
    return c


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _uniform(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float32)


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float32)


def _rotations(r, m):
    q, up = np.linalg.qr(r.normal(size=(m, 3, 3)))
    return (q * np.sign(np.diagonal(up, axis1=1, axis2=2))[:, None, :]).astype(np.float32)


def _surface(g, r, n, shapes=20, jitter=0.005):
    """Area-weighted samples of a union of random spheres and boxes."""
    ctr = r.uniform(-1.0, 1.0, (shapes, 3))
    rad = r.uniform(0.1, 0.4, shapes)
    half = r.uniform(0.05, 0.3, (shapes, 3))
    box = np.arange(shapes) % 2 == 1
    face = np.stack([half[:, 1] * half[:, 2], half[:, 0] * half[:, 2], half[:, 0] * half[:, 1]], 1)
    area = np.where(box, 8.0 * face.sum(1), 4.0 * math.pi * rad ** 2)

    def dev(a, t=torch.float32):
        return torch.as_tensor(np.ascontiguousarray(a), dtype=t, device=DEV)

    which = torch.multinomial(dev(area), n, replacement=True, generator=g)
    v = _normal(g, n, 3)
    on_sphere = v / v.norm(dim=1, keepdim=True) * dev(rad)[which][:, None]
    u = _uniform(g, n, 3) * 2 - 1
    axis = torch.multinomial(dev(face), n, replacement=True, generator=g)
    axis = axis[which, torch.arange(n, device=DEV)]
    sign = (_uniform(g, n, 1) < 0.5).float() * 2 - 1
    u = torch.where(torch.arange(3, device=DEV)[None, :] == axis[:, None], sign, u)
    rot = dev(_rotations(r, shapes))
    local = (rot[which] * (u * dev(half)[which])[:, None, :]).sum(2)
    p = torch.where(dev(box, torch.bool)[which][:, None], local, on_sphere)
    return (p + dev(ctr)[which] + jitter * _normal(g, n, 3)).contiguous()


def _sh(g, n, deg):
    sh = 0.1 * _normal(g, n, (deg + 1) ** 2, 3)
    sh[:, 0] += 0.5 / 0.28209
    return sh


def _radii(g, n, lo, hi):
    return torch.exp(math.log(lo) + _uniform(g, n) * (math.log(hi) - math.log(lo)))


def _deform(p, r, t):
    """Smooth displacement of a frame: four sinusoidal fields, amplitude 0.05."""
    out = p.double()
    for _ in range(4):
        a = r.normal(size=3)
        a /= np.linalg.norm(a)
        w, ph = r.uniform(1.0, 4.0, 3), r.uniform(0.0, 2 * math.pi)
        arg = (p.double() * torch.as_tensor(w, device=DEV)).sum(1) + ph + t
        out = out + 0.05 * torch.sin(arg)[:, None] * torch.as_tensor(a, device=DEV)
    return out.float().contiguous()


def _camera(eye, w, h, fov=50.0):
    eye = np.asarray(eye, np.float64)
    f = -eye / np.linalg.norm(eye)
    x = np.cross(f, (0.0, 1.0, 0.0) if abs(f[1]) < 0.99 else (0.0, 0.0, 1.0))
    x /= np.linalg.norm(x)
    R = np.stack([x, np.cross(f, x), f]).astype(np.float32)
    t = (-(R.astype(np.float64) @ eye)).astype(np.float32)
    fx = np.float32((w / 2.0) / math.tan(math.radians(fov) / 2.0))
    return dict(fx=fx, fy=fx, cx=np.float32(w / 2.0), cy=np.float32(h / 2.0), R=R, t=t,
                width=int(w), height=int(h))


def _sizes(case):
    return [tuple(int(x) for x in s.split("x")) for s in case["sizes"].split(",")]


def _cameras(case, r):
    """Cameras on a Fibonacci sphere of the orbit's radius, sizes in turn."""
    n, sizes, turn = case["views"], _sizes(case), r.uniform(0.0, 2 * math.pi)
    cams = []
    for i in range(n):
        y = 0.8 * ((2 * i + 1) / n - 1.0) if n > 1 else 0.3
        s, phi = math.sqrt(1.0 - y * y), i * math.pi * (3.0 - math.sqrt(5.0)) + turn
        eye = case.get("orbit", 4.0) * np.array([s * math.cos(phi), y, s * math.sin(phi)])
        cams.append(_camera(eye, *sizes[i % len(sizes)]))
    return cams


def _scenes(case, seed):
    """[(pos, sh, opacity, radius)] of the case's frames, the cameras and each
    camera's frame."""
    g, r = _gen(seed), np.random.default_rng(seed)
    n, deg = case["n"], case["deg"]
    if case["cloud"] == "box":
        pos = _uniform(g, n, 3) * 2 - 1
    else:
        pos = _surface(g, r, n, 20 if n < 700_000 else 40)
    sh, rad = _sh(g, n, deg), _radii(g, n, case["rmin"], case["rmax"])
    op = torch.full((n,), 0.8, device=DEV)
    frames = case.get("frames", 1)
    if case["kind"] == "serve":  # scenes of their own
        pts = [(pos, sh, op, rad)]
        for k in range(1, frames):
            m = max(1000, n // (k + 1))
            pts.append((_surface(g, r, m), _sh(g, m, (deg + k) % 4),
                        torch.full((m,), 0.8, device=DEV),
                        _radii(g, m, case["rmin"], case["rmax"])))
        return pts, _cameras(case, r), [v % frames for v in range(case["views"])]
    pts, fields = [], int(r.integers(1 << 30))
    for k in range(frames):
        p = pos if frames == 1 else _deform(pos, np.random.default_rng(fields),
                                            2 * math.pi * k / 30)
        pts.append((p, sh, op, rad))
    cams = _cameras(case, r)
    return pts, cams * frames, [k for k in range(frames) for _ in cams]


def _target(cams, seed):
    """A smooth image per view, packed [sum H W, 3]."""
    r = np.random.default_rng(seed + 5)
    out = []
    for c in cams:
        x = torch.arange(c["width"], device=DEV)[None, :, None] * (6.0 / c["width"])
        y = torch.arange(c["height"], device=DEV)[:, None, None] * (6.0 / c["height"])
        ph = torch.as_tensor(r.uniform(0, 6.28, (2, 1, 1, 3)), dtype=torch.float32, device=DEV)
        out.append((0.5 + 0.25 * torch.sin(x + ph[0]) + 0.2 * torch.cos(y + ph[1]))
                   .reshape(-1, 3))
    return torch.cat(out).contiguous()


def _masks(case, r):
    """Silhouettes of eight spheres, uint8 [H, W] per camera, packed."""
    ctr = torch.as_tensor(r.uniform(-0.7, 0.7, (8, 3)), device=DEV)
    rad = torch.as_tensor(r.uniform(0.15, 0.4, 8), device=DEV)
    cams, flat = _cameras(case, r), []
    for c in cams:
        R = torch.as_tensor(c["R"], device=DEV).double()
        eye = -(R.T @ torch.as_tensor(c["t"], device=DEV).double())
        x = (torch.arange(c["width"], device=DEV) + 0.5 - float(c["cx"])) / float(c["fx"])
        y = (torch.arange(c["height"], device=DEV) + 0.5 - float(c["cy"])) / float(c["fy"])
        d = torch.stack([x[None, :].expand(len(y), -1), y[:, None].expand(-1, len(x)),
                         torch.ones(len(y), len(x), device=DEV)], -1).double() @ R
        d = d / d.norm(dim=-1, keepdim=True)
        oc = eye - ctr
        b = d @ oc.T
        hit = (b * b - ((oc * oc).sum(1) - rad * rad) >= 0).any(-1)
        flat.append(hit.reshape(-1).to(torch.uint8))
    return cams, torch.cat(flat).contiguous()


def _refine_cloud(case, seed):
    """Surface points with 1% uniform outliers among them."""
    g, r = _gen(seed), np.random.default_rng(seed)
    n, out = case["n"], case["n"] // 100
    pos = torch.cat([_surface(g, r, n - out, 40), _uniform(g, out, 3) * 3 - 1.5])
    pos = pos[torch.randperm(n, generator=g, device=DEV)].contiguous()
    return (pos, _sh(g, n, case["deg"]), torch.full((n,), 0.8, device=DEV),
            _radii(g, n, 0.003, 0.01))


def _frame_pair(case, seed):
    """A trained frame and the next frame's noisy cloud, in another order."""
    g, r = _gen(seed), np.random.default_rng(seed)
    n, f = case["n"], int(r.integers(1 << 30))
    base = _surface(g, r, n)
    p1 = _deform(base, np.random.default_rng(f), 0.0)
    p2 = _deform(base, np.random.default_rng(f), 2 * math.pi / 30) + 0.005 * _normal(g, n, 3)
    p2 = p2[torch.randperm(n, generator=g, device=DEV)].contiguous()
    return (p1, _sh(g, n, case["deg"]), torch.full((n,), 0.8, device=DEV),
            _radii(g, n, 0.003, 0.01)), p2


def _opts(pbr, case):
    kw = {}
    if case.get("tile"):
        kw["tile"] = [int(x) for x in case["tile"].split("x")]
    if case.get("persistent"):
        kw["persistent"] = 1
    if case.get("cap"):
        kw["max_per_pixel"] = case["cap"]
    if case.get("world"):
        kw["dir_frame"] = 1
    if case.get("bg"):
        kw["bg"] = [case["bg"]] * 3
    return pbr.default_opts(**kw)


# --------------------------------------------------------- prepare and run
LR_POS, LR_SH = 4e-5, 1.6e-4  # Sec. 3.3's rates after forty epochs of decay


def prepare(case, seed):
    from paper_2205_14330_gb300 import pbr
    kind = case["kind"]
    s = dict(case=case, pbr=pbr, kind=kind, R=pbr.renderer(0))
    if kind == "refine":
        pts = _refine_cloud(case, seed)
        s["scene"] = pbr.Scene(*pts, case["deg"])
        s["store"] = [torch.zeros((2 * case["n"],) + a.shape[1:], device=DEV) for a in pts]
        return s
    if kind == "frame":
        pts, s["p2"] = _frame_pair(case, seed)
        s["prev"] = pbr.Scene(*pts, case["deg"])
        return s
    if kind == "hull":
        s["cams"], s["masks"] = _masks(case, np.random.default_rng(seed))
        s["seed"] = int(seed)
        return s
    pts, cams, sov = _scenes(case, seed)
    opts = _opts(pbr, case)
    if kind == "step":
        s["leaves"] = [a.requires_grad_() for a in pts[0][:3]]
        s.update(radius=pts[0][3], cams=cams, opts=opts, target=_target(cams, seed))
        return s
    if kind == "train":  # an iteration updates the scene in place
        pts = [(p.clone(), sh.clone(), op.clone(), rad) for p, sh, op, rad in pts]
    scenes = [pbr.Scene(*p, math.isqrt(p[1].shape[1]) - 1) for p in pts]
    s.update(scenes=scenes, cams=cams, sov=sov if len(scenes) > 1 else None, opts=opts)
    if kind == "serve":
        s["R"] = pbr.Renderer(0)  # a renderer runs one serving loop
        s["server"] = pbr.Server(s["R"], opts)
        s["ids"] = [s["server"].upload(x) for x in scenes]
        s["bufs"] = [torch.empty((c["width"] * c["height"], 3), device=DEV) for c in cams]
    elif kind in ("graph", "train"):
        s["G"] = pbr.Graph(s["R"], scenes, cams, opts, scene_of_view=s["sov"],
                           target=_target(cams, seed), loss="l2")
        if kind == "train":
            s["G"].set_optimizer(kind="adam", lr_pos=LR_POS, lr_sh=LR_SH, lambda_tv=0.01)
    return s


def run(s):
    pbr, kind, case = s["pbr"], s["kind"], s["case"]
    if kind == "view":
        img, _ = s["R"].forward(s["scenes"], s["cams"], s["opts"], scene_of_view=s["sov"],
                                keep_state=False)
        return {"image": img}
    if kind == "step":
        img = pbr.render(*s["leaves"], s["radius"], case["deg"], s["cams"], s["opts"])
        loss = ((img - s["target"]) ** 2).sum()
        gp, gs, go = torch.autograd.grad(loss, s["leaves"])
        return {"image": img.detach(), "grad_pos": gp, "grad_sh": gs, "grad_opacity": go}
    if kind in ("graph", "train"):
        G = s["G"]
        G.launch(pbr.Graph.TRAIN if kind == "train" else pbr.Graph.STEP)
        out = {"image": G.out, "loss": G.loss, "grad_pos": G.grad_pos, "grad_sh": G.grad_sh,
               "grad_opacity": G.grad_opacity}
        if kind == "train":
            out.update(pos=G.scenes[0].pos, sh=G.scenes[0].sh)
        return out
    if kind == "serve":
        sv = s["server"]
        rids = [sv.submit(s["ids"][k], c, out=b)[0]
                for k, c, b in zip(s["sov"] or [0] * len(s["cams"]), s["cams"], s["bufs"])]
        return {"images": s["bufs"], "status": [sv.wait(r) for r in rids]}
    if kind == "refine":
        sc, counts = pbr.refine_points(s["R"], s["scene"], n_vox=case["vox"], k=case["k"])
        for a, b in zip(s["store"], (sc.pos, sc.sh, sc.opacity, sc.radius)):
            a[:sc.n].copy_(b)  # the trainer's parameter storage
        return dict(zip(("pos", "sh", "opacity", "radius"), s["store"]), counts=list(counts))
    if kind == "frame":  # the descent moves the new cloud in place
        sc, hist = pbr.frame_init(s["R"], s["prev"], s["p2"].clone(), iters=case["iters"],
                                  k=case["k"])
        return {"pos": sc.pos, "sh": sc.sh, "opacity": sc.opacity, "radius": sc.radius,
                "loss": np.asarray(hist)}
    pos, sh, drawn = pbr.visual_hull_init(s["R"], (-1.5,) * 3, (1.5,) * 3, s["cams"], s["masks"],
                                          case["n"], seed=s["seed"], sh_degree=case["deg"])
    return {"pos": pos, "sh": sh, "drawn": drawn}


# -------------------------------------------------------------------- work
def _pairs(case):
    """Composited (pixel, point) pairs: what the splats cover, at most about
    28 points deep in half of the pixels (what the surfaces leave visible)."""
    sizes, n = _sizes(case), case["n"]
    frames = case.get("frames", 1) if case["kind"] != "serve" else 1
    total = 0.0
    for v in range(case["views"]):
        w, h = sizes[v % len(sizes)]
        s = 1.07 * w * 0.5 * (case["rmin"] + case["rmax"]) / case["orbit"]
        total += min(n * math.pi * 9.0 * s * s, w * h * 28.0, w * h * float(case.get("cap", 1e9)))
    return total * frames


def work(case):
    """Bytes: parameters read, images (targets, gradients) and results written
    once.  Flops: 17 a composited pair forward, 37 backward; a neighbour
    search's distances to its k neighbours' cells; a candidate's projection."""
    n, K = case["n"], (case["deg"] + 1) ** 2
    point = 4.0 * (5 + 3 * K)
    kind = case["kind"]
    if kind == "refine":
        return {"bytes": 3.0 * point * n, "flops": 8.0 * 27 * n * 2}
    if kind == "frame":
        return {"bytes": case["iters"] * n * (24.0 + 12 + 84) + 2 * point * n,
                "flops": case["iters"] * 2.0 * n * 8 * 27}
    if kind == "hull":
        return {"bytes": point * n, "flops": 30.0 * 40 * n}
    frames = case.get("frames", 1)
    pix = sum(w * h for v in range(case["views"])
              for w, h in [_sizes(case)[v % len(_sizes(case))]])
    pix *= frames if kind != "serve" else 1
    pairs = _pairs(case)
    if kind in ("view", "serve"):
        return {"bytes": point * n * frames + 12.0 * pix, "flops": 17.0 * pairs}
    b = 2 * point * n * frames + 24.0 * pix
    if kind == "train":
        b += 4.0 * (3 + 3 * K) * n * 5
    return {"bytes": b, "flops": (17.0 + 37.0) * pairs}


# ------------------------------------------------------------------- exact
# The renderer's definition in plain torch: which pixels a point reaches is
# decided by the documented fp32 operations (a splat's edge is a jump), every
# value is computed in 64 bits.
SH_K = [0.28209479177387814, 0.4886025119029199, 1.0925484305920792, 0.31539156525252005,
        0.5462742152960396, 0.5900435899266435, 2.890611442640554, 0.4570457994644658,
        0.3731763325901154, 1.445305721320277]
MOST_PAIRS = 1.5e9  # (pixel, point) pairs a case may visit


def _basis(v, deg):
    x, y, z = v.unbind(1)
    a, b, c, d, e, f, h, i, j, k = SH_K
    Y = [torch.full_like(x, a)]
    if deg >= 1:
        Y += [b * y, b * z, b * x]
    if deg >= 2:
        Y += [c * x * y, c * y * z, d * (3 * z * z - 1), c * x * z, e * (x * x - y * y)]
    if deg >= 3:
        Y += [f * y * (3 * x * x - y * y), h * x * y * z, i * y * (5 * z * z - 1),
              j * z * (5 * z * z - 3), i * x * (5 * z * z - 1), k * z * (x * x - y * y),
              f * x * (x * x - 3 * y * y)]
    return torch.stack(Y, 1)


def _reach(pos, rad, cam):
    """fp32: centre, squared cutoff, depth and pixel box of every point that
    is in front of the camera and meets the image."""
    R, t = [[float(a) for a in row] for row in cam["R"]], [float(a) for a in cam["t"]]
    X = [((R[k][0] * pos[:, 0] + R[k][1] * pos[:, 1]) + R[k][2] * pos[:, 2]) + t[k]
         for k in range(3)]
    fx, fy = float(cam["fx"]), float(cam["fy"])
    px = fx * (X[0] / X[2]) + float(cam["cx"])
    py = fy * (X[1] / X[2]) + float(cam["cy"])
    rc = 3.0 * ((fx * rad) / X[2])
    W, H = cam["width"], cam["height"]
    x0, x1 = (px - rc).floor() - 1, (px + rc).ceil()
    y0, y1 = (py - rc).floor() - 1, (py + rc).ceil()
    ok = (X[2] > 0.01) & (rc > 0) & (x1 >= 0) & (x0 <= W - 1) & (y1 >= 0) & (y0 <= H - 1)
    box = [x0.clamp(0, W - 1), x1.clamp(0, W - 1), y0.clamp(0, H - 1), y1.clamp(0, H - 1)]
    return ok, px, py, rc * rc, X[2], [torch.where(ok, b, 0).long() for b in box]


def _exact_view(pts, cam, case, grad=None):
    """The image of one view in 64 bits, [H W, 3]; with `grad` (a function of
    the image), also the gradients of position, SH and opacity."""
    pos, sh, op, rad = pts
    W, H = cam["width"], cam["height"]
    ok, px, py, rc2, z, (x0, x1, y0, y1) = _reach(pos, rad, cam)
    order = torch.sort(torch.where(ok, z, math.inf), stable=True).indices[: int(ok.sum())]
    wx = (x1 - x0 + 1)[order]
    area = wx * (y1 - y0 + 1)[order]
    pix, who = [], []
    ends = torch.cumsum(area, 0)
    cuts = torch.searchsorted(ends, torch.arange(
        1, int(ends[-1].item() // 100_000_000) + 1, device=DEV) * 100_000_000).tolist() \
        if len(order) else []
    for a, b in zip([0] + cuts, cuts + [len(order)]):
        if b <= a:
            continue
        o, w, m = order[a:b], wx[a:b], area[a:b]
        rep = torch.repeat_interleave(torch.arange(b - a, device=DEV), m)
        off = torch.arange(len(rep), device=DEV) - (torch.cumsum(m, 0) - m)[rep]
        x, y = x0[o][rep] + off % w[rep], y0[o][rep] + off // w[rep]
        i = o[rep]
        ex, ey = (x.float() + 0.5) - px[i], (y.float() + 0.5) - py[i]
        keep = ex * ex + ey * ey <= rc2[i]
        pix.append((y * W + x)[keep])
        who.append(i[keep])
    pix = torch.cat(pix) if pix else torch.zeros(0, dtype=torch.long, device=DEV)
    who = torch.cat(who) if who else pix
    pix, by = torch.sort(pix.int(), stable=True)
    pix, who = pix.long(), who[by]

    p64, sh64, op64 = [a.detach().double().requires_grad_(grad is not None)
                       for a in (pos, sh, op)]
    with torch.enable_grad():
        R = torch.as_tensor(cam["R"], device=DEV).double()
        X = p64 @ R.T + torch.as_tensor(cam["t"], device=DEV).double()
        fx, fy = float(cam["fx"]), float(cam["fy"])
        c = torch.stack([fx * X[:, 0] / X[:, 2] + float(cam["cx"]),
                         fy * X[:, 1] / X[:, 2] + float(cam["cy"])], 1)
        q = (X[:, 2] / (fx * rad.double())) ** 2
        v = X / X.norm(dim=1, keepdim=True)
        col = (_basis(v @ R if case.get("world") else v, case["deg"])[:, :, None] * sh64).sum(1)
        u = torch.stack([(pix % W).double() + 0.5, (pix // W).double() + 0.5], 1)
        d2 = ((u - c[who]) ** 2).sum(1)
        al = (op64[who] * torch.exp(-0.5 * q[who] * d2)).clamp(max=float(np.float32(0.99)))
        with torch.no_grad():  # what is composited before the pixel stops
            first = torch.searchsorted(pix, torch.arange(W * H, device=DEV))[pix]
            run_ = torch.cumsum(torch.log1p(-al), 0) - torch.log1p(-al)
            use = run_ - run_[first] >= math.log(1e-5)
            if case.get("cap"):
                use &= torch.arange(len(pix), device=DEV) - first < case["cap"]
        pix, who, al = pix[use], who[use], al[use]
        lg = torch.log1p(-al)
        run_ = torch.cumsum(lg, 0) - lg
        first = torch.searchsorted(pix, torch.arange(W * H, device=DEV))[pix]
        T = torch.exp(run_ - run_[first])
        img = torch.zeros(W * H, 3, dtype=torch.float64, device=DEV)
        img = img.index_add(0, pix, (T * al)[:, None] * col[who])
        if case.get("bg"):
            end = torch.zeros(W * H, dtype=torch.float64, device=DEV).index_add(0, pix, lg)
            img = img + torch.exp(end)[:, None] * float(case["bg"])
        if grad is None:
            return img.detach()
        g = torch.autograd.grad(img, [p64, sh64, op64], grad(img.detach()))
    return img.detach(), g


def _visits(case):
    sizes, total = _sizes(case), 0.0
    for v in range(case["views"]):
        w, _ = sizes[v % len(sizes)]
        s = 1.07 * w / case["orbit"]
        total += case["n"] * (6.0 * s * 0.5 * (case["rmin"] + case["rmax"]) + 3.0) ** 2
    return total * (case.get("frames", 1) if case["kind"] == "graph" else 1)


def _tv_grad(img, w, h):
    a = img.view(h, w, 3)
    g = torch.zeros_like(a)
    for d in (0, 1):
        s = torch.sign(a.diff(dim=d))
        g.narrow(d, 1, s.shape[d]).add_(s)
        g.narrow(d, 0, s.shape[d]).sub_(s)
    return g.reshape(-1, 3)


def _exact_render(case, seed):
    pts, cams, sov = _scenes(case, seed)
    kind = case["kind"]
    if kind in ("view", "serve"):
        imgs = []
        for v, c in enumerate(cams):
            p = pts[sov[v]]
            imgs.append(_exact_view(p, c, dict(case, deg=math.isqrt(p[1].shape[1]) - 1)))
        if kind == "serve":
            return {"images": imgs, "status": [None] * len(cams)}
        return {"image": torch.cat(imgs)}
    target = _target(cams, seed).double()
    imgs, at, loss = [], 0, 0.0
    sums = [[torch.zeros(a.shape, dtype=torch.float64, device=DEV) for a in p[:3]] for p in pts]
    for v, c in enumerate(cams):
        tgt = target[at:at + c["width"] * c["height"]]
        at += len(tgt)

        def dldi(img):
            g = 2.0 * (img - tgt)
            if kind == "train":
                g = g + 0.01 * _tv_grad(img, c["width"], c["height"])
            return g

        img, g = _exact_view(pts[sov[v]], c, case, dldi)
        loss += float(((img - tgt) ** 2).sum())
        if kind == "train":
            a = img.view(c["height"], c["width"], 3)
            loss += 0.01 * float(a.diff(dim=0).abs().sum() + a.diff(dim=1).abs().sum())
        imgs.append(img)
        for a, b in zip(sums[sov[v]], g):
            a += b
    out = {"image": torch.cat(imgs), "grad_pos": torch.cat([a[0] for a in sums]),
           "grad_sh": torch.cat([a[1].reshape(-1) for a in sums]),
           "grad_opacity": torch.cat([a[2] for a in sums])}
    if kind == "step":
        out["grad_sh"] = sums[0][1]
        return out
    out["loss"] = torch.tensor([loss], dtype=torch.float64)
    if kind == "train":  # the first Adam step: its moments' bias corrections cancel
        for name, a, g, lr in (("pos", pts[0][0], sums[0][0], LR_POS),
                               ("sh", pts[0][1], sums[0][1], LR_SH)):
            out[name] = a.double() - lr * g / (g.abs() + 1e-8)
    return out


def _splitmix(seed, i):
    """SplitMix64 outputs i (int64 tensor) of stream `seed`, 24 top bits."""
    def mul(a, c):
        return a * (c - (1 << 64) if c >= 1 << 63 else c)

    def shr(a, k):
        return (a >> k) & ((1 << (64 - k)) - 1)

    z = mul(i + 1, 0x9E3779B97F4A7C15) + seed
    z = mul(z ^ shr(z, 30), 0xBF58476D1CE4E5B9)
    z = mul(z ^ shr(z, 27), 0x94D049BB133111EB)
    return shr(z ^ shr(z, 31), 40)


def _exact_hull(case, seed):
    cams, masks = _masks(case, np.random.default_rng(seed))
    kept, n, step, j = [], 0, 1 << 22, 0
    while n < case["n"] and j < 64 * step:
        i = torch.arange(j, j + step, device=DEV)
        u = torch.stack([_splitmix(seed, 3 * i + a) for a in range(3)], 1)
        p = u.float() * 2.0 ** -24 * 3.0 + -1.5
        ok, at = torch.ones(step, dtype=torch.bool, device=DEV), 0
        for c in cams:
            R, t = [[float(a) for a in r] for r in c["R"]], [float(a) for a in c["t"]]
            X = [((R[k][0] * p[:, 0] + R[k][1] * p[:, 1]) + R[k][2] * p[:, 2]) + t[k]
                 for k in range(3)]
            x = float(c["fx"]) * (X[0] / X[2]) + float(c["cx"])
            y = float(c["fy"]) * (X[1] / X[2]) + float(c["cy"])
            inside = (X[2] > 0.01) & (x >= 0) & (y >= 0) & (x < c["width"]) & (y < c["height"])
            k = torch.where(inside, y.floor().long() * c["width"] + x.floor().long(), 0)
            ok &= inside & (masks[at + k] > 0)
            at += c["width"] * c["height"]
        kept.append((u[ok].double() * 2.0 ** -24 * 3.0 - 1.5))
        n, j = n + int(ok.sum()), j + step
    if n < case["n"]:
        return None
    m = case["n"] * 3 * (case["deg"] + 1) ** 2
    c = torch.arange(m, device=DEV)
    s = seed ^ 0x5DEECE66D
    u1 = (_splitmix(s, 2 * (c >> 1)).double() + 1.0) * 2.0 ** -24
    u2 = _splitmix(s, 2 * (c >> 1) + 1).double() * 2.0 ** -24
    r = torch.sqrt(-2.0 * torch.log(u1))
    ang = 2.0 * math.pi * u2
    sh = torch.where((c & 1) == 1, r * torch.sin(ang), r * torch.cos(ang))
    return {"pos": torch.cat(kept)[:case["n"]], "sh": sh.view(case["n"], -1, 3), "drawn": None}


def _knn(p, k):
    """k nearest others of every point, fp32 distances, ties by lower index."""
    out_i, out_d = [], []
    for a in range(0, len(p), 2048):
        d = p[a:a + 2048, None, :] - p[None, :, :]
        d2 = (d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1]) + d[..., 2] * d[..., 2]
        rows = torch.arange(len(d2), device=DEV)
        d2[rows, a + rows] = math.inf
        v, i = torch.topk(d2, k, dim=1, largest=False)
        out_i.append(i)
        out_d.append(v)
    return torch.cat(out_i), torch.cat(out_d)


def _exact_refine(case, seed):
    pos, sh, op, rad = _refine_cloud(case, seed)
    if case["n"] > 100_000:
        return None  # brute-force neighbours
    n, N, k = case["n"], case["vox"], case["k"]
    lo = pos.min(0).values
    h = ((pos.max(0).values - lo).max() / float(N)).float()
    c = ((pos - lo) / h).floor().clamp(0, N - 1).long()
    ids, inv = torch.unique((c[:, 2] * N + c[:, 1]) * N + c[:, 0], return_inverse=True)
    par = torch.cat([pos, sh.reshape(n, -1), op[:, None], rad[:, None]], 1).double()
    m = torch.zeros(len(ids), par.shape[1], dtype=torch.float64, device=DEV)
    m = m.index_add(0, inv, par) / torch.bincount(inv, minlength=len(ids))[:, None]
    _, d2 = _knn(m[:, :3].float(), k)
    dist = d2.sqrt()
    dev = ((dist - dist.mean(1, keepdim=True)) ** 2).mean(1).sqrt()
    m = m[dev <= 0.01]
    i, _ = _knn(m[:, :3].float(), k)
    m = torch.cat([m, m[i].mean(1)])
    m = torch.cat([m, torch.zeros(2 * n - len(m), m.shape[1], dtype=m.dtype, device=DEV)])
    return {"pos": m[:, :3].contiguous(), "sh": m[:, 3:-2].reshape(len(m), -1, 3),
            "opacity": m[:, -2].contiguous(), "radius": m[:, -1].contiguous(),
            "counts": [None] * 3}


def exact(case, seed):
    if case["kind"] == "refine":
        return _exact_refine(case, seed)
    if case["kind"] == "frame":
        return None  # an iterated descent, nearest points by brute force
    if case["kind"] == "hull":
        return _exact_hull(case, int(seed))
    if _visits(case) > MOST_PAIRS:
        return None
    return _exact_render(case, seed)
