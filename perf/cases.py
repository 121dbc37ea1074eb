"""Performance cases of the DRR splatting framework.

Each case is one pass through the package's public entry points on synthetic
CT-phantom inputs: a forward render, a render with its loss and backward pass,
a batch of uneven requests, or the RADS initialisation of a volume. `listed()`
names the cases, `draw(rng)` gives more of the same ranges, `prepare(case,
seed)` makes what a program holds before the call, `run(state)` is one pass,
`work(case)` what the pass cannot do without, and `exact(case, seed)` the same
outputs in 64 bits from plain torch, without the package.
"""
import math

import numpy as np
import torch

FOV, SDD, SID = 256.0, 1020.0, 816.0  # mm: phantom cube, source to detector, source to isocenter
BODY = (100.0, 80.0, 120.0)           # mm: semi-axes of the phantom's body
Q_MAX, ALPHA_MIN, ALPHA_MAX, T_MIN = 9.0, 1.0 / 255.0, 0.99, 1e-4
CLOUD = ("means", "log_scales", "quats", "opacity_logits", "feat_iso", "feat_dir", "b_iso", "B_dir")
GRADS = CLOUD + ("world_to_cam",)


def _case(name, kind, gaussians, views, height, width, **more):
    c = dict(kind=kind, scene="phantom", grid=256, gaussians=gaussians, views=views, height=height,
             width=width, poses="registration", k=8, degree=1, entangled=False, per_pixel=False,
             bf16=False, tile=8, depth=32, dilation=0.3, no_sync=False)
    c.update(more)
    return dict({"name": name}, **c) if name else c


def _rads(name, nx, ny, nz, n1=15000, n2=10000):
    c = dict(kind="rads", nx=nx, ny=ny, nz=nz, n1=n1, n2=n2)
    return dict({"name": name}, **c) if name else c


def listed():
    return [
        # an interactive viewer's frame: one small view of a small cloud at the default launch shape
        _case("render-4k-128", "render", 4096, 1, 128, 128, scene="cube", tile=16, depth=256),
        # one pose of a registration by a program that renders candidates one at a time, with a
        # cloud of the size that trained models have
        _case("pose-14k-1x256", "pose", 14478, 1, 256, 256, grid=128),
        # a fitting step of one radiograph: gradients of every parameter
        _case("fit-100k-1x512", "fit", 100_000, 1, 512, 512, grid=128, poses="orbit"),
        # the same through autograd at the default launch shape, several views of an odd size
        _case("autograd-100k-3x375x501", "autograd", 100_000, 3, 375, 501, grid=128, poses="orbit",
              tile=16, depth=256),
        # a batched registration step: many candidate poses of one patient, pose gradients
        _case("pose-500k-64x256", "pose", 500_000, 64, 256, 256, no_sync=True),
        # the same in the coarse first stage of a registration: a small, blurred detector
        _case("pose-500k-64x64-coarse", "pose", 500_000, 64, 64, 64, dilation=1.5, no_sync=True),
        # a large fitting step, direction-dependent features held in bfloat16
        _case("fit-2m-8x1024-bf16", "fit", 2_000_000, 8, 1024, 1024, grid=512, poses="orbit",
              bf16=True),
        # a serving batch: requests with clouds and detectors of very different sizes
        _case("batch-24-uneven", "batch", 24, 1, 128, 1024, grid=512, no_sync=True),
        # ray angles taken per pixel (a variant of the radiosity), all gradients
        _case("pixel-rays-200k-8x256", "fit", 200_000, 8, 256, 256, per_pixel=True),
        # both radiosity terms in every Gaussian, more features and a higher degree
        _case("entangled-k16-l3-100k-4x256", "fit", 100_000, 4, 256, 256, k=16, degree=3,
              entangled=True, tile=16, depth=256),
        # initialisation from a clinical volume
        _rads("rads-512", 512, 512, 512),
        # and from a cropped one with rows of no whole vectors
        _rads("rads-301x277x190", 301, 277, 190),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["render", "pose", "pose", "fit", "fit", "autograd", "batch", "variant", "rads"])
    if kind == "rads":
        return _rads(None, rng.randint(60, 512), rng.randint(60, 512), rng.randint(60, 400),
                     _log_int(rng, 2000, 20000), _log_int(rng, 1000, 12000))
    tile, depth = rng.choice([(8, 32), (8, 32), (16, 32), (16, 256)])
    if kind == "batch":
        return _case(None, "batch", rng.randint(3, 24), 1, rng.choice([96, 128, 200]),
                     rng.choice([512, 700, 1024]), grid=512, no_sync=rng.random() < 0.5,
                     tile=tile, depth=depth)
    n = _log_int(rng, 3000, 700_000)
    grid = 128 if n < 120_000 else 256
    views = _log_int(rng, 1, 48)
    side = _log_int(rng, 60, 700)
    # no more pixels, records or expected pixel pairs than the largest listed case
    while views > 1 and (views * side * side > 2_000_000 or views * n > 12_000_000
                         or views * n * max(4.0, (2.0 * grid / 128 * side / 256) ** 2) > 1.5e8):
        views = views // 2
    more = dict(grid=grid, poses=rng.choice(["registration", "orbit"]), tile=tile, depth=depth,
                dilation=rng.choice([0.3, 0.3, 0.8]), no_sync=rng.random() < 0.3)
    if kind == "variant":
        kind = "fit"
        if rng.random() < 0.5:
            more.update(per_pixel=True, entangled=rng.random() < 0.5)
        else:
            more.update(k=rng.choice([4, 16, 32]), degree=rng.choice([1, 2, 3]),
                        entangled=rng.random() < 0.5, bf16=rng.random() < 0.5)
    elif kind == "fit":
        more.update(bf16=rng.random() < 0.4)
    if kind == "autograd":
        more.update(no_sync=False)
    return _case(None, kind, n, views, side, max(40, int(side * rng.uniform(0.7, 1.3))), **more)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _rot(axis, a):
    c, s = math.cos(a), math.sin(a)
    i, j = [(1, 2), (2, 0), (0, 1)][axis]
    R = np.eye(3)
    R[i, i], R[i, j], R[j, i], R[j, j] = c, -s, s, c
    return R


def _structures(rng):
    """Ellipsoids (kind, centre, semi-axes, rotation, HU) inside the body: organs, bone shells
    with a 5 mm wall, and small lesions."""
    body, out = np.array(BODY), []
    for kind, count, lo, hi in (("organ", 6, 15, 40), ("bone", 4, 20, 60), ("lesion", 8, 3, 15)):
        for _ in range(count):
            ax = rng.uniform(lo, hi, 3) if kind != "lesion" else np.full(3, rng.uniform(lo, hi))
            lim = np.maximum(body - ax, 5.0) * 0.6
            R = _rot(2, rng.uniform(0, 6.28)) @ _rot(1, rng.uniform(0, 3.14)) @ _rot(0, rng.uniform(0, 6.28))
            hu = rng.uniform(400, 1500) if kind == "bone" else rng.uniform(0, 80) if kind == "organ" else rng.uniform(30, 100)
            out.append((kind, rng.uniform(-lim, lim), ax, R, hu))
    return out


def _hu_at(structs, p):
    """HU at points p [M, 3] (mm, isocenter at the origin), float32."""
    dev = p.device
    t = lambda a: torch.as_tensor(np.asarray(a), dtype=torch.float32, device=dev)
    inside = ((p / t(BODY)) ** 2).sum(1) <= 1.0
    hu = torch.where(inside, 40.0, -1000.0)
    for kind, c, ax, R, val in structs:
        loc = (p - t(c)) @ t(R)
        m = (((loc / t(ax)) ** 2).sum(1) <= 1.0) & inside
        if kind == "bone":
            m &= ((loc / t(np.maximum(ax - 5.0, 1.0))) ** 2).sum(1) > 1.0
        hu = torch.where(m, hu + val if kind == "lesion" else torch.full_like(hu, val), hu)
    return hu


def _voxel_centres(idx, grid):
    v = FOV / grid
    xyz = torch.stack([idx % grid, (idx // grid) % grid, idx // (grid * grid)], 1)
    return (xyz.float() + 0.5) * v - FOV / 2


def _body_voxels(grid, dev):
    c = ((torch.arange(grid, device=dev) + 0.5) * (FOV / grid) - FOV / 2) ** 2
    r = (c / BODY[2] ** 2)[:, None, None] + (c / BODY[1] ** 2)[:, None] + c / BODY[0] ** 2
    return (r.reshape(-1) <= 1.0).nonzero().squeeze(1)


def _poses(rng, kind, n):
    """World-to-camera [n, 3, 4]: candidate poses about the isocenter (+-15 degrees, +-20 mm) or a
    circular orbit from the anterior-posterior view."""
    R_ap = np.array([[1.0, 0, 0], [0, 0, -1.0], [0, 1.0, 0]])
    out = np.zeros((n, 3, 4))
    start = rng.uniform(0, 2 * math.pi)
    for v in range(n):
        if kind == "orbit":
            R, d = _rot(2, start + 2 * math.pi * v / n), np.zeros(3)
        else:
            a = np.deg2rad(rng.uniform(-15, 15, 3))
            R, d = _rot(2, a[0]) @ _rot(1, a[1]) @ _rot(0, a[2]), rng.uniform(-20, 20, 3)
        out[v, :, :3] = R_ap @ R
        out[v, :, 3] = R_ap @ d + np.array([0.0, 0.0, SID])
    return out.astype(np.float32)


def _cloud(c, n, rng, gen, candidates=None, at=0):
    """Tensors of a cloud of n Gaussians: the last fifth is direction-dependent."""
    dev = gen.device
    U = lambda lo, hi, *s: lo + (hi - lo) * torch.rand(*s, generator=gen, device=dev)
    N = lambda *s: torch.randn(*s, generator=gen, device=dev)
    k, rows, n_iso = c["k"], c["degree"] * (c["degree"] + 2), n - n // 5
    if c["scene"] == "cube":
        means, log_s, alpha = U(-1, 1, n, 3), U(-4, -2, n, 3), U(0.1, 0.9, n)
    else:
        idx = candidates[(torch.arange(n, device=dev) + at) % candidates.numel()]
        means = _voxel_centres(idx, c["grid"])
        log_s = math.log(0.5 * FOV / c["grid"]) + U(-0.25, 0.25, n, 3)
        alpha = (0.05 + 0.9 * (_hu_at(_structures(rng), means) + 800) / 2300).clamp(0.05, 0.95)
    q = N(n, 4)
    dirs = 0.1 * N(n - n_iso, k)
    return dict(means=means.contiguous(), log_scales=log_s, quats=q / q.norm(dim=1, keepdim=True),
                opacity_logits=torch.logit(alpha), feat_iso=U(0, 1, n_iso, k),
                feat_dir=dirs.bfloat16() if c["bf16"] else dirs, b_iso=N(k) / math.sqrt(k),
                B_dir=N(rows, k) / math.sqrt(k))


def _detector(c, n, width, dev):
    sdd, pitch = (4.0, 8.0 / width) if c["scene"] == "cube" else (SDD, 256.0 / width)
    return torch.tensor([[sdd, pitch, pitch, 0.0, 0.0]] * n, device=dev)


def _inputs(c, seed):
    """Clouds, poses, detectors, sizes and target images of a rendering case, one entry per
    request (one request unless the case is a batch)."""
    dev = torch.device("cuda")
    rng = np.random.default_rng(seed)
    gen = torch.Generator(dev)
    gen.manual_seed(seed)
    cand = None
    if c["scene"] == "phantom":
        cand = _body_voxels(c["grid"], dev)
        cand = cand[torch.randperm(cand.numel(), generator=gen, device=dev)]
    reqs = []
    sizes = [2 ** i for i in range(20) if c["height"] <= 2 ** i <= c["width"]] + [c["height"], c["width"]]
    for r in range(c["gaussians"] if c["kind"] == "batch" else 1):
        if c["kind"] == "batch":
            # the sizes of a batch are the case's own; the seed changes what is in the clouds
            pick = np.random.default_rng(1000 + r)
            n = int(10 ** pick.uniform(4, 6))
            H = W = int(pick.choice(sizes))
        else:
            n, H, W = c["gaussians"], c["height"], c["width"]
        cloud = _cloud(c, n, rng, gen, cand, at=0 if cand is None else int(rng.integers(cand.numel())))
        if c["scene"] == "cube":
            pose = np.concatenate([np.eye(3), [[0.0], [0.0], [2.0]]], 1)[None].astype(np.float32)
        else:
            pose = _poses(rng, c["poses"], c["views"])
        x = (torch.arange(W, device=dev) + 0.5) / W * 2 - 1
        y = (torch.arange(H, device=dev) + 0.5) / H * 2 - 1
        # the target radiograph: the smooth shadow of a body
        tgt = 0.6 * (1 - x ** 2 / 0.3 - (y ** 2 / 0.5)[:, None]).clamp(min=0).sqrt()
        tgt = tgt * (1 + 0.2 * torch.sin(7 * x + (5 * y)[:, None]))
        reqs.append(dict(cloud=cloud, pose=torch.from_numpy(pose).to(dev), H=H, W=W, target=tgt.contiguous(),
                         det=_detector(c, len(pose), W, dev)))
    return reqs


def _volume(c, seed):
    """An int16 HU volume [nz, ny, nx] of 0.5 mm voxels at 512^3 (the phantom's central crop, with
    the pixel noise that scanners have) and its geometry."""
    dev = torch.device("cuda")
    structs = _structures(np.random.default_rng(seed))
    gen = torch.Generator(dev)
    gen.manual_seed(seed)
    v = 0.5
    org = tuple(-0.5 * v * (m - 1) for m in (c["nx"], c["ny"], c["nz"]))
    ax = [torch.arange(m, device=dev) * v + o for m, o in zip((c["nx"], c["ny"], c["nz"]), org)]
    hu = torch.empty((c["nz"], c["ny"], c["nx"]), dtype=torch.int16, device=dev)
    for z in range(0, c["nz"], 16):
        g = torch.meshgrid(ax[2][z:z + 16], ax[1], ax[0], indexing="ij")
        h = _hu_at(structs, torch.stack([g[2].reshape(-1), g[1].reshape(-1), g[0].reshape(-1)], 1))
        h += 12 * torch.randn(h.shape, generator=gen, device=dev)
        hu[z:z + 16] = h.round().clamp(-1024, 3071).to(torch.int16).view(-1, c["ny"], c["nx"])
    return hu, (v, v, v), org


def prepare(case, seed):
    from paper_2406_02518_gb300 import binding as B

    c = case
    if c["kind"] == "rads":
        hu, spacing, org = _volume(c, seed)
        return dict(kind="rads", hu=hu, spacing=spacing, origin=org, n1=c["n1"], n2=c["n2"],
                    seed=seed, ws=B.Workspace())
    reqs = _inputs(c, seed)
    cfg = B.Config(near_plane=0.2 if c["scene"] == "cube" else 0.1 * SID, tile=c["tile"],
                   dilation=c["dilation"], batch_depth=c["depth"])
    ws = B.Workspace()
    clouds = [B.Cloud(**{k: r["cloud"][k].contiguous() for k in CLOUD}, entangled=c["entangled"],
                      per_pixel=c["per_pixel"]) for r in reqs]
    views = [B.Views(r["pose"], r["det"], r["H"], r["W"]) for r in reqs]
    s = dict(kind=c["kind"], cfg=cfg, ws=ws, cloud=clouds[0], views=views[0],
             target=reqs[0]["target"])
    if c["kind"] == "batch":
        s["batch"] = B.Batch(clouds, views)
        s["target"] = torch.cat([r["target"].reshape(-1) for r in reqs])
        s["grad"] = torch.cat([torch.full((r["H"] * r["W"],), 1.0 / (r["H"] * r["W"]), device="cuda") for r in reqs])
    if c["kind"] == "autograd":
        for k in CLOUD:
            getattr(s["cloud"], k).requires_grad_(True)
    if c["no_sync"]:
        # a loop that never waits for the GPU sizes the workspace once, from a first render
        B.render_batched(s["batch"], cfg, ws) if c["kind"] == "batch" else B.render(s["cloud"], s["views"], cfg, ws)
        torch.cuda.synchronize()
        tiles = sum(r["pose"].shape[0] * -(-r["H"] // cfg.tile) * -(-r["W"] // cfg.tile) for r in reqs)
        ws.reserve(sum(r["pose"].shape[0] * r["cloud"]["means"].shape[0] for r in reqs),
                   int(ws.pairs() * 1.1) + 4096, tiles)
        cfg.no_sync = True
    return s


def run(s):
    from paper_2406_02518_gb300 import binding as B

    kind, ws = s["kind"], s["ws"]
    if kind == "rads":
        r = B.rads(s["hu"], s["spacing"], s["origin"], s["n1"], s["n2"], seed=s["seed"], ws=ws)
        return {k: r[k] for k in ("means", "log_scales", "n_mc", "n_dw", "n_crossings", "n_iso")}
    if kind == "batch":
        img, tf, nl = B.render_batched(s["batch"], s["cfg"], ws)
        g = B.render_batched_backward(s["batch"], s["cfg"], ws, s["grad"], tf, nl)
        return dict(g, image=img, t_final=tf, n_last=nl)
    if kind == "autograd":
        img, tf, nl = B.render_differentiable(s["cloud"], s["views"], s["cfg"], ws)
        (img - s["target"]).abs().mean().backward()
        out = dict(image=img.detach(), t_final=tf, n_last=nl)
        for k in CLOUD:
            p = getattr(s["cloud"], k)
            out[k], p.grad = p.grad, None
        return out
    img, tf, nl = B.render(s["cloud"], s["views"], s["cfg"], ws)
    out = dict(image=img, t_final=tf, n_last=nl)
    if kind == "render":
        return out
    out["loss"], dL = B.l1_loss(img, s["target"])
    out.update(B.render_backward(s["cloud"], s["views"], s["cfg"], ws, dL, tf, nl,
                                 want=("world_to_cam",) if kind == "pose" else GRADS))
    return out


def work(case):
    c = case
    if c["kind"] == "rads":
        n = c["n1"] + c["n2"]
        # one reading of the volume; a point's distances to the points of the cells around it
        return {"bytes": 2.0 * c["nx"] * c["ny"] * c["nz"] + 24.0 * n, "flops": 8.0 * 27 * n}
    bytes_, pairs = 0.0, 0.0
    sizes = [2 ** i for i in range(20) if c["height"] <= 2 ** i <= c["width"]] + [c["height"], c["width"]]
    for r in range(c["gaussians"] if c["kind"] == "batch" else 1):
        n, H, W = c["gaussians"], c["height"], c["width"]
        if c["kind"] == "batch":
            pick = np.random.default_rng(1000 + r)
            n = int(10 ** pick.uniform(4, 6))
            H = W = int(pick.choice(sizes))
        n_iso = n - n // 5
        cloud = n * 44.0 + 4.0 * c["k"] * n_iso + (2.0 if c["bf16"] else 4.0) * c["k"] * (n - n_iso)
        grads = 0.0 if c["kind"] in ("render", "pose") else n * (44.0 + 4.0 * c["k"])
        bytes_ += cloud + grads + c["views"] * (H * W * 12.0 + 116.0)
        if c["kind"] != "render":
            bytes_ += H * W * 4.0
        # pixels inside a Gaussian's cutoff ellipse, at the mean scale and magnification
        s_px = (math.exp(-3.0) * 2.0 / (8.0 / W) if c["scene"] == "cube"
                else 0.5 * FOV / c["grid"] * (SDD / SID) / (256.0 / W))
        pairs += c["views"] * n * math.pi * Q_MAX * (s_px ** 2 + c["dilation"])
    return {"bytes": bytes_, "flops": pairs * (16.0 if c["kind"] == "render" else 62.0)}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------

def _harmonics(d, degree):
    """Real spherical harmonics of degrees 1..degree at unit directions d [..., 3]."""
    x, y, z = d.unbind(-1)
    p = math.pi
    Y = [-math.sqrt(3 / (4 * p)) * y, math.sqrt(3 / (4 * p)) * z, -math.sqrt(3 / (4 * p)) * x]
    if degree >= 2:
        a = 0.5 * math.sqrt(15 / p)
        Y += [a * x * y, -a * y * z, 0.25 * math.sqrt(5 / p) * (3 * z * z - 1), -a * x * z,
              0.5 * a * (x * x - y * y)]
    if degree >= 3:
        a, b, e = 0.25 * math.sqrt(35 / (2 * p)), 0.5 * math.sqrt(105 / p), 0.25 * math.sqrt(21 / (2 * p))
        Y += [-a * y * (3 * x * x - y * y), b * x * y * z, -e * y * (5 * z * z - 1),
              0.25 * math.sqrt(7 / p) * (5 * z ** 3 - 3 * z), -e * x * (5 * z * z - 1),
              0.5 * b * z * (x * x - y * y), -a * x * (x * x - 3 * y * y)]
    return torch.stack(Y, -1)


def _exact_view(c, p, pose, det, H, W, depth32):
    """Image and final transmittance [H W] of one view; p: the cloud's tensors in 64 bits."""
    dev = pose.device
    R, t = pose[:, :3], pose[:, 3]
    near = 0.2 if c["scene"] == "cube" else 0.1 * SID
    s = p["log_scales"].exp()
    w, x, y, z = (p["quats"] / p["quats"].norm(dim=1, keepdim=True)).unbind(1)
    M = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                     2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                     2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3) * s[:, None]
    xc = p["means"] @ R.T + t
    zc = xc[:, 2]
    fu, fv = det[0] / det[1], det[0] / det[2]
    u = fu * xc[:, 0] / zc + 0.5 * W + det[3]
    v = fv * xc[:, 1] / zc + 0.5 * H + det[4]
    A0 = (fu / zc)[:, None] * (R[0] - (xc[:, 0] / zc)[:, None] * R[2])
    A1 = (fv / zc)[:, None] * (R[1] - (xc[:, 1] / zc)[:, None] * R[2])
    B0, B1 = (A0[:, None] @ M).squeeze(1), (A1[:, None] @ M).squeeze(1)
    a, b, d = (B0 * B0).sum(1) + c["dilation"], (B0 * B1).sum(1), (B1 * B1).sum(1) + c["dilation"]
    det2 = a * d - b * b
    alpha = torch.sigmoid(p["opacity_logits"])
    n_iso = p["feat_iso"].shape[0]
    logit = torch.cat([p["feat_iso"] @ p["b_iso"], p["feat_dir"] @ p["b_iso"] * (1.0 if c["entangled"] else 0.0)])
    has_dir = torch.ones(len(s), dtype=torch.bool, device=dev)
    if not c["entangled"]:
        has_dir[:n_iso] = False
    h = torch.cat([p["feat_iso"], p["feat_dir"]]) @ p["B_dir"].T * has_dir[:, None]
    if not c["per_pixel"]:
        e = p["means"] + t @ R
        logit = logit + (_harmonics(e / e.norm(dim=1, keepdim=True), c["degree"]) * h).sum(1)
    with torch.no_grad():
        ok = (zc > near) & (zc < det[0]) & (det2 > 0)
        order = torch.sort(depth32, stable=True).indices  # ties: ascending index
        order = order[ok[order]]
        ex, ey = (Q_MAX * a[order]).sqrt(), (Q_MAX * d[order]).sqrt()
        x0 = (u[order] - ex - 0.5).ceil().clamp(0, W).long()
        y0 = (v[order] - ey - 0.5).ceil().clamp(0, H).long()
        nx = ((u[order] + ex - 0.5).floor().clamp(-1, W - 1).long() - x0 + 1).clamp(min=0)
        ny = ((v[order] + ey - 0.5).floor().clamp(-1, H - 1).long() - y0 + 1).clamp(min=0)
        cnt = nx * ny
        j = torch.repeat_interleave(torch.arange(len(order), device=dev), cnt)
        o = torch.arange(len(j), device=dev) - (cnt.cumsum(0) - cnt)[j]
        px, py, g = x0[j] + o % nx[j], y0[j] + o // nx[j], order[j]
        pix = py * W + px
        del j, o, px, py

    def pair(g, pix):
        dx, dy = u[g] - (pix % W + 0.5), v[g] - (pix // W + 0.5)
        q = (d[g] * dx * dx - 2 * b[g] * dx * dy + a[g] * dy * dy) / det2[g]
        aG = alpha[g] * torch.exp(-0.5 * q)
        return q, torch.where(aG > ALPHA_MAX, torch.full_like(aG, ALPHA_MAX), aG)

    with torch.no_grad():
        q, sigma = pair(g, pix)
        keep = (q <= Q_MAX) & (sigma >= ALPHA_MIN)
        g, pix = g[keep], pix[keep]
        del q, sigma, keep
        pix, o = torch.sort(pix, stable=True)
        g = g[o]
        first = torch.ones_like(pix, dtype=torch.bool)
        first[1:] = pix[1:] != pix[:-1]
        seg = first.nonzero().squeeze(1)[first.long().cumsum(0) - 1]
        del o, first
    _, sigma = pair(g, pix)
    lt = torch.log1p(-sigma)
    cum = lt.cumsum(0)
    before = (cum - lt) - (cum - lt)[seg]
    with torch.no_grad():
        live = torch.exp(before + lt) >= T_MIN
    z = logit[g]
    if c["per_pixel"]:
        yy, xx = torch.meshgrid(torch.arange(H, device=dev), torch.arange(W, device=dev), indexing="ij")
        ray = torch.stack([(xx + 0.5 - 0.5 * W - det[3]) * det[1], (yy + 0.5 - 0.5 * H - det[4]) * det[2],
                           torch.zeros_like(xx) + det[0]], -1).view(-1, 3) @ R
        z = z + (_harmonics(ray / ray.norm(dim=1, keepdim=True), 1)[pix] * h[g]).sum(1)
    zero = torch.zeros(H * W, dtype=torch.float64, device=dev)
    img = zero.index_add(0, pix, torch.sigmoid(z) * sigma * before.exp() * live)
    tf = zero.index_add(0, pix, lt * live).exp()
    return img, tf


def _exact_render(c, seed):
    out = {k: [] for k in ("image", "t_final", "loss") + GRADS}
    want = () if c["kind"] == "render" else ("world_to_cam",) if c["kind"] == "pose" else GRADS
    for r in _inputs(c, seed):
        p = {k: v.double().requires_grad_(k in want) for k, v in r["cloud"].items()}
        pose = r["pose"].double().requires_grad_("world_to_cam" in want)
        g = {k: torch.zeros_like(p[k] if k in p else pose) for k in want}
        H, W, V = r["H"], r["W"], len(r["pose"])
        img, tf, loss = [], [], []
        for i in range(V):
            T, mu = r["pose"][i], r["cloud"]["means"]
            # the depth that orders a ray is the 32-bit one, one rounding an operation
            depth = T[2, 0] * mu[:, 0] + T[2, 1] * mu[:, 1]
            depth = depth + T[2, 2] * mu[:, 2]
            depth = depth + T[2, 3]
            with torch.set_grad_enabled(bool(want)):
                im, tr = _exact_view(c, p, pose[i], r["det"][i].double(), H, W, depth)
                tgt = r["target"].double().reshape(-1)
                obj = im.sum() / (H * W) if c["kind"] == "batch" else (im - tgt).abs().sum() / (H * W)
            if want:
                got = torch.autograd.grad(obj / (V if c["kind"] == "autograd" else 1),
                                          [p[k] if k in p else pose for k in want], allow_unused=True)
                for k, x in zip(want, got):
                    if x is not None:
                        g[k] += x
                del got
            img.append(im.detach())
            tf.append(tr.detach())
            loss.append(obj.detach())
            del im, tr, obj
        out["image"].append(torch.stack(img).view(V, H, W))
        out["t_final"].append(torch.stack(tf).view(V, H, W))
        out["loss"].append(torch.stack(loss))
        for k in want:
            out[k].append(g[k])
    if c["kind"] == "batch":
        res = {k: torch.cat([x.reshape(-1) for x in out[k]]) for k in ("image", "t_final")}
        res.update({k: torch.stack(out[k]) if k in ("b_iso", "B_dir") else torch.cat(out[k]) for k in GRADS})
    else:
        res = {k: v[0] for k, v in out.items() if v}
        if c["kind"] in ("render", "autograd"):
            res.pop("loss")
        if c["kind"] == "autograd":
            res.pop("world_to_cam")
            if c["bf16"]:
                res["feat_dir"] = None
    return dict(res, n_last=None)


def _splitmix(seed, i):
    """Output i + 1 of SplitMix64 seeded with `seed`, as the bits of an int64."""
    s64 = lambda x: x - (1 << 64) if x >= 1 << 63 else x
    shr = lambda z, k: (z >> k) & ((1 << (64 - k)) - 1)
    z = s64(seed % (1 << 64)) + (i + 1) * s64(0x9E3779B97F4A7C15)
    z = (z ^ shr(z, 30)) * s64(0xBF58476D1CE4E5B9)
    z = (z ^ shr(z, 27)) * s64(0x94D049BB133111EB)
    return z ^ shr(z, 31)


def _exact_rads(c, seed):
    hu, sp, org = _volume(c, seed)
    dev = hu.device
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    lo, hi = int(hu.min()), int(hu.max())
    above = 2 * hu.int() > lo + hi
    step = (1, nx, nx * ny)
    edges = []
    for axis in range(3):
        dim = 2 - axis
        m = torch.zeros_like(above)
        k = above.shape[dim] - 1
        m.narrow(dim, 0, k).copy_(above.narrow(dim, 0, k) != above.narrow(dim, 1, k))
        edges.append(m.reshape(-1).nonzero().squeeze(1) * 3 + axis)
    e = torch.sort(torch.cat(edges)).values
    M, n1, n2 = e.numel(), min(c["n1"], e.numel()), c["n2"] if hi > lo else 0
    if M > n1:
        high = (_splitmix(seed, e) >> 32) & 0xFFFFFFFF
        key = ((high - (1 << 31)) << 32) | e  # the unsigned order as a signed one
        e = e[torch.sort(torch.topk(key, n1, largest=False).indices).values]
    v, axis = e // 3, e % 3
    flat = hu.reshape(-1).double()
    d = torch.tensor(step, device=dev)[axis]
    f0, f1 = flat[v], flat[v + d]
    xyz = torch.stack([v % nx, (v // nx) % ny, v // (nx * ny)], 1).double()
    xyz[torch.arange(len(e), device=dev), axis] += (0.5 * (lo + hi) - f0) / (f1 - f0)
    weight = (hu.reshape(-1).long() - lo).cumsum(0)
    total = int(weight[-1])
    h = _splitmix((1 << 64) - 1 - seed, torch.arange(n2, device=dev)).tolist()
    at = torch.tensor([((x % (1 << 64)) * total) >> 64 for x in h], dtype=torch.int64, device=dev)
    v = torch.searchsorted(weight, at, right=True)
    del weight
    pts = torch.cat([xyz, torch.stack([v % nx, (v // nx) % ny, v // (nx * ny)], 1).double()])
    # the geometry as the call gets it, in 32 bits
    f32 = lambda a: torch.tensor([float(np.float32(q)) for q in a], dtype=torch.float64, device=dev)
    pts = pts * f32(sp) + f32(org)
    best = []
    for q in pts.split(2048):
        d2 = sum((q[:, None, i] - pts[None, :, i]) ** 2 for i in range(3))
        best.append(torch.topk(d2, 4, dim=1, largest=False).values[:, 1:].mean(1))
    ls = 0.5 * torch.log(torch.cat(best).clamp(min=1e-7))
    return dict(means=pts, log_scales=ls[:, None].expand(-1, 3).contiguous(), n_mc=None, n_dw=None,
                n_crossings=None, n_iso=None)


def exact(case, seed):
    return _exact_rads(case, seed) if case["kind"] == "rads" else _exact_render(case, seed)
