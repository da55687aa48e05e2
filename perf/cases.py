"""What the framework's speed is measured on: its layers, blocks and whole calls over their real range.

A case names an entry point (``kind``) and its sizes; inputs are made on the GPU from a seed alone.
Scenes are the two synthetic ones the tests and the benchmark use: Gaussians in a cube in front of one
camera, and an outdoor-like ring (a noisy ground plane and five boxes) seen by cameras on the ring.

  forward    Raster.forward: a stateless render with its per-pixel outputs
  render     Field.render: a resident field seen from a new camera (a viewer, an evaluation)
  loss       Raster.loss: L1 + D-SSIM of rendered views against their targets, with its gradient
  backward   Raster.backward: gradients of the last forward for a given dL/dimage
  grad       forward, loss and backward of one training step on caller-owned tensors
  adam       adam_step on caller-owned tensors
  integrate  an arriving image: its pixels from pinned memory, the Local & Semi-Global iterations over it
             and its neighbours (graph-replayed steps with the fused Adam), and the field read back
"""
import math

import numpy as np
import torch

import paper_2503_13086_gb300 as gs

NP = 59
LAMBDA_SSIM = 0.2
LRS = [1.6e-4, 5e-3, 1e-3, 0.05, 2.5e-3, 1.25e-4]
RING_FOCAL = 1000.0
SIZE_CYCLE = (1.0, 0.74, 0.99, 1.23)  # mixed resolutions of the views of one step


def listed():
    return [
        # the smallest calls: launches, copies and waits count
        {"name": "forward_tiny", "kind": "forward", "scene": "cube", "n": 512, "width": 64, "height": 48, "views": 1},
        # the plain single-view workload: 4,096 Gaussians in a cube, 256 x 256
        {"name": "grad_256", "kind": "grad", "scene": "cube", "n": 4096, "width": 256, "height": 256, "views": 1},
        # scene scale, an odd image width: 200k Gaussians on a ring, 1297 x 840
        {"name": "forward_scene", "kind": "forward", "scene": "ring", "n": 200_000, "width": 1297, "height": 840, "views": 1},
        {"name": "loss_scene", "kind": "loss", "scene": "ring", "n": 2_000, "width": 1297, "height": 840, "views": 1},
        {"name": "backward_scene", "kind": "backward", "scene": "ring", "n": 200_000, "width": 1297, "height": 840, "views": 1},
        # the batched local and semi-global step: 9 views at mixed resolutions
        {"name": "grad_batch", "kind": "grad", "scene": "ring", "n": 500_000, "width": 1297, "height": 840, "views": 9},
        # a field late in a stream, one view per step, a count that is no multiple of anything
        {"name": "grad_large", "kind": "grad", "scene": "ring", "n": 1_900_001, "width": 1297, "height": 840, "views": 1},
        # a 3M-Gaussian field of the serving workload rendered at full HD
        {"name": "render_hd", "kind": "render", "scene": "ring", "n": 3_000_000, "width": 1920, "height": 1080, "views": 1},
        # the optimizer alone on a large field
        {"name": "adam_large", "kind": "adam", "scene": "ring", "n": 1_500_013, "width": 0, "height": 0, "views": 1},
        # arrivals: a young field of small images, scene scale, and a grown field with 3 views per step
        {"name": "integrate_small", "kind": "integrate", "scene": "ring", "n": 20_000, "width": 640, "height": 361, "views": 1,
         "iters": 200, "adam_state": True},
        {"name": "integrate_scene", "kind": "integrate", "scene": "ring", "n": 200_000, "width": 1297, "height": 840, "views": 1,
         "iters": 200, "adam_state": False},
        {"name": "integrate_large", "kind": "integrate", "scene": "ring", "n": 1_500_000, "width": 1297, "height": 840, "views": 3,
         "iters": 201, "adam_state": False},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forward", "grad", "grad", "backward", "render", "loss", "adam", "integrate"])
    width = _log_int(rng, 48, 1920)
    height = max(33, int(width * rng.uniform(0.5, 0.9)))
    c = {"kind": kind, "scene": "ring", "n": _log_int(rng, 1_000, 2_000_000), "width": width, "height": height, "views": 1}
    if kind in ("forward", "grad", "backward"):
        c["scene"] = rng.choice(["ring", "ring", "cube"]) if c["n"] <= 50_000 else "ring"
        c["views"] = rng.choice([1, 1, 2, 4, 7])
        c["n"] = min(c["n"], 3_000_000 // c["views"])
        if width > 1400:
            c["views"] = min(c["views"], 4)
    elif kind == "loss":
        c["n"] = 1_000
        c["views"] = rng.choice([1, 2, 5])
    elif kind == "adam":
        c["width"] = c["height"] = 0
    elif kind == "integrate":
        c["n"] = _log_int(rng, 2_000, 500_000)
        c["views"] = rng.choice([1, 1, 2, 3])
        c["iters"] = rng.randrange(40, 160)
        c["adam_state"] = c["n"] < 30_000
    return c


# ---------------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------------
def _gen(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * int(seed) + salt)
    return g


def _gaussians(case, seed):
    """(59, stride) parameters on the GPU, component-major."""
    n = case["n"]
    stride = (n + 31) // 32 * 32
    g = _gen(seed)

    def uni(lo, hi, *shape):
        return lo + (hi - lo) * torch.rand(*shape, generator=g, device="cuda")

    def normal(mu, sigma, *shape):
        return mu + sigma * torch.randn(*shape, generator=g, device="cuda")

    p = torch.zeros(NP, stride, device="cuda")
    if case["scene"] == "cube":
        p[0:2, :n] = uni(-1, 1, 2, n)
        p[2, :n] = uni(2, 4, n)
        p[3:6, :n] = normal(-4.0, 0.5, 3, n)
    else:
        n_ground = int(round(0.6 * n))
        r = torch.sqrt(uni(16.0, 100.0, n_ground))
        th = uni(0, 2 * math.pi, n_ground)
        p[0, :n_ground] = r * torch.cos(th)
        p[1, :n_ground] = normal(0.0, 0.05, n_ground)
        p[2, :n_ground] = r * torch.sin(th)
        m = n - n_ground
        cr, ct, size = uni(5.0, 9.0, 5), uni(0, 2 * math.pi, 5), uni(0.6, 1.6, 5, 3)
        which = torch.randint(0, 5, (m,), generator=g, device="cuda")
        local = uni(-0.5, 0.5, m, 3) * size[which]
        p[0, n_ground:n] = cr[which] * torch.cos(ct[which]) + local[:, 0]
        p[1, n_ground:n] = -(local[:, 1] + 0.5 * size[which, 1])
        p[2, n_ground:n] = cr[which] * torch.sin(ct[which]) + local[:, 2]
        p[3:6, :n] = normal(-4.5, 0.7, 3, n)
    q = normal(0, 1, 4, n)
    p[6:10, :n] = q / q.norm(dim=0, keepdim=True)
    p[10, :n] = normal(0, 1, n)
    p[11:59, :n] = normal(0, 0.2, 48, n)
    return p


def _view_sizes(case):
    if case["views"] == 1 or case["kind"] == "integrate":
        return [(case["width"], case["height"])] * case["views"]
    return [(max(33, round(case["width"] * f)), max(33, round(case["height"] * f)))
            for f in (SIZE_CYCLE[k % len(SIZE_CYCLE)] for k in range(case["views"]))]


def _ring_camera(theta, w, h, rng):
    eye = np.array([7.0 * np.cos(theta), -1.5, 7.0 * np.sin(theta)]) + rng.normal(0, 0.03, 3)
    fwd = np.array([0.0, -0.3, 0.0]) + rng.normal(0, 0.03, 3) - eye
    fwd /= np.linalg.norm(fwd)
    x = np.cross(fwd, [0.0, -1.0, 0.0])
    x /= np.linalg.norm(x)
    R = np.stack([x, np.cross(fwd, x), fwd])
    f = RING_FOCAL * w / 1297.0
    return dict(R=R, t=-R @ eye, fx=f, fy=f, cx=w / 2.0, cy=h / 2.0, width=w, height=h)


def _cameras(case, seed, sizes):
    rng = np.random.default_rng([int(seed), 7])
    base = rng.uniform(0, 2 * np.pi)
    if case["scene"] == "cube":
        cams = []
        for k, (w, h) in enumerate(sizes):
            a = 0.05 * k
            R = np.array([[math.cos(a), 0, -math.sin(a)], [0, 1, 0], [math.sin(a), 0, math.cos(a)]])
            c = np.array([0.0, 0.0, 3.0])
            cams.append(dict(R=R, t=c - R @ c, fx=float(w), fy=float(w), cx=w / 2.0, cy=h / 2.0, width=w, height=h))
        return cams
    return [_ring_camera(base + 0.12 * (k - len(sizes) // 2), w, h, rng) for k, (w, h) in enumerate(sizes)]


def _photo(w, h, g):
    """A (3, h, w) picture in [0, 1]: smooth shading, edges and sensor noise."""
    y = torch.arange(h, device="cuda", dtype=torch.float32)[:, None] / h
    x = torch.arange(w, device="cuda", dtype=torch.float32)[None, :] / w
    k = torch.rand(3, 4, generator=g, device="cuda") * 12
    img = torch.stack([0.5 + 0.2 * torch.sin(k[c, 0] * x + k[c, 1]) * torch.cos(k[c, 2] * y + k[c, 3])
                       + 0.15 * torch.sign(torch.sin(3 * k[c, 1] * x + 2 * k[c, 3] * y)) for c in range(3)])
    return (img + 0.05 * torch.randn(3, h, w, generator=g, device="cuda")).clamp_(0, 1)


def _photos(sizes, seed):
    g = _gen(seed, 1)
    return torch.cat([_photo(w, h, g).reshape(-1) for w, h in sizes])


def _prepare_integrate(case, seed):
    n_img = 10
    w, h = case["width"], case["height"]
    # learning rates of a late refinement (a thousandth of the defaults): every step does the work of any
    # other, and the field a pass leaves is close to the one it found, so passes can be compared
    field = gs.Field(scene_extent=7.0, lambda_ssim=LAMBDA_SSIM, use_graph=1, async_steps=16, tiling=(16, 16, 256),
                     T_I=case["iters"], batch_views=case["views"], seed=int(seed) & 0x7FFFFFFF, add_dist_thresh=100.0,
                     eta0=1.6e-7, etaf=1.6e-9, lr_scale=5e-6, lr_rot=1e-6, lr_opacity=5e-5, lr_sh_dc=2.5e-6,
                     lr_sh_rest=1.25e-7, initial_capacity=case["n"] + 4096)
    p = _gaussians(case, seed)
    field.set_gaussians(p[:, :case["n"]].cpu().numpy())
    cams = _cameras(dict(case), seed, [(w, h)] * n_img)
    rng = np.random.default_rng([int(seed), 8])
    n_pts = 400
    idx = rng.integers(0, case["n"], n_pts * (n_img + 2) // 2)
    xyz = p[0:3, torch.from_numpy(idx).cuda()].T.contiguous().cpu().numpy()
    g = _gen(seed, 2)
    for k, c in enumerate(cams):
        at = slice(k * n_pts // 2, k * n_pts // 2 + n_pts)  # half of an image's tracks are its neighbour's too
        pts = xyz[at]
        last = field.add_image(c, _photo(w, h, g), pts, rng.uniform(0, 1, (len(pts), 3)).astype(np.float32),
                               np.arange(at.start, at.start + len(pts), dtype=np.int32))
    pinned = _photo(w, h, g).permute(1, 2, 0).contiguous().cpu().pin_memory()  # the arriving image as decoded
    torch.cuda.synchronize()
    return dict(case=case, field=field, id=last, pixels=pinned)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "integrate":
        return _prepare_integrate(case, seed)
    if kind == "adam":
        p = _gaussians(case, seed)
        g = _gen(seed, 3)
        grads = 1e-6 * torch.randn(p.shape, generator=g, device="cuda")
        m = 1e-6 * torch.randn(p.shape, generator=g, device="cuda")
        v = 1e-12 * torch.rand(p.shape, generator=g, device="cuda")
        return dict(case=case, p=p, grads=grads, m=m, v=v, step=50)
    sizes = _view_sizes(case)
    p = _gaussians(case, seed)
    cams = _cameras(case, seed, sizes)
    if kind == "render":
        field = gs.Field(scene_extent=7.0, tiling=(16, 16, 256))
        field.set_gaussians(p[:, :case["n"]].cpu().numpy())
        return dict(case=case, field=field, cam=cams[0])
    s = dict(case=case, p=p, cams=cams, raster=gs.Raster())
    if kind in ("grad", "loss"):
        s["target"] = _photos(sizes, seed)
    if kind == "loss":
        s["raster"].forward(p, case["n"], cams)  # the loss reads the views of the last forward
        s["image"] = (s["target"] + 0.1 * torch.randn(s["target"].shape, generator=_gen(seed, 4), device="cuda")).clamp_(0, 1)
    if kind == "backward":
        s["out"] = s["raster"].forward(p, case["n"], cams)
        npix = sum(w * h for w, h in sizes)
        s["dimage"] = torch.randn(3 * npix, generator=_gen(seed, 5), device="cuda") / (3 * npix)
    return s


def run(s):
    case = s["case"]
    kind, n = case["kind"], case["n"]
    if kind == "forward":
        o = s["raster"].forward(s["p"], n, s["cams"])
        return {k: o[k] for k in ("image", "T", "last", "gp", "pairs")}
    if kind == "render":
        image, T = s["field"].render(s["cam"], want_T=True)
        return {"image": image, "T": T}
    if kind == "loss":
        value, dimage = s["raster"].loss(s["image"], s["target"], LAMBDA_SSIM)
        return {"loss": value, "dimage": dimage}
    if kind == "backward":
        return {"grads": s["raster"].backward(s["p"], s["out"]["image"], s["out"]["last"], s["dimage"])[0]}
    if kind == "grad":
        o = s["raster"].forward(s["p"], n, s["cams"])
        value, dimage = s["raster"].loss(o["image"], s["target"], LAMBDA_SSIM)
        grads, _ = s["raster"].backward(s["p"], o["image"], o["last"], dimage)
        return {"image": o["image"], "last": o["last"], "pairs": o["pairs"], "loss": value, "grads": grads}
    if kind == "adam":
        s["step"] += 1
        gs.adam_step(s["p"], s["grads"], s["m"], s["v"], n, LRS, s["step"])
        return {"params": s["p"], "m": s["m"], "v": s["v"]}
    field = s["field"]
    field.set_image(s["id"], s["pixels"])
    stats = field.integrate(s["id"])
    if case["adam_state"]:
        params, m, v = field.get_gaussians(with_adam=True)
        return {"loss": stats["mean_loss"], "params": params, "m": m, "v": v}
    return {"loss": stats["mean_loss"], "params": field.get_gaussians()}


def work(case):
    """Bytes: inputs once, outputs once (and, per optimisation step, the parameters and moments read and
    written).  Flops: projection and colour per Gaussian and view, blending of about 6 Gaussians per pixel,
    the separable 11-tap windows of the loss, the chain rule and the update."""
    kind, n = case["kind"], case["n"]
    pix = sum(w * h for w, h in _view_sizes(case))
    row = 4 * NP * n
    views = len(_view_sizes(case))
    fwd = {"bytes": row + 24 * pix, "flops": 350 * n * views + 6 * 25 * pix}
    loss = {"bytes": 36 * pix, "flops": 3 * (2 * 154 + 60) * pix}
    bwd = {"bytes": 2 * row + 28 * pix, "flops": 900 * n * views + 6 * 60 * pix}
    if kind in ("forward", "render"):
        return fwd
    if kind == "loss":
        return loss
    if kind == "backward":
        return bwd
    if kind == "grad":
        return {k: fwd[k] + loss[k] + bwd[k] for k in fwd}
    if kind == "adam":
        return {"bytes": 7 * row, "flops": 14 * NP * n}
    steps = -(-case["iters"] // case["views"])
    return {"bytes": steps * (6 * row + 24 * pix) + row + 24 * case["width"] * case["height"],
            "flops": steps * (fwd["flops"] + loss["flops"] + bwd["flops"] + 14 * NP * n)}


# ---------------------------------------------------------------------------------------------
# The same results in 64 bits, as plain torch gives them
# ---------------------------------------------------------------------------------------------
def _sh(d):
    x, y, z = d[0], d[1], d[2]
    xx, yy, zz = x * x, y * y, z * z
    pi = math.pi
    a1, b1, c1 = math.sqrt(3 / (4 * pi)), math.sqrt(15 / pi) / 2, math.sqrt(5 / pi) / 4
    e1, f1, g1 = math.sqrt(35 / (2 * pi)) / 4, math.sqrt(105 / pi) / 2, math.sqrt(21 / (2 * pi)) / 4
    h1, i1 = math.sqrt(7 / pi) / 4, math.sqrt(105 / pi) / 4
    one = torch.ones_like(x)
    return torch.stack([
        0.5 / math.sqrt(pi) * one, -a1 * y, a1 * z, -a1 * x, b1 * x * y, -b1 * y * z, c1 * (2 * zz - xx - yy), -b1 * x * z,
        b1 / 2 * (xx - yy), -e1 * y * (3 * xx - yy), f1 * x * y * z, -g1 * y * (4 * zz - xx - yy),
        h1 * z * (2 * zz - 3 * xx - 3 * yy), -g1 * x * (4 * zz - xx - yy), i1 * z * (xx - yy), -e1 * x * (xx - 3 * yy)])


def _project(p, cam):
    """2D records of the Gaussians of (59, n) float64 parameters, near to far, and which are visible."""
    R = torch.tensor(np.asarray(cam["R"], np.float32), device="cuda").double()
    t = torch.tensor(np.asarray(cam["t"], np.float32), device="cuda").double()
    fx, fy, cx, cy = (float(np.float32(cam[k])) for k in ("fx", "fy", "cx", "cy"))
    w, h = cam["width"], cam["height"]
    pc = R @ p[0:3] + t[:, None]
    z = pc[2]
    near = z > 0.2
    zs = torch.where(near, z, torch.ones_like(z))
    q = p[6:10] / p[6:10].norm(dim=0, keepdim=True)
    qw, qx, qy, qz = q[0], q[1], q[2], q[3]
    Rq = torch.stack([1 - 2 * (qy * qy + qz * qz), 2 * (qx * qy - qw * qz), 2 * (qx * qz + qw * qy),
                      2 * (qx * qy + qw * qz), 1 - 2 * (qx * qx + qz * qz), 2 * (qy * qz - qw * qx),
                      2 * (qx * qz - qw * qy), 2 * (qy * qz + qw * qx), 1 - 2 * (qx * qx + qy * qy)]).reshape(3, 3, -1)
    M = Rq * torch.exp(p[3:6])[None]
    Sig = torch.einsum("acn,bcn->abn", M, M)
    limx, limy = 1.3 * w / (2 * fx), 1.3 * h / (2 * fy)
    txz, tyz = (pc[0] / zs).clamp(-limx, limx), (pc[1] / zs).clamp(-limy, limy)
    zero = torch.zeros_like(zs)
    J = torch.stack([fx / zs, zero, -fx * txz / zs, zero, fy / zs, -fy * tyz / zs]).reshape(2, 3, -1)
    T = torch.einsum("abn,bc->acn", J, R)
    cov = torch.einsum("abn,bcn,dcn->adn", T, Sig, T)
    a, b, c = cov[0, 0] + 0.3, cov[0, 1], cov[1, 1] + 0.3
    det = a * c - b * b
    u, v = fx * pc[0] / zs + cx, fy * pc[1] / zs + cy
    with torch.no_grad():
        mid = 0.5 * (a + c)
        r = torch.ceil(3 * torch.sqrt(mid + torch.sqrt((mid * mid - det).clamp_min(0.1))))
        gx, gy = -(-w // 16), -(-h // 16)
        x0, x1 = ((u - r) / 16).floor().clamp(0, gx), ((u + r + 15) / 16).floor().clamp(0, gx)
        y0, y1 = ((v - r) / 16).floor().clamp(0, gy), ((v + r + 15) / 16).floor().clamp(0, gy)
        keep = (near & (det > 0) & (x1 > x0) & (y1 > y0)).nonzero()[:, 0]
        keep = keep[torch.argsort(z[keep].float(), stable=True)]
    campos = -(R.T @ t)
    d = p[0:3] - campos[:, None]
    col = torch.einsum("kn,kcn->cn", _sh(d / d.norm(dim=0, keepdim=True)), p[11:59].reshape(16, 3, -1)) + 0.5
    rec = torch.stack([u, v, c / det, -b / det, a / det, torch.sigmoid(p[10]), *col.clamp_min(0)])[:, keep]
    return rec, torch.stack([x0, x1, y0, y1])[:, keep]


def _blend(rec, rect, w, rows):
    """(3, rows, w) colours, (rows, w) transmittance of image rows `rows` (a tensor), black background."""
    px = torch.arange(w, device="cuda", dtype=torch.float64)
    x, y = px.repeat(len(rows)), rows.double().repeat_interleave(w)
    tx, ty = (x / 16).floor()[None], (y / 16).floor()[None]
    inside = (tx >= rect[0, :, None]) & (tx < rect[1, :, None]) & (ty >= rect[2, :, None]) & (ty < rect[3, :, None])
    dx, dy = rec[0][:, None] - x, rec[1][:, None] - y
    power = -0.5 * (rec[2][:, None] * dx * dx + rec[4][:, None] * dy * dy) - rec[3][:, None] * dx * dy
    alpha = (rec[5][:, None] * torch.exp(power)).clamp_max(0.99)
    alpha = torch.where(inside & (power <= 0) & (alpha >= 1 / 255), alpha, torch.zeros_like(alpha))
    after = torch.cumprod(1 - alpha, dim=0)
    with torch.no_grad():
        on = after >= 1e-4
    alpha = torch.where(on, alpha, torch.zeros_like(alpha))
    after = torch.cumprod(1 - alpha, dim=0)
    before = torch.cat([torch.ones_like(after[:1]), after[:-1]])
    wgt = alpha * before
    T = after[-1] if len(after) else torch.ones_like(x)
    return (rec[6:9] @ wgt).reshape(3, len(rows), w), T.reshape(len(rows), w)


def _chunks(h, w, n):
    step = max(1, min(h, 20_000_000 // max(1, w * n)))
    return [torch.arange(r, min(h, r + step), device="cuda") for r in range(0, h, step)]


def _exact_images(p, cams):
    with torch.no_grad():
        views = []
        for cam in cams:
            rec, rect = _project(p, cam)
            parts = [_blend(rec, rect, cam["width"], rows) for rows in _chunks(cam["height"], cam["width"], rec.shape[1])]
            views.append((torch.cat([c for c, _ in parts], 1), torch.cat([t for _, t in parts], 0)))
    return views


def _exact_loss(images, targets):
    """Loss and its gradient; images and targets: lists of (3, h, w) float64."""
    k = torch.exp(-(torch.arange(11, device="cuda", dtype=torch.float64) - 5) ** 2 / (2 * 1.5 ** 2))
    k = k / k.sum()

    def blur(m):
        m = torch.nn.functional.pad(m, (5, 5, 5, 5))
        m = sum(k[i] * m[:, :, i:m.shape[2] - 10 + i] for i in range(11))
        return sum(k[i] * m[:, i:m.shape[1] - 10 + i] for i in range(11))

    total, grads = 0.0, []
    for img, tgt in zip(images, targets):
        x = img.detach().requires_grad_(True)
        mx, my = blur(x), blur(tgt)
        sx, sy, sxy = blur(x * x) - mx * mx, blur(tgt * tgt) - my * my, blur(x * tgt) - mx * my
        ssim = ((2 * mx * my + 1e-4) * (2 * sxy + 9e-4)) / ((mx * mx + my * my + 1e-4) * (sx + sy + 9e-4))
        value = ((1 - LAMBDA_SSIM) * (x - tgt).abs().mean() + LAMBDA_SSIM * (1 - ssim.mean())) / len(images)
        value.backward()
        total += float(value.detach())
        grads.append(x.grad)
    return total, grads


def _exact_grads(p, cams, dimages):
    p = p.detach().requires_grad_(True)
    for cam, dimg in zip(cams, dimages):
        rec, rect = _project(p, cam)
        leaf = rec.detach().requires_grad_(True)
        for rows in _chunks(cam["height"], cam["width"], 4 * rec.shape[1]):
            img, _ = _blend(leaf, rect, cam["width"], rows)
            img.backward(dimg[:, rows])
        if leaf.grad is not None:
            rec.backward(leaf.grad)
    return p.grad


def _split(flat, sizes):
    out, at = [], 0
    for w, h in sizes:
        out.append(flat[at:at + 3 * w * h].reshape(3, h, w).double())
        at += 3 * w * h
    return out


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    if kind in ("render", "integrate"):
        return None
    sizes = _view_sizes(case)
    if kind == "adam":
        s = prepare(case, seed)
        t, b1, b2 = s["step"] + 1, 0.9, 0.999
        b1, b2 = float(np.float32(b1)), float(np.float32(b2))
        g = s["grads"].double()
        m, v, p = s["m"].double(), s["v"].double(), s["p"].double()
        m[:, :n] = b1 * m[:, :n] + (1 - b1) * g[:, :n]
        v[:, :n] = b2 * v[:, :n] + (1 - b2) * g[:, :n] ** 2
        lr = torch.tensor(np.repeat(np.float32(LRS), [3, 3, 4, 1, 3, 45]), device="cuda").double()[:, None]
        p[:, :n] -= lr * (m[:, :n] / (1 - b1 ** t)) / (torch.sqrt(v[:, :n] / (1 - b2 ** t)) + float(np.float32(1e-15)))
        return {"params": p, "m": m, "v": v}
    if kind == "loss":
        target = _photos(sizes, seed)
        image = (target + 0.1 * torch.randn(target.shape, generator=_gen(seed, 4), device="cuda")).clamp_(0, 1)
        value, d = _exact_loss(_split(image, sizes), _split(target, sizes))
        return {"loss": value, "dimage": torch.cat([x.reshape(-1) for x in d])}
    pix = sum(w * h for w, h in sizes)
    if n * pix > 300_000_000:
        return None
    given = _gaussians(case, seed)
    cams = _cameras(case, seed, sizes)
    p = given[:, :n].double()
    views = _exact_images(p, cams)
    image = torch.cat([c.reshape(-1) for c, _ in views])
    if kind == "forward":
        return {"image": image, "T": torch.cat([t.reshape(-1) for _, t in views]), "last": None, "gp": None, "pairs": None}
    if kind == "backward":
        d = torch.randn(3 * pix, generator=_gen(seed, 5), device="cuda") / (3 * pix)
        value, dimages = None, _split(d, sizes)
    else:
        value, dimages = _exact_loss([c for c, _ in views], _split(_photos(sizes, seed), sizes))
    grads = torch.zeros(given.shape, device="cuda", dtype=torch.float64)
    grads[:, :n] = _exact_grads(p, cams, dimages)
    if kind == "backward":
        return {"grads": grads}
    return {"image": image, "last": None, "pairs": None, "loss": value, "grads": grads}
