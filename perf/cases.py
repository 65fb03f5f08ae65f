"""What the library is used for, as cases that can be timed: mapping iterations over one keyframe
and over a window, with each loss and mode, the differentiable render, novel views, map growth
(insertion, splitting) and the learned initialiser (training, prediction).

Scenes are Gaussians on the surfaces of a furnished room, seen by a camera path inside it, with the
image sizes, Gaussian counts and options of this repository's benchmark, tests and stream (1200x680
with 300k Gaussians, eight views of 640x480 with 150k, 160x120 with 2k, 96 points a keyframe, 4,096
rows a training step), and odd sizes between. Learning rates are those of a keyframe's last
iterations (a thousandth of the initial ones), so that a map that is iterated on for long stays the
map that was prepared.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2504_02437_gb300.api import MLP, GaussianMap, rasterize

DEV = "cuda"
LR = (1e-6, 5e-6, 1e-6, 5e-5, 2.5e-6)
HALF = (3.0, 1.5, 3.0)          # the room's half extents, y down
SIGMA = 32.0                    # dominated pixels above which a Gaussian is split
N_IN, N_HID, N_OUT, N_OUT_PAD = 80, 128, 11, 16


def listed():
    def it(name, n, views, width, height, ssim=0.0, det=0, tile=16):
        return dict(name=name, kind="iterate", n=n, views=views, width=width, height=height, ssim=ssim, det=det,
                    tile=tile)
    return [
        # the first keyframes of a stream: a small map and image, where launches and latency count
        it("iterate_160x120_2k", 2_000, 1, 160, 120),
        # one dense keyframe, the benchmark's headline (layout left to the autotuner, as there)
        it("iterate_1200x680_300k", 300_000, 1, 1200, 680, tile=0),
        # a window of eight keyframes as a mapping stream optimises it, the largest call
        it("iterate_8x640x480_150k", 150_000, 8, 640, 480, tile=0),
        # the paper's L1 + SSIM loss, at an odd image size
        it("iterate_ssim_2x641x479_60k", 60_000, 2, 641, 479, ssim=0.2),
        # the bitwise repeatable mode, a three-view window of a young map
        it("iterate_det_3x321x243_20k", 20_000, 3, 321, 243, det=1),
        # a caller's own loss through autograd: render and adjoint by themselves
        dict(name="rasterize_2x333x251_30k", kind="rasterize", n=30_000, views=2, width=333, height=251),
        # a view of the finished map with its transmittance and dominant Gaussians, for evaluation
        dict(name="view_1200x680_300k", kind="view", n=300_000, views=1, width=1200, height=680),
        # a keyframe's points offered to a grown map
        dict(name="insert_96_150k", kind="insert", n=150_000, points=96, width=640, height=480, learned=False),
        # the same with the learned initialiser, early in a stream
        dict(name="insert_learned_96_5k", kind="insert", n=5_000, points=96, width=640, height=480, learned=True),
        # the clarity split after a keyframe
        dict(name="densify_640x480_150k", kind="densify", n=150_000, views=1, width=640, height=480),
        # one training step of the learned initialiser
        dict(name="mlp_train_4096", kind="mlp_train", rows=4096),
        # features and predictions for one keyframe's points, the smallest call
        dict(name="mlp_predict_96", kind="mlp_predict", rows=96, width=640, height=480),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def image(pixels):
        h = max(48, int(math.sqrt(pixels / rng.uniform(1.2, 1.9))))
        return dict(width=max(64, pixels // h), height=h)

    kind = rng.choice(["iterate", "iterate", "iterate", "ssim", "det", "rasterize", "view", "insert", "densify",
                       "mlp_train", "mlp_predict"])
    if kind in ("iterate", "ssim", "det"):
        views = rng.choice([1, 1, 2, 3, 5, 8])
        size = image(log(19_000, 800_000 // max(1, views // 2)))
        n = log(2_000, 250_000 if views < 3 else 130_000)
        return dict(kind="iterate", n=n, views=views, **size, ssim=0.2 if kind == "ssim" else 0.0,
                    det=1 if kind == "det" else 0, tile=rng.choice([0, 16]) if kind == "iterate" else 16)
    if kind == "rasterize":
        return dict(kind=kind, n=log(2_000, 200_000), views=rng.choice([1, 2, 3]), **image(log(19_000, 300_000)))
    if kind == "view":
        return dict(kind=kind, n=log(2_000, 300_000), views=1, **image(log(19_000, 800_000)))
    if kind == "insert":
        return dict(kind=kind, n=log(200, 200_000), points=log(16, 400), **image(log(19_000, 400_000)),
                    learned=rng.random() < 0.4)
    if kind == "densify":
        return dict(kind=kind, n=log(2_000, 200_000), views=rng.choice([1, 1, 2]), **image(log(19_000, 300_000)))
    if kind == "mlp_train":
        return dict(kind=kind, rows=log(64, 16_384))
    return dict(kind="mlp_predict", rows=log(16, 8_192), **image(log(19_000, 400_000)))


# --------------------------------------------------------------------------- inputs


class Camera:
    """Pinhole camera with a world-to-camera pose (what the library's calls take)."""

    def __init__(self, width, height, f, center, target):
        self.width, self.height = width, height
        self.fx = self.fy = float(np.float32(f))
        self.cx, self.cy = float(np.float32(width / 2)), float(np.float32(height / 2))
        z = np.asarray(target, float) - center
        z /= np.linalg.norm(z)
        x = np.cross([0.0, 1.0, 0.0], z)
        x /= np.linalg.norm(x)
        R = np.stack([x, np.cross(z, x), z])
        self.R = R.astype(np.float32).astype(np.float64)
        self.t = (-R @ np.asarray(center, float)).astype(np.float32).astype(np.float64)


def cameras(case, seed):
    """Consecutive keyframes of a path through the room, looking across it."""
    r = np.random.RandomState(seed % (1 << 31))
    a0, step = r.uniform(0, 2 * math.pi), r.uniform(0.08, 0.2)
    f = case["width"] * (0.5 if case["width"] > 1000 else 0.82)
    out = []
    for v in range(case.get("views", 1)):
        a = a0 + step * v
        c = np.array([2.2 * math.cos(a), -0.3 + 0.1 * math.sin(3 * a), 2.2 * math.sin(a)])
        out.append(Camera(case["width"], case["height"], f, c, [-1.2 * math.cos(a + 0.3), 0.6, -1.2 * math.sin(a + 0.3)]))
    return out


def generator(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed((seed * 1_000_003 + salt) & 0x7FFFFFFFFFFF)
    return g


def uniform(g, *shape):
    return torch.rand(*shape, device=DEV, generator=g)


def normal(g, *shape):
    return torch.randn(*shape, device=DEV, generator=g)


def surface_points(n, seed, salt=1):
    """Points on the room's six walls and on sixteen boxes that stand on its floor (y down)."""
    g = generator(seed, salt)
    gb = generator(seed, 2)
    ext = torch.cat([torch.tensor([HALF], device=DEV), uniform(gb, 16, 3) * 0.3 + 0.1])
    mid = torch.cat([torch.zeros(1, 3, device=DEV), (uniform(gb, 16, 3) * 2 - 1) * 2.2])
    mid[1:, 1] = HALF[1] - ext[1:, 1]
    box = torch.where(uniform(g, n) < 0.5, 0, 1 + (uniform(g, n) * 16).long().clamp(max=15))
    p = uniform(g, n, 3) * 2 - 1
    axis = (uniform(g, n) * 3).long().clamp(max=2)
    p.scatter_(1, axis[:, None], torch.where(uniform(g, n) < 0.5, -1.0, 1.0)[:, None])
    return mid[box] + p * ext[box], axis


def make_map(n, seed, keep_all=True):
    """[14, n] parameters of a map in the middle of its optimisation; with keep_all False the part of
    the room beyond x = 0.8 has not been mapped yet."""
    g = generator(seed, 3)
    p, axis = surface_points(n, seed)
    if not keep_all:
        p[:, 0] = torch.where(p[:, 0] > 0.8, 0.8 - p[:, 0], p[:, 0])
    rgb = torch.stack([0.5 + 0.3 * torch.sin((3 + k) * p[:, 0] + k) * torch.cos((4 - k) * p[:, 2] + axis) for k in range(3)])
    out = torch.empty(14, n, device=DEV)
    out[0:3] = p.T
    out[3:6] = normal(g, 3, n) * 0.5 - 4.0 + 0.2 * math.log(3e5 / n)
    out[6:10] = F.normalize(normal(g, 4, n), dim=0)
    out[10] = normal(g, n) + 1.0
    out[11:14] = (rgb + 0.05 * normal(g, 3, n)).clamp(0, 1)
    return out


def images(case, seed, views=None):
    """Photographs: smooth shading with finer texture, values in [0, 1]."""
    g = generator(seed, 4)
    V, H, W = views or case.get("views", 1), case["height"], case["width"]
    coarse = F.interpolate(uniform(g, V, 3, 9, 12), size=(H, W), mode="bilinear", align_corners=True)
    fine = F.interpolate(normal(g, V, 3, H // 6 + 2, W // 6 + 2), size=(H, W), mode="bilinear", align_corners=True)
    return (coarse + 0.08 * fine).clamp(0, 1).contiguous()


def mlp_weights(seed):
    """Flat parameters W1 [128][80], b1, W2 [128][128], b2, W3 [16][128], b3 (output rows 11.. zero)."""
    g = generator(seed, 5)
    w1 = (uniform(g, N_HID, N_IN) * 2 - 1) / math.sqrt(N_IN)
    w2 = (uniform(g, N_HID, N_HID) * 2 - 1) / math.sqrt(N_HID)
    w3 = (uniform(g, N_OUT_PAD, N_HID) * 2 - 1) / math.sqrt(N_HID)
    b = [0.05 * normal(g, k) for k in (N_HID, N_HID, N_OUT_PAD)]
    w3[N_OUT:] = 0
    b[2][N_OUT:] = 0
    return torch.cat([w1.flatten(), b[0], w2.flatten(), b[1], w3.flatten(), b[2]])


def mlp_rows(rows, seed):
    """Training pairs: patches of photographs with depth and position, and converged parameters."""
    g = generator(seed, 6)
    x = torch.zeros(rows, N_IN, device=DEV)
    base = uniform(g, rows, 1, 3)
    x[:, :75] = (base + 0.1 * normal(g, rows, 25, 3)).clamp(0, 1).reshape(rows, 75)
    x[:, 75] = uniform(g, rows) * 5 + 0.5
    x[:, 76:78] = normal(g, rows, 2)
    x[:, 78] = x[:, 75]
    y = torch.zeros(rows, N_OUT_PAD, device=DEV)
    y[:, 0:3] = 0.5 * normal(g, rows, 3) - 4.0
    y[:, 3:7] = F.normalize(normal(g, rows, 4).abs() + torch.tensor([2.0, 0, 0, 0], device=DEV), dim=1)
    y[:, 7] = normal(g, rows)
    y[:, 8:11] = base[:, 0] + 0.05 * normal(g, rows, 3)
    return x, y


def vo_points(n, seed):
    g = generator(seed, 7)
    return (surface_points(n, seed, 8)[0] + 0.01 * normal(g, n, 3)).contiguous()


def prepare(case, seed):
    k = case["kind"]
    s = {"kind": k}
    if k == "mlp_train":
        s["mlp"] = MLP(seed=1)
        s["mlp"].set_params(mlp_weights(seed))
        s["x"], s["y"] = mlp_rows(case["rows"], seed)
        return s
    s["cams"] = cameras(case, seed)
    if k == "mlp_predict":
        s["mlp"] = MLP(seed=1)
        s["mlp"].set_params(mlp_weights(seed))
        s["image"], s["points"] = images(case, seed)[0], vo_points(case["rows"], seed)
        return s
    n, W, H, V = case["n"], case["width"], case["height"], case.get("views", 1)
    size = dict(max_views=V, max_width=W, max_height=H)
    s["params"] = make_map(n, seed, keep_all=k != "insert")
    if k == "iterate":
        s["map"] = GaussianMap(capacity=n, lr=LR, lambda_photo=case["ssim"], deterministic=case["det"],
                               tile_size=case["tile"], **size)
        s["map"].set_params(s["params"])
        s["target"] = images(case, seed)
        s["loss"], s["rgb"] = torch.empty(3, device=DEV), torch.empty(V, 3, H, W, device=DEV)
    elif k == "rasterize":
        s["map"] = GaussianMap(capacity=n, **size)
        s["target"] = images(case, seed)
        s["params"].requires_grad_(True)
    elif k == "view":
        s["map"] = GaussianMap(capacity=n, **size)
        s["map"].set_params(s["params"])
    elif k == "insert":
        s["map"] = GaussianMap(capacity=n + case["points"], **size)
        s["image"], s["points"] = images(case, seed)[0], vo_points(case["points"], seed)
        if case["learned"]:
            s["mlp"] = MLP(seed=1)
            s["mlp"].set_params(mlp_weights(seed))
            s["map"].set_initializer(s["mlp"])
    elif k == "densify":
        s["map"] = GaussianMap(capacity=2 * n, clarity_sigma=SIGMA, **size)
        s["normals"] = normal(generator(seed, 9), n, 2, 3)
    return s


def whole(gm):
    """The map's parameters in a buffer of its capacity, zero beyond its Gaussians, however many it has grown to."""
    return F.pad(gm.params(), (0, gm.cfg.capacity - gm.n))


def run(s):
    k, gm = s["kind"], s.get("map")
    if k == "iterate":
        gm.iterate(s["cams"], s["target"], s["loss"], s["rgb"])
        return {"loss": s["loss"], "rgb": s["rgb"], "grads": gm.grads(), "params": gm.params()}
    if k == "rasterize":
        s["params"].grad = None
        rgb = rasterize(s["params"], gm, s["cams"])
        loss = (rgb - s["target"]).abs().mean()
        loss.backward()
        return {"rgb": rgb.detach(), "loss": loss.detach(), "grads": s["params"].grad}
    if k == "view":
        rgb, T, top = gm.render(s["cams"], want_T=True, want_argmax=True)
        return {"rgb": rgb, "T": T, "top": top}
    if k == "insert":
        gm.set_params(s["params"])          # the map as this keyframe finds it
        count, mask = gm.insert(s["cams"][0], s["image"], s["points"], return_mask=True)
        return {"count": count, "mask": mask, "params": whole(gm)}
    if k == "densify":
        gm.set_params(s["params"])
        gm.count_dominant(s["cams"])
        split = gm.densify(s["normals"])
        return {"split": split, "params": whole(gm)}
    if k == "mlp_train":
        loss = s["mlp"].backward(s["x"], s["y"])
        grads = s["mlp"].grads()
        s["mlp"].step(1e-6)
        return {"loss": loss, "grads": grads, "params": s["mlp"].params()}
    feats = MLP.features(s["cams"][0], s["image"], s["points"])
    return {"features": feats, "out": s["mlp"].forward(feats)}


# --------------------------------------------------------------------------- work


def blended(case):
    """About how many (pixel, Gaussian) pairs blend: a Gaussian covers the ellipse where its alpha
    is at least 1/255; about a third of the map is in a view, and a pixel is full after some forty."""
    V, W, H, n = case.get("views", 1), case["width"], case["height"], case["n"]
    s = math.exp(-4.0 + 0.2 * math.log(3e5 / n)) * 1.2
    f = W * (0.5 if W > 1000 else 0.82)
    area = math.pi * ((f * s / 3.0) ** 2 + 0.3) * 2 * math.log(255 * 0.7)
    return V * min(n / 3 * area, 40 * W * H)


def work(case):
    """Each input read once and each output written once; multiplications and additions of the
    blended pairs (some 20 forward, 60 more in the adjoint) or of the network's products."""
    k = case["kind"]
    mac = N_HID * N_IN + N_HID * N_HID + N_OUT_PAD * N_HID
    flat = 4 * (mac + 2 * N_HID + N_OUT_PAD)
    if k == "mlp_train":
        # forward, input gradients and weight gradients; weights, moments and gradients in and out
        return {"bytes": case["rows"] * 4 * (N_IN + N_OUT_PAD) + 8 * flat,
                "flops": 2 * case["rows"] * (3 * mac - N_HID * N_IN)}
    if k == "mlp_predict":
        return {"bytes": case["rows"] * 4 * (3 + 75 + 2 * N_IN + N_OUT_PAD) + flat, "flops": 2 * case["rows"] * mac}
    n, px = case["n"], case.get("views", 1) * case["width"] * case["height"]
    row = 4 * 14 * n
    if k == "iterate":
        # parameters and moments in and out, gradients and parameters returned; target in, image out
        return {"bytes": 7 * row + 24 * px, "flops": 80 * blended(case) + (500 * px if case["ssim"] else 0)}
    if k == "rasterize":
        return {"bytes": 2 * row + 24 * px, "flops": 80 * blended(case)}
    if k == "view":
        return {"bytes": row + 20 * px, "flops": 20 * blended(case)}
    if k == "insert":
        return {"bytes": 2 * row + 4 * 80 * case["points"] + flat * case["learned"],
                "flops": 20 * blended(case) + 9 * n * case["points"]}
    return {"bytes": 2 * row + 24 * n, "flops": 20 * blended(case)}


# --------------------------------------------------------------------------- the same in 64 bits


def project64(P, cam):
    """Screen quantities of [14, N] float64 parameters: (u, v, a, b, c, opacity, rgb) [9, N], depth,
    radius, in front of the camera."""
    R, t = torch.tensor(cam.R, device=DEV), torch.tensor(cam.t, device=DEV)
    x, y, z = R @ P[0:3] + t[:, None]
    w, i, j, k = P[6:10] / P[6:10].norm(dim=0)
    rot = torch.stack([1 - 2 * (j * j + k * k), 2 * (i * j - w * k), 2 * (i * k + w * j),
                       2 * (i * j + w * k), 1 - 2 * (i * i + k * k), 2 * (j * k - w * i),
                       2 * (i * k - w * j), 2 * (j * k + w * i), 1 - 2 * (i * i + j * j)]).view(3, 3, -1)
    M = rot * P[3:6].exp()[None]
    S = torch.einsum("akn,bkn->abn", M, M)
    front = z > np.float64(np.float32(0.2))
    z = torch.where(front, z, torch.ones_like(z))
    lx, ly = 1.3 * 0.5 * cam.width / cam.fx, 1.3 * 0.5 * cam.height / cam.fy
    o = torch.zeros_like(z)
    J = torch.stack([cam.fx / z, o, -cam.fx * (x / z).clamp(-lx, lx) / z,
                     o, cam.fy / z, -cam.fy * (y / z).clamp(-ly, ly) / z]).view(2, 3, -1)
    T = torch.einsum("rkn,kc->rcn", J, R)
    C = torch.einsum("ran,abn,sbn->rsn", T, S, T)
    A, B, D = C[0, 0] + 0.3, C[0, 1], C[1, 1] + 0.3
    det = A * D - B * B
    mid = 0.5 * (A + D)
    radius = torch.ceil(3 * (mid + (mid * mid - det).clamp(min=0.1).sqrt()).sqrt()).detach()
    scr = torch.stack([cam.fx * x / z + cam.cx, cam.fy * y / z + cam.cy, D / det, -B / det, A / det,
                       torch.sigmoid(P[10]), P[11], P[12], P[13]])
    return scr, z.detach(), radius, front & (det.detach() > 0)


def bins64(scr, z, radius, ok, W, H, tile=16):
    """Ids sorted by (tile, depth) and the ranges of the tiles."""
    with torch.no_grad():
        u, v = scr[0], scr[1]
        x0, x1 = (u - radius).ceil().clamp(min=0), (u + radius).floor().clamp(max=W - 1)
        y0, y1 = (v - radius).ceil().clamp(min=0), (v + radius).floor().clamp(max=H - 1)
        ok = ok & (x0 <= x1) & (y0 <= y1)
        ids = torch.nonzero(ok)[:, 0]
        ids = ids[torch.sort(z[ids].float(), stable=True)[1]]
        tx, ty = (x0[ids] // tile).long(), (y0[ids] // tile).long()
        w, h = (x1[ids] // tile).long() - tx + 1, (y1[ids] // tile).long() - ty + 1
        cnt = w * h
        own = torch.repeat_interleave(torch.arange(ids.numel(), device=DEV), cnt)
        loc = torch.arange(own.numel(), device=DEV) - (cnt.cumsum(0) - cnt)[own]
        nx, ny = (W + tile - 1) // tile, (H + tile - 1) // tile
        key = (ty[own] + loc // w[own]) * nx + tx[own] + loc % w[own]
        key, order = torch.sort(key, stable=True)
        count = torch.bincount(key, minlength=nx * ny)
        return ids[own[order]], count.cumsum(0) - count, count, nx


def composite64(scr, z, radius, ok, W, H, upstream=None, tile=16):
    """Image [3, H, W] and transmittance [H, W]; with `upstream` [3, H, W] the gradient of scr instead."""
    ids, first, count, nx = bins64(scr, z, radius, ok, W, H, tile)
    rgb, Tm = torch.zeros(3, H, W, device=DEV, dtype=torch.float64), torch.ones(H, W, device=DEV, dtype=torch.float64)
    grad = torch.zeros_like(scr)
    amin, amax, tmin = (float(np.float32(q)) for q in (1 / 255, 0.99, 1e-4))
    order = torch.sort(count, descending=True)[1]
    lens = count[order].cpu()
    px = torch.arange(tile * tile, device=DEV)
    b = 0
    while b < len(lens) and int(lens[b]) > 0:
        L = int(lens[b])
        e = min(len(lens), b + max(1, (1 << 24) // (L * tile * tile)))
        t = order[b:e]
        b = e
        slot = torch.arange(L, device=DEV)[None]
        there = slot < count[t][:, None]
        g = ids[(first[t][:, None] + slot).clamp(max=ids.numel() - 1)]
        X, Y = (t % nx)[:, None] * tile + px % tile, (t // nx)[:, None] * tile + px // tile
        inside = (X < W) & (Y < H)
        Xc, Yc = X.clamp(max=W - 1), Y.clamp(max=H - 1)
        with torch.enable_grad() if upstream is not None else torch.no_grad():
            q = scr.detach()[:, g].requires_grad_(upstream is not None)
            dx, dy = X[:, None].double() - q[0][..., None], Y[:, None].double() - q[1][..., None]
            power = -0.5 * (q[2][..., None] * dx * dx + q[4][..., None] * dy * dy) - q[3][..., None] * dx * dy
            alpha = (q[5][..., None] * power.exp()).clamp(max=amax)
            r = radius[g][..., None]
            hit = (there[..., None] & (dx.abs() <= r) & (dy.abs() <= r) & (alpha >= amin)).detach()
            l = torch.log1p(-alpha * hit)
            c = l.cumsum(1)
            on = hit & (c.detach() >= math.log(tmin))
            wgt = alpha * on * (c - l).exp()
            col = torch.einsum("clk,lkp->clp", q[6:9], wgt)
            if upstream is None:
                Tl = (l * on).sum(1).exp()
                rgb[:, Yc[inside], Xc[inside]] = col[:, inside]
                Tm[Yc[inside], Xc[inside]] = Tl[inside]
            else:
                (col * (upstream[:, Yc, Xc] * inside)).sum().backward()
                grad.index_add_(1, g.reshape(-1), q.grad.reshape(9, -1))
    return grad if upstream is not None else (rgb, Tm)


def render64(P, cams):
    P = P.detach().double()
    out = [composite64(*project64(P, c), c.width, c.height) for c in cams]
    return torch.stack([o[0] for o in out]), torch.stack([o[1] for o in out])


def gradients64(P, cams, upstream):
    """Gradient of sum(upstream * image) with respect to the parameters."""
    P = P.detach().double().requires_grad_(True)
    for c, up in zip(cams, upstream):
        scr, z, radius, ok = project64(P, c)
        g = composite64(scr.detach(), z, radius, ok, c.width, c.height, up)
        torch.autograd.backward(scr, g)
    return P.grad


def ssim64(x, y):
    k = torch.arange(11, device=DEV, dtype=torch.float64) - 5
    w = torch.exp(-k * k / (2 * 1.5 ** 2))
    w = w / w.sum()

    def blur(a):
        a = a.flatten(0, 1)[:, None]
        a = F.pad(a, (5, 5, 5, 5))
        a = sum(w[i] * a[..., i:i + a.shape[-1] - 10] for i in range(11))
        a = sum(w[i] * a[..., i:i + a.shape[-2] - 10, :] for i in range(11))
        return a[:, 0].view_as(x)
    mx, my = blur(x), blur(y)
    c1, c2 = 0.01 ** 2, 0.03 ** 2
    return ((2 * mx * my + c1) * (2 * (blur(x * y) - mx * my) + c2)
            / ((mx * mx + my * my + c1) * (blur(x * x) - mx * mx + blur(y * y) - my * my + c2)))


def mlp64(flat, x):
    w = flat.split([N_HID * N_IN, N_HID, N_HID * N_HID, N_HID, N_OUT_PAD * N_HID, N_OUT_PAD])
    h = F.gelu(x @ w[0].view(N_HID, N_IN).T + w[1])
    h = F.gelu(h @ w[2].view(N_HID, N_HID).T + w[3])
    return h @ w[4].view(N_OUT_PAD, N_HID).T + w[5]


def features64(cam, image, pts):
    R, t = torch.tensor(cam.R, device=DEV), torch.tensor(cam.t, device=DEV)
    x, y, z = R @ pts.double().T + t[:, None]
    zz = z.clamp(min=1e-6)
    u = torch.floor(cam.fx * x / zz + cam.cx + 0.5).clamp(0, cam.width - 1).long()
    v = torch.floor(cam.fy * y / zz + cam.cy + 0.5).clamp(0, cam.height - 1).long()
    d = torch.arange(-2, 3, device=DEV)
    X = (u[:, None, None] + d[None, None, :]).clamp(0, cam.width - 1).expand(-1, 5, 5)
    Y = (v[:, None, None] + d[None, :, None]).clamp(0, cam.height - 1).expand(-1, 5, 5)
    patch = image.double()[:, Y, X].permute(1, 2, 3, 0).reshape(len(pts), 75)
    return torch.cat([patch, torch.stack([z, x, y, z, torch.zeros_like(z)], 1)], 1)


def adam64(p, g, lr, eps):
    """The first step from zero moments: the bias corrections cancel the decays."""
    return p - lr * g / (g.abs() + eps)


def exact(case, seed):
    k = case["kind"]
    if k == "mlp_train":
        w = mlp_weights(seed).double().requires_grad_(True)
        x, y = mlp_rows(case["rows"], seed)
        loss = (mlp64(w, x.double()) - y.double())[:, :N_OUT].square().mean()
        loss.backward()
        g = w.grad.clone()
        return {"loss": loss.detach().view(1), "grads": g, "params": adam64(w.detach(), g, float(np.float32(1e-6)), 1e-8)}
    cams = cameras(case, seed)
    if k == "mlp_predict":
        f = features64(cams[0], images(case, seed)[0], vo_points(case["rows"], seed))
        return {"features": f, "out": mlp64(mlp_weights(seed).double(), f)}
    P = make_map(case["n"], seed, keep_all=k != "insert").double()
    if k == "densify":
        return None      # which Gaussians split hangs on counts of pixels at a threshold
    if k == "view":
        rgb, T = render64(P, cams)
        return {"rgb": rgb, "T": T, "top": None}
    if k == "insert":
        return {"count": None, "mask": None, "params": insert64(case, seed, P, cams[0])}
    rgb = render64(P, cams)[0].requires_grad_(True)
    tgt = images(case, seed).double()
    if k == "rasterize":
        loss = (rgb - tgt).abs().mean()
        loss.backward()
        return {"rgb": rgb.detach(), "loss": loss.detach(), "grads": gradients64(P, cams, rgb.grad)}
    lp = float(np.float32(case["ssim"]))
    photo = sum((1 - lp) * (a - b).abs().mean() for a, b in zip(rgb, tgt))
    if lp:
        photo = photo + sum(lp * (1 - s.mean()) for s in ssim64(rgb, tgt))
    photo.backward()
    scales = P[3:6].detach().clone().requires_grad_(True)
    reg = scales.exp().min(dim=0).values.clamp(min=float(np.float32(0.01))).mean()
    reg.backward()
    g = gradients64(P, cams, rgb.grad)
    g[3:6] += scales.grad
    lr = torch.tensor([LR[i] for i in (0, 0, 0, 1, 1, 1, 2, 2, 2, 2, 3, 4, 4, 4)], device=DEV, dtype=torch.float32)
    return {"loss": torch.stack([photo + reg, photo, reg]).detach(), "rgb": rgb.detach(), "grads": g,
            "params": adam64(P, g, lr.double()[:, None], 1e-15)}


def insert64(case, seed, P, cam):
    pts, image = vo_points(case["points"], seed), images(case, seed)[0]
    T = render64(P, [cam])[1][0]
    R, t = torch.tensor(cam.R, device=DEV), torch.tensor(cam.t, device=DEV)
    x, y, z = R @ pts.double().T + t[:, None]
    front = z > 0.2
    zz = torch.where(front, z, torch.ones_like(z))
    u, v = torch.floor(cam.fx * x / zz + cam.cx + 0.5), torch.floor(cam.fy * y / zz + cam.cy + 0.5)
    seen = front & (u >= 0) & (u < cam.width) & (v >= 0) & (v < cam.height)
    u, v = torch.where(seen, u, 0).long(), torch.where(seen, v, 0).long()
    keep = ~(seen & (1 - T[v, u] > 0.99))
    d2 = (pts.double()[:, None, :] - P[0:3].T[None]).square().sum(-1) if case["n"] else None
    rms = d2.topk(3, dim=1, largest=False)[0].mean(1).sqrt()
    new = torch.zeros(14, len(pts), device=DEV, dtype=torch.float64)
    new[0:3] = pts.double().T
    new[3:6] = rms.clamp(min=1e-30).log().clamp(-7, -1)
    new[6] = 1
    new[11:14] = image.double()[:, v, u]
    if case["learned"]:
        o = mlp64(mlp_weights(seed).double(), features64(cam, image, pts))
        fine = ((o[:, 0:3] >= -9) & (o[:, 0:3] <= 1)).all(1) & (o[:, 3:7].square().sum(1) > 1e-8)
        new[3:14] = torch.where(fine[None], o[:, :11].T, new[3:14])
    return F.pad(torch.cat([P, new[:, keep]], 1), (0, int((~keep).sum())))
