"""What this framework's speed is measured on: the work its users have it do, through its public entry points.

A scene of trained Gaussians is converted into triangle fans (plain, three fans per Gaussian, or behind the learned
initializer), the fans are rendered, differentiated, fine-tuned and pruned, the initializer is trained on targets drawn from
the source Gaussians, and the finished mesh is ray traced.  Every family has one listed case or two; `draw` spreads the sizes
of the same families.  Scenes are flat Gaussians on a sphere and a torus (half of them in blobs where "clustered"), stored in
Morton order of their means as the framework's documentation asks for, or a random cloud for the smallest calls.

`exact` computes the same outputs in 64 bits with plain torch: pairs of triangles and pixels enumerated from bounding boxes,
sorted by (pixel, depth) and composited in full.
"""
import math

import torch

import paper_2502_07754_gb300 as ms
from paper_2502_07754_gb300 import api
from paper_2502_07754_gb300.finetune import FanFineTune

DEV = "cuda"
F64 = torch.float64
SPHERE_AREA = 4.0 * math.pi
TORUS_R, TORUS_r = 1.6, 0.3
TORUS_AREA = 4.0 * math.pi ** 2 * TORUS_R * TORUS_r
SCALE_MUL, OPAC_MUL = 2.7, 0.2
PRUNE_THRESHOLD = math.exp(-4.0)
LIGHT = (2.5, 3.0, 3.5)


def listed():
    return [
        # a trained scene loaded for rendering: conversion with degree-3 colour, coefficients kept in bfloat16
        {"name": "convert-1M", "do": "convert", "n": 1_000_000, "K": 8, "degree": 3, "bf16": True, "how": "flat"},
        # a scene of full 3D Gaussians: three fans each, float32 coefficients
        {"name": "convert3d-200k", "do": "convert", "n": 200_000, "K": 8, "degree": 3, "bf16": False, "how": "three"},
        # conversion with the learned initializer's corrections predicted in the same call
        {"name": "convert-init-3M", "do": "convert", "n": 3_000_000, "K": 8, "degree": 3, "bf16": True, "how": "mlp"},
        # the smallest render and adjoint in use (a thumbnail, a test scene): latency and launches
        {"name": "view-1k-128", "do": "view", "n": 1000, "K": 8, "w": 128, "h": 128, "scene": "random", "tile": 16, "kbuf": 8},
        # a NeRF-synthetic sized view of a mid-size scene, differentiated to the vertices
        {"name": "view-200k-800", "do": "view", "n": 200_000, "K": 8, "w": 800, "h": 800, "scene": "surface", "tile": 16, "kbuf": 8},
        # a viewer's frame: forward only
        {"name": "render-1M-1080p", "do": "render", "n": 1_000_000, "K": 8, "w": 1920, "h": 1080, "scene": "clustered", "tile": 16, "kbuf": 8},
        # one fine-tuning step of the paper on one view: render, L1 + SSIM, adjoint, Adam
        {"name": "step-1M-1080p", "do": "step", "n": 1_000_000, "K": 8, "w": 1920, "h": 1080, "scene": "clustered"},
        # a batch of sixteen views of mixed resolution, six triangles a fan, forward and adjoint
        {"name": "batch-3M-16views", "do": "batch", "n": 3_000_000, "K": 6, "views": 16, "w": 1920, "h": 1080, "tile": 8},
        # one full-batch training step of the initializer on the pairs of four scenes
        {"name": "train-500k", "do": "train", "n": 500_000, "K": 8},
        # the source Gaussians themselves drawn into eight views: the targets the initializer's pairs come from
        {"name": "targets-250k-8views", "do": "targets", "n": 250_000, "views": 8, "w": 1920, "h": 1080},
        # a finished mesh ray traced with a point light's shadows, its BVH built for the frame
        {"name": "trace-200k-800", "do": "trace", "n": 200_000, "K": 8, "w": 800, "h": 800, "light": True},
        # the pruning step between epochs, with face masks and the optimizer's moments
        {"name": "prune-1M", "do": "prune", "n": 1_000_000, "K": 8},
    ]


def draw(rng):
    def log(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    do = rng.choice(["convert", "convert", "convert", "view", "view", "render", "step", "batch", "train", "targets", "trace", "prune"])
    if do == "convert":
        how = rng.choice(["flat", "three", "mlp"])
        n = log(1000, {"flat": 1_000_000, "three": 200_000, "mlp": 3_000_000}[how])
        return {"do": do, "n": n, "K": rng.choice([5, 6, 8, 8, 12]), "degree": rng.choice([0, 1, 2, 3, 3]), "bf16": rng.random() < 0.5, "how": how}
    if do == "view":
        return {"do": do, "n": log(1000, 200_000), "K": rng.choice([5, 6, 8, 8, 12]), "w": log(96, 800), "h": log(96, 800),
                "scene": rng.choice(["random", "surface", "surface"]), "tile": rng.choice([8, 16, 16]), "kbuf": rng.choice([8, 8, 16])}
    if do == "render":
        return {"do": do, "n": log(200_000, 1_000_000), "K": rng.choice([6, 8, 8]), "w": log(640, 1920), "h": log(480, 1080),
                "scene": rng.choice(["surface", "clustered"]), "tile": rng.choice([8, 16, 16]), "kbuf": 8}
    if do == "step":
        return {"do": do, "n": log(200_000, 1_000_000), "K": rng.choice([6, 8, 8]), "w": log(640, 1920), "h": log(480, 1080), "scene": rng.choice(["surface", "clustered"])}
    if do == "batch":
        return {"do": do, "n": log(300_000, 3_000_000), "K": rng.choice([6, 8]), "views": rng.randint(2, 8), "w": log(640, 1920), "h": log(480, 1080),
                "tile": rng.choice([8, 16])}
    if do == "train":
        return {"do": do, "n": log(20_000, 500_000), "K": rng.choice([6, 8, 12])}
    if do == "targets":
        return {"do": do, "n": log(50_000, 250_000), "views": rng.randint(2, 8), "w": log(512, 1920), "h": log(400, 1080)}
    if do == "trace":
        return {"do": do, "n": log(5000, 200_000), "K": rng.choice([6, 8]), "w": log(200, 800), "h": log(200, 800), "light": rng.random() < 0.5}
    return {"do": do, "n": log(50_000, 1_000_000), "K": rng.choice([6, 8, 8])}


# ---------------------------------------------------------------- cameras and scenes


class Camera:
    """Pinhole camera in the form the framework takes: OpenCV axes, rows of R_cw = right, down, forward."""

    def __init__(self, centre, w, h, fov_y=60.0):
        f = float(torch.tensor((h / 2.0) / math.tan(math.radians(fov_y) / 2.0), dtype=torch.float32))
        self.width, self.height, self.fx, self.fy, self.cx, self.cy, self.znear = w, h, f, f, w / 2.0, h / 2.0, 0.01
        C = torch.tensor(centre, dtype=F64)
        z = -C / C.norm()
        up = torch.tensor([0.0, 1.0, 0.0] if abs(float(z[1])) < 0.99 else [0.0, 0.0, 1.0], dtype=F64)
        x = torch.linalg.cross(z, up)
        x = x / x.norm()
        self.R_cw = torch.stack([x, torch.linalg.cross(z, x), z]).float()
        self.C = C.float()


def cameras(case):
    """One camera on an orbit, or `views` of them on a Fibonacci sphere (of mixed sizes up to w x h in a batch)."""
    w, h = case["w"], case["h"]
    if "views" not in case:
        d, e = (4.0 if case.get("scene") == "random" else 3.0), math.radians(0.0 if case.get("scene") == "random" else 20.0)
        return [Camera((0.0, d * math.sin(e), d * math.cos(e)), w, h)]
    n, out = case["views"], []
    for i in range(n):
        z = 1.0 - 2.0 * (i + 0.5) / n
        r, phi = math.sqrt(1.0 - z * z), math.pi * (3.0 - math.sqrt(5.0)) * (i + 0.5)
        mixed = case["do"] == "batch"
        d = 3.0 + 2.0 * (0.61803398875 * i % 1.0) if mixed else 3.5
        s = (1.0, 0.42, 0.67, 0.74)[i % 4] if mixed else 1.0
        out.append(Camera((d * r * math.cos(phi), d * z, d * r * math.sin(phi)), max(16, int(w * s)), max(16, int(h * s))))
    return out


def rng_of(seed, salt=0):
    return torch.Generator(DEV).manual_seed(int(seed) * 1000003 + salt)


def randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=F64)


def rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=F64)


def unit(v):
    return v / v.norm(dim=-1, keepdim=True)


def morton(means):
    lo, hi = means.amin(0), means.amax(0)
    q = ((means - lo) / (hi - lo).clamp_min(1e-30) * 1023.0).long().clamp(0, 1023)
    code = torch.zeros(len(means), dtype=torch.long, device=means.device)
    for b in range(10):
        for a in range(3):
            code |= ((q[:, a] >> b) & 1) << (3 * b + a)
    return code.sort(stable=True).indices


def surface_points(g, n, clustered):
    """Points and normals on a unit sphere and a torus, by area; with `clustered` half of them in 256 blobs."""
    on_torus = rand(g, n) < TORUS_AREA / (SPHERE_AREA + TORUS_AREA)
    u, v, s = rand(g, n) * 2 * math.pi, rand(g, n) * 2 * math.pi, unit(randn(g, n, 3))
    v = v - (TORUS_r / TORUS_R) * torch.sin(v)  # denser on the outer side, as by area
    if clustered:
        cs, cu, cv = unit(randn(g, 256, 3)), rand(g, 256) * 2 * math.pi, rand(g, 256) * 2 * math.pi
        blob, pick = rand(g, n) < 0.5, torch.randint(0, 256, (n,), generator=g, device=DEV)
        off = 0.05 * randn(g, n, 3)
        s = torch.where(blob[:, None], unit(cs[pick] + off), s)
        u = torch.where(blob, cu[pick] + off[:, 0] / (TORUS_R + TORUS_r * torch.cos(cv[pick])), u)
        v = torch.where(blob, cv[pick] + off[:, 1] / TORUS_r, v)
    nt = torch.stack([torch.cos(v) * torch.cos(u), torch.cos(v) * torch.sin(u), torch.sin(v)], 1)
    pt = nt * TORUS_r + TORUS_R * torch.stack([torch.cos(u), torch.sin(u), torch.zeros_like(u)], 1)
    return torch.where(on_torus[:, None], pt, s), torch.where(on_torus[:, None], nt, s)


def quat_of(R):
    """(w, x, y, z) of rotation matrices: the column of the symmetric 4 x 4 form with the largest diagonal."""
    m = R.reshape(-1, 9).T
    t = torch.stack([m[0] + m[4] + m[8], m[0] - m[4] - m[8], m[4] - m[0] - m[8], m[8] - m[0] - m[4]], 1)
    a, b, c = m[7] - m[5], m[2] - m[6], m[3] - m[1]
    d, e, f = m[1] + m[3], m[2] + m[6], m[5] + m[7]
    rows = torch.stack([torch.stack([1 + t[:, 0], a, b, c], 1), torch.stack([a, 1 + t[:, 1], d, e], 1),
                        torch.stack([b, d, 1 + t[:, 2], f], 1), torch.stack([c, e, f, 1 + t[:, 3]], 1)], 1)
    return unit(rows[torch.arange(len(t), device=t.device), t.argmax(1)])


def gaussians(case, seed):
    """means, log_scales, quats, opacity, sh (float32, sh as bfloat16 where asked), as a loaded scene holds them."""
    g, n = rng_of(seed), case["n"]
    degree = case.get("degree", 0)
    kind = case.get("scene", "clustered")
    if kind == "random":
        means, ls, quats = rand(g, n, 3) * 2 - 1, rand(g, n, 3) * 2 - 4, unit(randn(g, n, 4))
    else:
        means, nrm = surface_points(g, n, kind == "clustered")
        helper = torch.where(nrm[:, 2:].abs() < 0.9, torch.tensor([[0.0, 0.0, 1.0]], dtype=F64, device=DEV), torch.tensor([[1.0, 0.0, 0.0]], dtype=F64, device=DEV))
        t1 = unit(torch.linalg.cross(nrm, helper))
        t2, phi = torch.linalg.cross(nrm, t1), rand(g, n, 1) * 2 * math.pi
        r2 = torch.cos(phi) * t1 + torch.sin(phi) * t2
        quats = quat_of(torch.stack([nrm, r2, torch.linalg.cross(nrm, r2)], 2))
        s12 = math.log(0.5 * math.sqrt((SPHERE_AREA + TORUS_AREA) / n)) + 0.25 * randn(g, n, 2)
        thin = math.log(1.0 / 3.0) if case.get("how") == "three" else math.log(1e-3)
        ls = torch.cat([s12[:, :1] + thin, s12], 1)
    opacity = torch.sigmoid(randn(g, n))
    if case["do"] == "prune":  # late in a fine-tune: a fifth of the fans have faded below the threshold
        p = (torch.arange(n, device=DEV, dtype=F64) + 0.5) / n
        opacity = torch.sigmoid(2.0 * math.sqrt(2.0) * torch.erfinv(2 * p - 1) - 2.5)[torch.randperm(n, generator=g, device=DEV)]
    sh = torch.randn(n, (degree + 1) ** 2, 3, generator=g, device=DEV) * 0.2
    sh[:, 0] *= 2.5
    if kind != "random":
        p = morton(means)
        means, ls, quats, opacity, sh = means[p], ls[p], quats[p], opacity[p], sh[p]
    sh = sh.bfloat16() if case.get("bf16") else sh
    return [t.contiguous() for t in (means.float(), ls.float(), quats.float(), opacity.float(), sh)]


def sh_colour(sh, means, centre):
    """Colour of every Gaussian seen from `centre`: 0.5 + sum of real spherical harmonics, clamped at zero."""
    sh = sh.to(F64)
    nb = sh.shape[1]
    x, y, z = unit(means.to(F64) - centre.to(F64)).unbind(1)
    c = math.sqrt
    pi = math.pi
    Y = [torch.full_like(x, 0.5 * c(1 / pi))]
    if nb > 1:
        k = c(3 / (4 * pi))
        Y += [-k * y, k * z, -k * x]
    if nb > 4:
        k = 0.5 * c(15 / pi)
        Y += [k * x * y, -k * y * z, 0.25 * c(5 / pi) * (2 * z * z - x * x - y * y), -k * x * z, 0.5 * k * (x * x - y * y)]
    if nb > 9:
        a, b, d = 0.125 * c(70 / pi), 0.25 * c(105 / pi), 0.125 * c(42 / pi)
        t = 4 * z * z - x * x - y * y
        Y += [-a * y * (3 * x * x - y * y), 2 * b * x * y * z, -d * y * t, 0.25 * c(7 / pi) * z * (2 * z * z - 3 * x * x - 3 * y * y), -d * x * t,
              b * z * (x * x - y * y), -a * x * (x * x - 3 * y * y)]
    return (0.5 + torch.einsum("nb,nbc->nc", torch.stack(Y, 1), sh)).clamp_min(0.0)


def rotations(quats):
    w, x, y, z = unit(quats.to(F64)).unbind(1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y), 2 * (x * y + w * z), 1 - 2 * (x * x + z * z),
                        2 * (y * z - w * x), 2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)


def kept_axes(ls):
    """The two axes left when the smallest scale is dropped (the first of equal ones)."""
    drop = ls.argmin(1)
    return (drop == 0).long(), torch.where(drop == 2, 1, 2)


def fans(G, K, centre, three=False, corr=None):
    """The conversion in 64 bits: (xyz, rgb, alpha) of the fans' vertices."""
    means, ls, quats, opacity, sh = G
    n, R, s = len(means), rotations(quats), SCALE_MUL * torch.exp(ls.to(F64))
    th = -math.pi + 2 * math.pi * torch.arange(K, device=DEV, dtype=F64) / K
    ia, ib = kept_axes(ls)
    pairs = [(0, 1), (0, 2), (1, 2)] if three else [(ia, ib)]
    col, m, sig, at = sh_colour(sh, means, centre), means.to(F64), opacity.to(F64), torch.arange(n, device=DEV)
    xyz, alpha = [], []
    for a, b in pairs:
        va = (R[:, :, a] * s[:, a, None]) if three else R[at, :, a] * s[at, a, None]
        vb = (R[:, :, b] * s[:, b, None]) if three else R[at, :, b] * s[at, b, None]
        off = torch.cos(th)[None, :, None] * va[:, None] + torch.sin(th)[None, :, None] * vb[:, None]
        op = torch.cat([sig[:, None], (OPAC_MUL * sig)[:, None].expand(n, K)], 1)
        if corr is not None:
            off = off * (1 + corr[:, 1:K + 1, None])
            op = (op * torch.exp(corr[:, K + 1:])).clamp(0, 1)
        xyz.append(torch.cat([m[:, None], m[:, None] + off], 1))
        alpha.append(op)
    rgb = col[:, None].expand(n, len(pairs) * (K + 1), 3)
    return torch.cat(xyz, 1).reshape(-1, 3), rgb.reshape(-1, 3), torch.cat(alpha, 1).reshape(-1)


def soup(case, seed):
    """The fan soup that a loaded and converted scene leaves in hand (float32)."""
    G = gaussians(case, seed)
    cams = cameras(case) if "w" in case else None
    out = fans(G, case["K"], cams[0].C.to(DEV) if cams else torch.tensor([0.0, 1.0, 3.0], device=DEV))
    return [t.float().contiguous() for t in out]


def upstream(case, seed, npx):
    """An image loss's gradient: of every channel, about 1 / pixels in size."""
    return torch.randn(npx, 4, generator=rng_of(seed, 7), device=DEV) / npx


def target(case, seed, cam):
    """A photograph to fine-tune against: smooth structure and texture in [0, 1]."""
    g = rng_of(seed, 11)
    t = torch.zeros(1, 3, cam.height, cam.width, device=DEV)
    for s, a in ((64, 0.5), (8, 0.2), (2, 0.05)):
        low = torch.randn(1, 3, cam.height // s + 2, cam.width // s + 2, generator=g, device=DEV)
        t += a * torch.nn.functional.interpolate(low, size=(cam.height, cam.width), mode="bilinear")
    out = torch.ones(cam.height * cam.width, 4, device=DEV)
    out[:, :3] = torch.sigmoid(t)[0].permute(1, 2, 0).reshape(-1, 3)
    return out


def moments(case, seed, V):
    """Adam's moments in the middle of a fine-tune, [xyz | rgb | alpha]."""
    g = rng_of(seed, 13)
    size = torch.cat([torch.full((3 * V,), 1e-5, device=DEV), torch.full((4 * V,), 1e-6, device=DEV)])
    root = size * torch.exp(0.5 * torch.randn(7 * V, generator=g, device=DEV))
    return 0.3 * root * torch.randn(7 * V, generator=g, device=DEV), root.square() * 0.1


def weights(case, seed):
    g, no = rng_of(seed, 17), 2 * (case["K"] + 1)
    return [torch.randn(a, b, generator=g, device=DEV) * s for a, b, s in ((16, 128, math.sqrt(2 / 16)), (128, 128, math.sqrt(2 / 128)), (128, no, 0.01))]


def features(G):
    """The initializer's sixteen inputs."""
    _, ls, quats, opacity, sh = [t.to(F64) for t in G]
    d = ls.sort(1, descending=True).values
    return torch.cat([ls, unit(quats), opacity[:, None], sh[:, 0], torch.exp(d - d[:, :1]), d[:, 2:] - d[:, 1:2], torch.ones_like(d[:, :1])], 1)


def pairs(case, seed):
    """Inputs and corrections of training pairs taken from fine-tunes of a scene."""
    X, g, K = features(gaussians(case, seed)).float(), rng_of(seed, 19), case["K"]
    r = X @ (torch.randn(16, 2 * (K + 1), generator=g, device=DEV) * 0.02)
    T = torch.tanh(r) * 0.3 + 0.05 * torch.randn(len(X), 2 * (K + 1), generator=g, device=DEV)
    T[:, 0] = 0.0
    return X.contiguous(), T.contiguous()


# ---------------------------------------------------------------- the cases


def prepare(case, seed):
    do, K = case["do"], case.get("K", 8)
    s = {"case": case}
    if do == "convert":
        s["G"], s["centre"] = gaussians(case, seed), (0.0, 1.0, 3.0)
        s["net"] = ms.FanMLP(K=K, weights=[w.cpu() for w in weights(case, seed)]) if case["how"] == "mlp" else None
    elif do in ("render", "view"):
        cam = cameras(case)[0]
        s["soup"] = soup(case, seed)
        s["r"] = ms.Renderer(case["n"], K, cam, ms.render_params(tile=case["tile"], kbuf=case["kbuf"]))
        s["dL"] = upstream(case, seed, cam.width * cam.height).view(cam.height, cam.width, 4)
    elif do == "step":
        cams, S = cameras(case), soup(case, seed)
        ft = FanFineTune(*S, K, cams, target(case, seed, cams[0]), lr_color=5e-4, prune_every=0)
        ft.adam.m, ft.adam.v = moments(case, seed, len(S[0]))
        ft.adam.t = 100
        s["ft"] = ft
    elif do == "batch":
        s["soup"] = soup(case, seed)
        s["r"] = ms.BatchRenderer(case["n"], K, cameras(case), ms.render_params(tile=case["tile"]))
        s["flat"] = s["r"].new_flat()
        s["dL"] = upstream(case, seed, s["r"].n_pixels)
    elif do == "train":
        s["X"], s["T"] = pairs(case, seed)
        s["net"] = net = ms.FanMLP(K=K, weights=[w.cpu() for w in weights(case, seed)])
        net.m, net.v = train_moments(case, seed, net.W.numel())
        net.step.fill_(100)
    elif do == "targets":
        G = gaussians(case, seed)
        s["G"] = G[:4] + [sh_colour(G[4], G[0], cameras(case)[0].C.to(DEV)).float().contiguous()]
        s["r"] = ms.SplatRenderer(case["n"], cameras(case))
        s["flat"] = s["r"].new_flat()
    elif do == "trace":
        s["soup"], s["cam"] = soup(case, seed), cameras(case)[0]
        s["r"] = ms.RayTracer(case["n"] * K, K)
    elif do == "prune":
        s["soup"] = soup(case, seed)
        s["m"], s["v"] = moments(case, seed, len(s["soup"][0]))
        s["mask"] = torch.randint(1, 1 << K, (case["n"],), generator=rng_of(seed, 23), device=DEV, dtype=torch.int32)
    if do in ("view", "render", "batch"):  # a renderer sizes its buffers on its first frame
        s["r"].forward(*s["soup"])
    elif do == "step":
        s["ft"].loss()
    elif do == "targets":
        s["r"].render(*s["G"], flat=s["flat"])
    return s


def train_moments(case, seed, n):
    g = rng_of(seed, 29)
    root = 1e-3 * torch.exp(0.5 * torch.randn(n, generator=g, device=DEV))
    return 0.3 * root * torch.randn(n, generator=g, device=DEV), root.square() * 0.1


def run(s):
    case = s["case"]
    do, K = case["do"], case.get("K", 8)
    if do == "convert":
        if case["how"] == "three":
            return ms.mesh_build_3d(*s["G"], case["degree"], K=K, cam_center=s["centre"])
        return ms.mesh_build(*s["G"], case["degree"], K=K, cam_center=s["centre"], mlp=s["net"])
    if do == "render":
        return s["r"].forward(*s["soup"])
    if do == "view":
        img = s["r"].forward(*s["soup"])
        return (img,) + tuple(s["r"].backward(*s["soup"], img, s["dL"]))
    if do == "step":
        ft = s["ft"]
        loss = ft.step()
        return loss, ft.xyz, ft.rgb, ft.alpha
    if do == "batch":
        s["r"].forward(*s["soup"], s["flat"])
        return (s["flat"],) + tuple(s["r"].backward(*s["soup"], s["flat"], s["dL"]))
    if do == "train":
        net = s["net"]
        loss = net.train_step(s["X"], s["T"], lr=2e-3)
        return loss, net.grads, net.W, net.m, net.v
    if do == "targets":
        return s["r"].render(*s["G"], flat=s["flat"])
    if do == "trace":
        s["r"].build(s["soup"][0])
        return s["r"].trace(*s["soup"], s["cam"], light=LIGHT if case["light"] else None, ambient=0.3 if case["light"] else 1.0, T_eps=1e-5)
    return ms.prune_faces(*s["soup"], K, face_mask=s["mask"], m=s["m"], v=s["v"])


def work(case):
    do, n, K = case["do"], case["n"], case.get("K", 8)
    V = n * (K + 1)
    px = sum(c.width * c.height for c in cameras(case)) if "w" in case else 0
    mlp = 2 * (16 * 128 + 128 * 128 + 128 * 2 * (K + 1))
    if do == "convert":
        rows = n * (44 + 3 * (case["degree"] + 1) ** 2 * (2 if case["bf16"] else 4))
        return {"bytes": rows + 28 * V * (3 if case["how"] == "three" else 1), "flops": n * (mlp if case["how"] == "mlp" else 0) + 12 * V}
    views = case.get("views", 1)
    project = 30 * V * views  # a vertex to the screen
    if do == "render":
        return {"bytes": 28 * V + 16 * px, "flops": project}
    if do in ("view", "batch"):
        return {"bytes": 56 * V + 32 * px, "flops": 3 * project}
    if do == "step":
        return {"bytes": 7 * 24 * V + 16 * px, "flops": 3 * project + 7 * 12 * V + 400 * px}
    if do == "train":
        return {"bytes": n * 4 * (16 + 2 * (K + 1)), "flops": 3 * n * mlp}
    if do == "targets":
        return {"bytes": 56 * n + 16 * px, "flops": 60 * n * views}
    if do == "trace":
        return {"bytes": 28 * V + 16 * px, "flops": 30 * V}
    return {"bytes": 84 * V + 4 * n + 0.6 * (84 * V + 4 * n), "flops": V}


# ---------------------------------------------------------------- 64 bits


def view_space(cam, p):
    R, C = cam.R_cw.to(DEV, F64), cam.C.to(DEV, F64)
    q = (p - C) @ R.T
    return q, cam.fx * q[..., 0] / q[..., 2] + cam.cx, cam.fy * q[..., 1] / q[..., 2] + cam.cy


def boxes(cam, x, y, ok):
    """Every (row, pixel x, pixel y) with the pixel's centre in the row's bounding box; x, y: rows x points."""
    i0, i1 = (x.amin(1) - 0.5).ceil().clamp(0, cam.width).long(), (x.amax(1) - 0.5).floor().clamp(-1, cam.width - 1).long()
    j0, j1 = (y.amin(1) - 0.5).ceil().clamp(0, cam.height).long(), (y.amax(1) - 0.5).floor().clamp(-1, cam.height - 1).long()
    w, h = (i1 - i0 + 1).clamp_min(0), (j1 - j0 + 1).clamp_min(0)
    cnt = torch.where(ok, w * h, 0)
    row = torch.arange(len(x), device=DEV).repeat_interleave(cnt)
    k = torch.arange(len(row), device=DEV) - (cnt.cumsum(0) - cnt)[row]
    return row, i0[row] + k % w[row], j0[row] + k // w[row]


def fan_vertices(tri, K):
    f, j = tri // K, tri % K
    c = f * (K + 1)
    return torch.stack([c, c + 1 + j, c + 1 + (j + 1) % K], 1)


def barycentrics(cam, P, px, py):
    """Perspective-correct weights of a pixel's centre in triangles P (rows x 3 x 3), their depth there, and whether it is inside."""
    q, x, y = view_space(cam, P)
    ux, uy = x - (px + 0.5)[:, None], y - (py + 0.5)[:, None]
    a, b = ux[:, [1, 2, 0]], uy[:, [1, 2, 0]]
    c, d = ux[:, [2, 0, 1]], uy[:, [2, 0, 1]]
    E = a * d - b * c
    inside = (E > 0).all(1) | (E < 0).all(1)
    w = E / q[..., 2]
    W = w.sum(1, keepdim=True)
    return w / W, E.sum(1) / W[:, 0], inside


def fragments(S, K, cam):
    """(pixel, triangle, depth, weights) of every covered pixel centre."""
    xyz, T, out = S[0].to(F64), (len(S[0]) // (K + 1)) * K, []
    for t0 in range(0, T, 1 << 21):
        tri = torch.arange(t0, min(T, t0 + (1 << 21)), device=DEV)
        P = xyz[fan_vertices(tri, K)]
        q, x, y = view_space(cam, P)
        row, px, py = boxes(cam, x, y, (q[..., 2] > cam.znear).all(1))
        del q, x, y
        for r0 in range(0, len(row), 1 << 22):
            k = slice(r0, r0 + (1 << 22))
            mu, z, inside = barycentrics(cam, P[row[k]], px[k], py[k])
            out.append(((py[k] * cam.width + px[k])[inside], tri[row[k]][inside], z[inside], mu[inside]))
    return [torch.cat(v) for v in zip(*out)]


def by_layer(pix, z, npx):
    """Order of the fragments by their rank in their pixel (nearest first), and the ranks' bounds."""
    o = z.argsort()
    o = o[pix[o].argsort(stable=True)]
    cnt = torch.bincount(pix, minlength=npx)
    rank = torch.empty_like(o)
    rank[o] = torch.arange(len(o), device=DEV) - (cnt.cumsum(0) - cnt)[pix[o]]
    o = rank.argsort(stable=True)
    return o, [0] + torch.bincount(rank).cumsum(0).tolist()


def composite(pix, col, al, npx, o, ends, g=None):
    """Front-to-back image (npx x 4); with an upstream gradient g also dL/dcolour and dL/dopacity of every fragment."""
    C, T = torch.zeros(npx, 3, device=DEV, dtype=F64), torch.ones(npx, device=DEV, dtype=F64)
    front = torch.empty_like(al)
    for a, b in zip(ends, ends[1:]):
        k = o[a:b]
        p, x = pix[k], al[k]
        front[k] = T[p]
        C[p] += (T[p] * x)[:, None] * col[k]
        T[p] *= 1 - x
    img = torch.cat([C, (1 - T)[:, None]], 1)
    if g is None:
        return img, None, None
    gc, ga = torch.empty_like(col), torch.empty_like(al)
    B, Tb = torch.zeros_like(C), torch.ones_like(T)
    for a, b in reversed(list(zip(ends, ends[1:]))):
        k = o[a:b]
        p, x = pix[k], al[k]
        gp = g[p].to(F64)
        gc[k] = gp[:, :3] * (front[k] * x)[:, None]
        ga[k] = front[k] * ((gp[:, :3] * (col[k] - B[p])).sum(1) + gp[:, 3] * Tb[p])
        B[p] = x[:, None] * col[k] + (1 - x)[:, None] * B[p]
        Tb[p] *= 1 - x
    return img, gc, ga


def exact_view(S, K, cam, g=None, loss=None):
    """The image of a fan soup and, with g (or with loss(image) -> (value, g)), the gradients of its vertices."""
    pix, tri, z, mu = fragments(S, K, cam)
    vid = fan_vertices(tri, K)
    rgb, alpha = S[1].to(F64), S[2].to(F64)
    col, al = torch.einsum("nk,nkc->nc", mu, rgb[vid]), (mu * alpha[vid]).sum(1)
    npx = cam.width * cam.height
    o, ends = by_layer(pix, z, npx)
    value = None
    if loss is not None:
        value, g = loss(composite(pix, col, al, npx, o, ends)[0])
    img, gc, ga = composite(pix, col, al, npx, o, ends, g)
    if g is None:
        return img, None, value
    d = [torch.zeros(t.shape, device=DEV, dtype=F64) for t in S]
    for r0 in range(0, len(pix), 1 << 21):
        k = slice(r0, r0 + (1 << 21))
        P, c, a = S[0].to(F64)[vid[k]].requires_grad_(), rgb[vid[k]].requires_grad_(), alpha[vid[k]].requires_grad_()
        w = barycentrics(cam, P, (pix[k] % cam.width).to(F64), (pix[k] // cam.width).to(F64))[0]
        total = (gc[k] * torch.einsum("nk,nkc->nc", w, c)).sum() + (ga[k] * (w * a).sum(1)).sum()
        for t, x in zip(d, torch.autograd.grad(total, (P, c, a))):
            t.index_add_(0, vid[k].reshape(-1), x.reshape(-1, *t.shape[1:]))
    return img, d, value


def loss_of(img, tgt, H, W, lam=0.6):
    """0.6 L1 + 0.4 (1 - SSIM), an 11 x 11 Gaussian window with sigma 1.5, zeros outside; and its gradient."""
    x = img.view(H, W, 4)[..., :3].permute(2, 0, 1).detach().requires_grad_()
    y = tgt.to(F64).view(H, W, 4)[..., :3].permute(2, 0, 1)
    win = torch.exp(-torch.arange(-5, 6, dtype=F64, device=DEV) ** 2 / 4.5)
    win = win / win.sum()

    def blur(t):
        t = torch.nn.functional.pad(t, (5, 5, 5, 5))
        t = sum(win[k] * t[:, k:k + H] for k in range(11))
        return sum(win[k] * t[:, :, k:k + W] for k in range(11))

    mx, my = blur(x), blur(y)
    sxx, syy, sxy = blur(x * x) - mx * mx, blur(y * y) - my * my, blur(x * y) - mx * my
    S = (2 * mx * my + 1e-4) * (2 * sxy + 9e-4) / ((mx * mx + my * my + 1e-4) * (sxx + syy + 9e-4))
    value = lam * (x - y).abs().mean() + (1 - lam) * (1 - S).mean()
    g = torch.zeros_like(img)
    g[:, :3] = torch.autograd.grad(value, x)[0].permute(1, 2, 0).reshape(-1, 3)
    return value.detach(), g


def adam(p, g, m, v, t, lr, eps):
    m = 0.9 * m.to(F64) + 0.1 * g
    v = 0.999 * v.to(F64) + 0.001 * g * g
    return p.to(F64) - lr * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + eps), m, v


def forward_mlp(X, W):
    gelu = torch.nn.functional.gelu
    return gelu(gelu(X @ W[0]) @ W[1]) @ W[2]


def exact(case, seed):
    do, n, K = case["do"], case["n"], case.get("K", 8)
    if do == "convert":
        G, corr = gaussians(case, seed), None
        if case["how"] == "mlp":
            W, X = [w.to(F64) for w in weights(case, seed)], features(G)
            corr = torch.cat([forward_mlp(x, W) for x in X.split(1 << 19)])
        return fans(G, K, torch.tensor([0.0, 1.0, 3.0], device=DEV), case["how"] == "three", corr)
    if do == "render":
        cam = cameras(case)[0]
        return exact_view(soup(case, seed), K, cam)[0].view(cam.height, cam.width, 4)
    if do == "view":
        cam, S = cameras(case)[0], soup(case, seed)
        img, d, _ = exact_view(S, K, cam, upstream(case, seed, cam.width * cam.height))
        return (img.view(cam.height, cam.width, 4),) + tuple(d)
    if do == "batch":
        cams, S = cameras(case), soup(case, seed)
        gs = upstream(case, seed, sum(c.width * c.height for c in cams)).split([c.width * c.height for c in cams])
        imgs, total = [], None
        for c, g in zip(cams, gs):
            img, d, _ = exact_view(S, K, c, g)
            imgs.append(img)
            total = d if total is None else [a + b for a, b in zip(total, d)]
        return (torch.cat(imgs),) + tuple(total)
    if do == "step":
        cam, S = cameras(case)[0], soup(case, seed)
        tgt = target(case, seed, cam)
        _, d, value = exact_view(S, K, cam, loss=lambda img: loss_of(img, tgt, cam.height, cam.width))
        V = len(S[0])
        m, v = [t.split([3 * V, 3 * V, V]) for t in moments(case, seed, V)]
        p = [adam(S[k].reshape(-1), d[k].reshape(-1), m[k], v[k], 101, 5e-4 * (math.exp(-3.0) if k == 0 else 1.0), 1e-15)[0] for k in range(3)]
        return value.reshape(1), p[0].view(V, 3), p[1].view(V, 3), p[2].clamp(0, 1)
    if do == "train":
        X, T = [t.to(F64) for t in pairs(case, seed)]
        W = [w.to(F64).requires_grad_() for w in weights(case, seed)]
        value, grads = 0.0, 0.0
        for x, t in zip(X.split(1 << 17), T.split(1 << 17)):
            e = (forward_mlp(x, W) - t).square().sum() / T.numel()
            grads = grads + torch.cat([d.reshape(-1) for d in torch.autograd.grad(e, W)])
            value = value + e.detach()
        flat = torch.cat([w.detach().reshape(-1) for w in W])
        return (value.reshape(1), grads) + adam(flat, grads, *train_moments(case, seed, len(flat)), 101, 2e-3, 1e-8)
    if do == "targets":
        G = gaussians(case, seed)
        colour = sh_colour(G[4], G[0], cameras(case)[0].C.to(DEV)).float().to(F64)
        return torch.cat([exact_splats(G, colour, c) for c in cameras(case)])
    if do == "trace":
        if case["light"]:
            return None  # every crossing's segment to the light against every triangle: far over the time there is
        cam = cameras(case)[0]
        return exact_view(soup(case, seed), K, cam)[0].view(cam.height, cam.width, 4)
    S = soup(case, seed)
    m, v = moments(case, seed, len(S[0]))
    mask = torch.randint(1, 1 << K, (n,), generator=rng_of(seed, 23), device=DEV, dtype=torch.int32)
    low = S[2].view(n, K + 1) < torch.tensor(PRUNE_THRESHOLD, dtype=torch.float32, device=DEV)
    face = ~(low[:, :1] & low[:, 1:] & low[:, 1:].roll(-1, 1))
    mask = mask & (face.int() << torch.arange(K, device=DEV, dtype=torch.int32)).sum(1, dtype=torch.int32)
    keep = mask != 0

    def rows(t, w):
        return t.view(n, -1)[keep].reshape(-1, w) if w > 1 else t.view(n, -1)[keep].reshape(-1)

    V = len(S[0])
    mv = [torch.cat([x.view(n, -1)[keep].reshape(-1) for x in t.split([3 * V, 3 * V, V])]) for t in (m, v)]
    return rows(S[0], 3), rows(S[1], 3), rows(S[2], 1), mv[0], mv[1], mask[keep], int(keep.sum())


def exact_splats(G, colour, cam):
    """The flat Gaussians themselves: sigma exp(-(u^2 / sa^2 + v^2 / sb^2) / 2) on their planes, cut at 2.7 scales."""
    means, ls, quats, opacity = G[:4]
    n, R = len(means), rotations(quats)
    at = torch.arange(n, device=DEV)
    ia, ib = kept_axes(ls)
    s = torch.exp(ls.to(F64))
    sa, sb, ua, ub = s[at, ia], s[at, ib], R[at, :, ia], R[at, :, ib]
    th = 2 * math.pi * (torch.arange(8, device=DEV, dtype=F64) + 0.5) / 8
    rad = 2.7 / math.cos(math.pi / 8) * 1.0001
    P = means.to(F64)[:, None] + rad * (torch.cos(th)[None, :, None] * (sa[:, None] * ua)[:, None] + torch.sin(th)[None, :, None] * (sb[:, None] * ub)[:, None])
    q, x, y = view_space(cam, P)
    row, px, py = boxes(cam, x, y, (q[..., 2] > cam.znear).all(1))
    Rc = cam.R_cw.to(DEV, F64)
    mc = view_space(cam, means.to(F64))[0]
    ca, cb = ua @ Rc.T, ub @ Rc.T
    nrm = torch.linalg.cross(ca, cb)
    out = []
    for r0 in range(0, len(row), 1 << 22):
        k = slice(r0, r0 + (1 << 22))
        f = row[k]
        d = torch.stack([(px[k] + 0.5 - cam.cx) / cam.fx, (py[k] + 0.5 - cam.cy) / cam.fy, torch.ones(len(f), device=DEV, dtype=F64)], 1)
        t = (mc[f] * nrm[f]).sum(1) / (d * nrm[f]).sum(1)
        w = t[:, None] * d - mc[f]
        u, v = (w * ca[f]).sum(1) / sa[f], (w * cb[f]).sum(1) / sb[f]
        hit = (t > cam.znear) & (u * u + v * v <= 2.7 * 2.7)
        out.append(((py[k] * cam.width + px[k])[hit], f[hit], t[hit], (opacity.to(F64)[f] * torch.exp(-0.5 * (u * u + v * v)))[hit]))
    pix, f, t, al = [torch.cat(v) for v in zip(*out)]
    npx = cam.width * cam.height
    o, ends = by_layer(pix, t, npx)
    return composite(pix, colour[f], al, npx, o, ends)[0]
