"""The work that users of the GES rasterizer have it do, as timed cases.

Each case is one pass through a public entry point (the Python layer of libges.so), with inputs
made on the GPU from a seed. Scenes follow the distributions of `scenes.make_scene` (uniform,
object, heightfield), views the cosine dynamic-resolution schedule, and the rasterizer settings
are the defaults for eager calls and the persistent queue with 16x8 tiles for captured steps (what
the autotuner picks on the 8-view batch).

`exact` restates the method in 64-bit torch operations (a dense evaluation per image block, its
gradient by autograd), sharing no code with the package.
"""
import math

import torch
import torch.nn.functional as F

from paper_2411_09156_gb300 import api
from paper_2411_09156_gb300.autograd import rasterize
from paper_2411_09156_gb300.batch import BatchPlan
from paper_2411_09156_gb300.drt import drt_sizes
from paper_2411_09156_gb300.scenes import look_at

DEV = "cuda"


def _case(name, kind, scene="object", n=100_000, views=1, w=800, h=800, sh=3, storage=0, tile="16x16", persistent=0,
          grads=True, steps=32):
    return dict(name=name, kind=kind, scene=scene, n=n, views=views, w=w, h=h, sh=sh, storage=storage, tile=tile,
                persistent=persistent, grads=grads, steps=steps)


def listed():
    return [
        # the smallest differentiable call: a small fit or a unit test, one RGB view, bound by latency
        _case("autograd-tiny-1k-128", "autograd", "uniform", 1_000, 1, 128, 128, sh=-1),
        # a viewer's or an evaluation's render of an object: forward only, default settings
        _case("render-object-100k-800", "render", "object", 100_000, 1, 800, 800),
        # fitting an object from a ragged view, the colours stored in 16 bits
        _case("autograd-object-100k-613x407-half", "autograd", "object", 100_000, 1, 613, 407, storage=1),
        # one iteration of scene training at full resolution: render, Eq. 8 loss, backward
        _case("train-scene-1.5M-1600x1040", "train", "heightfield", 1_500_000, 1, 1600, 1040, tile="16x8", persistent=1),
        # one iteration of training on a batch of ragged views, RGB colours in the odd-sized scene
        _case("train-views4-300k-rgb", "train", "heightfield", 300_007, 4, 997, 661, sh=-1, tile="16x8", persistent=1),
        # the batched dynamic-resolution step with gradients on every output
        _case("step-drt8-1.5M", "step", "heightfield", 1_500_000, 8, 1600, 1040, tile="16x8", persistent=1),
        # the largest batch: 16 views up to 1920x1080 of 3M splats
        _case("step-drt16-3M", "step", "heightfield", 3_000_000, 16, 1920, 1080, tile="16x8", persistent=1),
        # the reconstruction loss and its gradient for callers that render by other means
        _case("loss-drt8-1600x1040", "loss", views=8, w=1600, h=1040),
        # the neighbour lists that training refreshes every few hundred iterations
        _case("knn-1.5M", "knn", "heightfield", 1_500_000),
        # the surface regularization at one sample per splat: a small scene and a large one
        _case("gsr-object-100k", "gsr", "object", 100_000),
        _case("gsr-1.5M", "gsr", "heightfield", 1_500_000),
        # mesh extraction: a point for every pixel of a rendered view
        _case("levelset-1.5M-1600x1040", "levelset", "heightfield", 1_500_000, 1, 1600, 1040),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["autograd", "render", "train", "step", "loss", "knn", "gsr", "levelset"])
    scene = rng.choice(["uniform", "object", "heightfield"])
    # the uniform cloud's splats are large (log-scale -3): it stands for small fits only
    n = _log_int(rng, 500, 5_000 if scene == "uniform" else 2_000_000)
    views = rng.choice([1, 1, 2, 3, 5, 8]) if kind in ("train", "step", "loss", "autograd") else 1
    # the smallest view (a quarter of the full width in a batch) has at least a pixel per 30 splats, as
    # the smallest views of the dynamic-resolution batches do
    least = math.sqrt(n / 24.0) * (4.0 if views > 1 else 1.0) if kind not in ("loss", "knn", "gsr") else 64.0
    w = _log_int(rng, max(64.0, least), 400 if scene == "uniform" and kind != "loss" else 1700)
    h = max(16, int(w * rng.uniform(0.8 if least > 64.0 else 0.55, 1.1)))
    case = _case("", kind, scene, n, views, w, h, sh=rng.choice([-1, 0, 1, 2, 3, 3, 3]),
                 storage=rng.choice([0, 0, 0, 1, 2]), tile=rng.choice(["16x16", "16x8", "16x8", "8x16", "8x8", "32x8"]),
                 persistent=1 if kind in ("train", "step") else rng.choice([0, 1]), grads=rng.random() < 0.7,
                 steps=rng.choice([7, 16, 32, 33]))
    del case["name"]
    return case


# --------------------------------------------------------------------------- inputs
def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1009 + salt)
    return g


def _quat_of(m):
    """Unit quaternions (w, x, y, z) of rotation matrices whose trace may be anything: the eigenvector
    form through the largest of the four squared components."""
    t = torch.stack([m[:, 0, 0] + m[:, 1, 1] + m[:, 2, 2], m[:, 0, 0] - m[:, 1, 1] - m[:, 2, 2],
                     m[:, 1, 1] - m[:, 0, 0] - m[:, 2, 2], m[:, 2, 2] - m[:, 0, 0] - m[:, 1, 1]], 1)
    a, b, c = m[:, 2, 1] - m[:, 1, 2], m[:, 0, 2] - m[:, 2, 0], m[:, 1, 0] - m[:, 0, 1]
    d, e, f = m[:, 0, 1] + m[:, 1, 0], m[:, 0, 2] + m[:, 2, 0], m[:, 1, 2] + m[:, 2, 1]
    one = t + 1.0
    cand = torch.stack([torch.stack([one[:, 0], a, b, c], 1), torch.stack([a, one[:, 1], d, e], 1),
                        torch.stack([b, d, one[:, 2], f], 1), torch.stack([c, e, f, one[:, 3]], 1)], 1)
    q = cand[torch.arange(m.shape[0], device=m.device), t.argmax(1)]
    return q / q.norm(dim=1, keepdim=True)


def _scene(case, seed):
    """(pos_op, lscale_beta, quat, color) with the distributions of scenes.make_scene."""
    n, kind, sh = case["n"], case["scene"], case["sh"]
    g = _gen(seed, 1)
    rnd = lambda *s: torch.rand(*s, generator=g, device=DEV)
    nrm = lambda *s: torch.randn(*s, generator=g, device=DEV)
    if kind == "uniform":
        mu, ls, q = 2.0 * rnd(n, 3) - 1.0, -3.0 + 0.5 * nrm(n, 3), nrm(n, 4)
        op, beta = torch.sigmoid(nrm(n)), 1.0 + 3.0 * rnd(n)
    elif kind == "object":
        mu, ls, q = 0.5 * nrm(n, 3), -4.5 + 0.7 * nrm(n, 3), nrm(n, 4)
        op, beta = torch.sigmoid(1.5 * nrm(n)), 1.0 + 5.0 * rnd(n)
    else:
        amps, freqs = 0.02 + 0.055 * rnd(4), 0.5 + 2.5 * rnd(4)
        angs, phases = 2.0 * math.pi * rnd(4), 2.0 * math.pi * rnd(4)
        kx, ky = freqs * torch.cos(angs), freqs * torch.sin(angs)
        xy = 4.0 * rnd(n, 2) - 2.0
        arg = xy[:, :1] * kx + xy[:, 1:] * ky + phases
        z = (amps * torch.sin(arg)).sum(1)
        hx, hy = (amps * kx * torch.cos(arg)).sum(1), (amps * ky * torch.cos(arg)).sum(1)
        mu = torch.cat([xy, z[:, None]], 1) + 0.02 * nrm(n, 3)
        nv = F.normalize(torch.stack([-hx, -hy, torch.ones_like(hx)], 1), dim=1)
        t1 = torch.zeros_like(nv)
        t1[:, 0] = 1.0
        t1 = F.normalize(t1 - nv * nv[:, :1], dim=1)
        t2 = torch.linalg.cross(nv, t1)
        th = 2.0 * math.pi * rnd(n, 1)
        a1 = torch.cos(th) * t1 + torch.sin(th) * t2
        q = _quat_of(torch.stack([a1, torch.linalg.cross(nv, a1), nv], 2))
        ls = torch.cat([-5.0 + 0.8 * nrm(n, 2), -9.0 + 0.3 * nrm(n, 1)], 1)
        op, beta = torch.sigmoid(nrm(n)), 1.0 + 5.0 * rnd(n)
    q = F.normalize(q, dim=1) * (0.5 + 1.5 * rnd(n, 1))
    color = rnd(n, 3) if sh < 0 else 0.2 * nrm(n, (sh + 1) ** 2, 3)
    color = color.to(api.COLOR_DTYPES[case["storage"]])
    return [torch.cat([mu, op[:, None]], 1).contiguous(), torch.cat([ls, beta[:, None]], 1).contiguous(),
            q.contiguous(), color.contiguous()]


def _cameras(case, seed):
    sizes = drt_sizes(case["w"], case["h"], case["views"])
    d = torch.randn(case["views"], 3, generator=torch.Generator().manual_seed(int(seed) * 1009 + 2))
    if case["scene"] == "heightfield":  # cameras above the surface
        d[:, 2] = d[:, 2].abs() + 0.7
    d = (d / d.norm(dim=1, keepdim=True)).tolist()
    r = 4.0 if case["views"] == 1 else 5.0
    return [look_at([r * x for x in d[k]], (0.0, 0.0, 0.0), *sizes[k]) for k in range(case["views"])]


def _config(case):
    tw, th = (int(x) for x in case["tile"].split("x"))
    return api.GESConfig(tile_w=tw, tile_h=th, batch=128, sh_degree=case["sh"], persistent=case["persistent"],
                         color_storage=case["storage"])


def _upstream(case, seed, pixels):
    g = _gen(seed, 3)
    return [torch.randn(k * pixels, generator=g, device=DEV) for k in (3, 1, 1, 3)]


def _images(case, seed, sizes, salt):
    """Images with photograph-like structure: smooth shapes with some texture, planar per view."""
    g = _gen(seed, salt)
    out = []
    for w, h in sizes:
        img = 0.5 * torch.ones(1, 3, h, w, device=DEV)
        for cells, amp in ((3, 0.25), (17, 0.12), (61, 0.08)):
            low = torch.randn(1, 3, cells, cells, generator=g, device=DEV)
            img = img + amp * F.interpolate(low, size=(h, w), mode="bilinear", align_corners=True)
        out.append((img + 0.02 * torch.randn(1, 3, h, w, generator=g, device=DEV)).clamp(0.0, 1.0).reshape(-1))
    return torch.cat(out).contiguous()


def _samples(case, seed):
    n = case["n"]
    return torch.arange(n, dtype=torch.int32, device=DEV), torch.randn(n, 3, generator=_gen(seed, 5), device=DEV)


# --------------------------------------------------------------------------- the cases
def prepare(case, seed):
    kind = case["kind"]
    if kind == "loss":
        sizes = drt_sizes(case["w"], case["h"], case["views"])
        target = _images(case, seed, sizes, 6)
        noise = torch.randn(target.shape, generator=_gen(seed, 7), device=DEV)
        return dict(kind=kind, color=(target + 0.05 * noise).clamp(0.0, 1.0), target=target, sizes=sizes)
    x = _scene(case, seed)
    st = dict(kind=kind, x=x)
    if kind == "knn":
        return st
    if kind == "gsr":
        splat, z = _samples(case, seed)
        return st | dict(knn=api.knn(x[0]), splat=splat, z=z, cfg=_config(case), grads=case["grads"])
    cams, cfg = _cameras(case, seed), _config(case)
    sizes = [(c.width, c.height) for c in cams]
    pixels = sum(w * h for w, h in sizes)
    if kind == "train":
        st["plan"] = BatchPlan(case["n"], cams, cfg, x, target=_images(case, seed, sizes, 6))
    elif kind == "step":
        st["plan"] = BatchPlan(case["n"], cams, cfg, x, upstream=_upstream(case, seed, pixels))
    else:
        st["rast"] = api.Rasterizer(case["n"], cams, cfg)
    if kind == "autograd":
        st["x"] = [t.requires_grad_(True) for t in x]
        st["up"] = _upstream(case, seed, pixels)
    if kind == "levelset":
        out = st["rast"].forward(*x)
        pix = torch.arange(pixels, dtype=torch.int32, device=DEV)
        return dict(kind=kind, x=x, cams=cams, cfg=cfg, steps=case["steps"], depth=out["depth"].clone(),
                    alpha=out["alpha"].clone(), pixels=torch.stack([torch.zeros_like(pix), pix], 1).contiguous())
    return st


def run(st):
    kind = st["kind"]
    if kind == "autograd":
        out = rasterize(*st["x"], st["rast"])
        grads = torch.autograd.grad(out, st["x"], st["up"])
        return dict(out=list(out), grads=list(grads))
    if kind == "render":
        return st["rast"].forward(*st["x"])
    if kind == "train":
        plan = st["plan"]
        grads = plan.step()
        return dict(loss=plan.loss, color=plan.rast.out["color"], grads=grads)
    if kind == "step":
        plan = st["plan"]
        grads = plan.step()
        return dict(out={k: plan.rast.out[k] for k in ("color", "depth", "alpha", "normal")}, grads=grads)
    if kind == "loss":
        loss, g = api.loss_rgb(st["color"], st["target"], st["sizes"])
        return dict(loss=loss, g=g)
    if kind == "knn":
        return api.knn(st["x"][0])
    if kind == "gsr":
        r = api.gsr(*st["x"][:3], st["knn"], st["splat"], st["z"], st["cfg"], grads=st["grads"])
        return {k: v for k, v in r.items() if v is not None}
    return api.levelset(*st["x"][:3], st["cams"], st["depth"], st["alpha"], st["pixels"], n_steps=st["steps"],
                        cfg=st["cfg"])


def work(case):
    """Inputs read once and outputs written once; operations by the method's own count: about 40
    blended splats per pixel at 26 flops forward and 104 backward (measured on the 8-view batch, an
    eighth as many in the small uniform cloud's), 300 and 500 per (splat, view) for projection."""
    n, kind = case["n"], case["kind"]
    pixels = sum(w * h for w, h in drt_sizes(case["w"], case["h"], case["views"]))
    col = (1 if case["sh"] < 0 else (case["sh"] + 1) ** 2) * 3 * (2 if case["storage"] else 4)
    gcol = (1 if case["sh"] < 0 else (case["sh"] + 1) ** 2) * 12
    nv, blends = n * case["views"], pixels * (5 if n < 10_000 else 40)
    if kind == "loss":
        return dict(bytes=36 * pixels, flops=1188 * pixels)
    if kind == "knn":
        return dict(bytes=80 * n, flops=8 * 100 * n)
    if kind == "gsr":
        return dict(bytes=(48 + 64 + 16 + (48 if case["grads"] else 0)) * n, flops=16 * (210 if case["grads"] else 45) * n)
    if kind == "levelset":
        return dict(bytes=48 * n + (16 + 32) * pixels, flops=pixels * (8 * 100 + 16 * 12 * case["steps"]))
    if kind == "render":
        return dict(bytes=(48 + col) * n + 44 * pixels, flops=300 * nv + 26 * blends)
    out = 32 if kind != "train" else 12 + 12
    return dict(bytes=(2 * 48 + col + gcol) * n + (out + 32 if kind != "train" else out) * pixels,
                flops=800 * nv + 130 * blends + (1188 * pixels if kind == "train" else 0))


# --------------------------------------------------------------------------- 64-bit values
# Equations of the method (exp(-1/2 Q^(beta/2)) falloff, EWA projection, front-to-back compositing)
# as plain torch operations on float64.
ALPHA_MIN, ALPHA_MAX, T_MIN, LOWPASS, RHO, CLAMP, ZNEAR = 1.0 / 255.0, 0.99, 1e-4, 0.3, 0.1, 1.3, 0.2


def _rotation(q):
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y), 2 * (x * y + w * z),
                        1 - 2 * (x * x + z * z), 2 * (y * z - w * x), 2 * (x * z - w * y), 2 * (y * z + w * x),
                        1 - 2 * (x * x + y * y)], 1).reshape(-1, 3, 3)


def _scales(lsb):
    return (2.0 / (1.0 + torch.exp(-RHO * (lsb[:, 3:] - 2.0)))) * torch.exp(lsb[:, :3])


def _harmonics(deg, d):
    """Real spherical harmonics with the Condon-Shortley phase, l-major, m = -l..l."""
    x, y, z = d.unbind(1)
    pi = math.pi
    out = [torch.full_like(x, math.sqrt(1 / (4 * pi)))]
    if deg >= 1:
        k = math.sqrt(3 / (4 * pi))
        out += [-k * y, k * z, -k * x]
    if deg >= 2:
        a, b = math.sqrt(15 / (4 * pi)), math.sqrt(5 / (16 * pi))
        out += [a * x * y, -a * y * z, b * (3 * z * z - 1), -a * x * z, 0.5 * a * (x * x - y * y)]
    if deg >= 3:
        a, b = math.sqrt(35 / (32 * pi)), math.sqrt(105 / (4 * pi))
        c, e = math.sqrt(21 / (32 * pi)), math.sqrt(7 / (16 * pi))
        out += [-a * y * (3 * x * x - y * y), b * x * y * z, -c * y * (5 * z * z - 1), e * z * (5 * z * z - 3),
                -c * x * (5 * z * z - 1), 0.5 * b * z * (x * x - y * y), -a * x * (x * x - 3 * y * y)]
    return torch.stack(out, 1)


def _project(x, case, cam):
    """Per visible splat, in depth order: screen values [m, 15] (u, v, Sigma' xx xy yy, o, beta, r, g,
    b, z, normal) with their graph back to x, their cut Q and their indices."""
    po, lsb, quat, color = x
    vm = torch.as_tensor(cam.viewmat, dtype=torch.float64, device=DEV)
    f32 = lambda v: float(torch.tensor(v, dtype=torch.float32))
    fx, fy, cx, cy = f32(cam.fx), f32(cam.fy), f32(cam.cx), f32(cam.cy)
    t = po[:, :3] @ vm[:, :3].T + vm[:, 3]
    keep = torch.nonzero((t[:, 2] > ZNEAR) & (po[:, 3] >= ALPHA_MIN)).squeeze(1).detach()
    keep = keep[torch.argsort(t[keep, 2].detach(), stable=True)]
    po, lsb, quat, color, t = po[keep], lsb[keep], quat[keep], color[keep], t[keep]
    R, s = _rotation(quat), _scales(lsb)
    iz = 1.0 / t[:, 2]
    limx, limy = CLAMP * 0.5 * cam.width / fx, CLAMP * 0.5 * cam.height / fy
    rx, ry = (t[:, 0] * iz).clamp(-limx, limx), (t[:, 1] * iz).clamp(-limy, limy)
    zero = torch.zeros_like(iz)
    J = torch.stack([torch.stack([fx * iz, zero, -fx * rx * iz], 1), torch.stack([zero, fy * iz, -fy * ry * iz], 1)], 1)
    U = (J @ vm[:, :3]) @ (R * s[:, None, :])
    S = U @ U.transpose(1, 2) + LOWPASS * torch.eye(2, dtype=torch.float64, device=DEV)
    center = -vm[:, :3].T @ vm[:, 3]
    if case["sh"] >= 0:
        view = po[:, :3] - center
        Y = _harmonics(case["sh"], view / view.norm(dim=1, keepdim=True))
        rgb = (0.5 + (Y[:, :, None] * color).sum(1)).clamp(min=0.0)
    else:
        rgb = color.clone()
    axis = lsb[:, :3].argmin(1)
    nv = R[torch.arange(R.shape[0], device=DEV), :, axis]
    sign = torch.where(((center - po[:, :3].detach()) * nv.detach()).sum(1) < 0, -1.0, 1.0)
    q_cut = (2.0 * torch.log(po[:, 3].detach() / ALPHA_MIN)) ** (2.0 / lsb[:, 3].detach())
    vals = torch.cat([(fx * t[:, 0] * iz + cx)[:, None], (fy * t[:, 1] * iz + cy)[:, None],
                      torch.stack([S[:, 0, 0], S[:, 0, 1], S[:, 1, 1]], 1), po[:, 3:], lsb[:, 3:], rgb, t[:, 2:],
                      nv * sign[:, None]], 1)
    return vals, q_cut


def _block(vals, q_cut, px, py):
    """Colour, depth, alpha and normal [8, pixels] of a block from its splats in depth order."""
    dx, dy = px[None] - vals[:, 0:1], py[None] - vals[:, 1:2]
    A, B, C = vals[:, 2:3], vals[:, 3:4], vals[:, 4:5]
    Q = (C * dx * dx - 2.0 * B * dx * dy + A * dy * dy) / (A * C - B * B)
    Qp = Q.clamp(min=1e-300)
    a = (vals[:, 5:6] * torch.exp(-0.5 * Qp ** (0.5 * vals[:, 6:7]))).clamp(max=ALPHA_MAX)
    a = torch.where((Q <= q_cut[:, None]) & (a >= ALPHA_MIN), a, torch.zeros_like(a))
    T = torch.cumprod(1.0 - a, 0)
    on = (T >= T_MIN).to(a.dtype)
    a = a * on
    before = torch.cat([torch.ones_like(T[:1]), T[:-1]], 0)
    chan = vals[:, 7:14].T @ (a * before)  # r g b z n
    # T after the last blended splat
    last = (T * on + (1.0 - on) * 2.0).min(0).values.clamp(max=1.0)
    return torch.cat([chan[:4], (1.0 - last)[None], chan[4:]], 0)


def _render(x, case, cam, up=None, side=32):
    """The view's channels [8, H, W] (colour, depth, alpha, normal); with `up` (8 upstream images) the
    gradients of the four inputs too."""
    with torch.enable_grad():
        vals, q_cut = _project(x, case, cam)
    flat = vals.detach()
    grad = torch.zeros_like(flat)
    rad_x, rad_y = torch.sqrt(flat[:, 2] * q_cut), torch.sqrt(flat[:, 4] * q_cut)
    out = torch.zeros(8, cam.height, cam.width, dtype=torch.float64, device=DEV)
    for y0 in range(0, cam.height, side):
        y1 = min(y0 + side, cam.height)
        row = torch.nonzero((flat[:, 1] + rad_y > y0) & (flat[:, 1] - rad_y < y1)).squeeze(1)
        u, ru = flat[row, 0], rad_x[row]
        for x0 in range(0, cam.width, side):
            x1 = min(x0 + side, cam.width)
            idx = row[(u + ru > x0) & (u - ru < x1)]
            if idx.numel() == 0:
                continue
            py, px = torch.meshgrid(torch.arange(y0, y1, device=DEV), torch.arange(x0, x1, device=DEV), indexing="ij")
            leaf = flat[idx].requires_grad_(up is not None)
            with torch.set_grad_enabled(up is not None):
                img = _block(leaf, q_cut[idx], px.reshape(-1) + 0.5, py.reshape(-1) + 0.5)
            out[:, y0:y1, x0:x1] = img.detach().reshape(8, y1 - y0, x1 - x0)
            if up is not None:
                grad[idx] += torch.autograd.grad(img, leaf, up[:, y0:y1, x0:x1].reshape(8, -1))[0]
    if up is None:
        return out
    return out, torch.autograd.grad(vals, x, grad, allow_unused=True)


def _ssim_loss(color, target, lam=0.2):
    """Eq. 8 of one view (images [3, H, W]) and its gradient."""
    c = color.detach().requires_grad_(True)
    d = torch.arange(11, dtype=torch.float64, device=DEV) - 5.0
    g = torch.exp(-d * d / (2.0 * 1.5 * 1.5))
    win = torch.outer(g / g.sum(), g / g.sum())[None, None]
    blur = lambda t: F.conv2d(t[:, None], win, padding=5)[:, 0]
    with torch.enable_grad():
        mx, my = blur(c), blur(target)
        sxx, syy, sxy = blur(c * c) - mx * mx, blur(target * target) - my * my, blur(c * target) - mx * my
        ssim = (2 * mx * my + 1e-4) * (2 * sxy + 9e-4) / ((mx * mx + my * my + 1e-4) * (sxx + syy + 9e-4))
        loss = (1 - lam) * (c - target).abs().mean() + lam * (1 - ssim.mean())
    return loss.detach(), torch.autograd.grad(loss, c)[0]


def _nearest(pos):
    """The 16 nearest centres of every centre by brute force (ties to the lower index)."""
    p = pos[:, :3]
    out = []
    for i in range(0, p.shape[0], 1024):
        q = p[i:i + 1024]
        d = (q[:, None, 0] - p[None, :, 0]) ** 2
        d = d + (q[:, None, 1] - p[None, :, 1]) ** 2
        d = d + (q[:, None, 2] - p[None, :, 2]) ** 2
        out.append(torch.topk(d, 16, dim=1, largest=False).indices)
    return torch.cat(out)


def _gsr_sum(x, nbr, splat, z):
    """Sums of Eq. 12's and Eq. 13's terms over some samples, each drawn from its splat."""
    po, lsb, quat = x
    R, s = _rotation(quat), _scales(lsb)
    pt = po[splat, :3] + (R[splat] @ (s[splat] * z)[:, :, None])[:, :, 0]
    nb = nbr[splat]
    delta = pt[:, None] - po[nb, :3]
    loc = (R[nb].transpose(2, 3) @ delta[..., None])[..., 0] / s[nb]
    Q = (loc * loc).sum(-1)
    hb = 0.5 * lsb[nb, 3]
    P = Q ** hb
    best = P.detach().argmin(1)
    d = (po[nb, 3] * torch.exp(-0.5 * P)).sum(1).clamp(1e-30, 1.0)
    pmin = P.detach().min(1, keepdim=True).values
    ct = po[nb, 3] * torch.exp(-0.5 * (P - pmin)) * hb * P / Q
    w = (ct[..., None] * (R[nb] @ (loc / s[nb])[..., None])[..., 0]).sum(1)
    u = w / w.norm(dim=1, keepdim=True)
    ar = torch.arange(pt.shape[0], device=DEV)
    gs = nb[ar, best]
    axis = lsb[gs, :3].detach().argmin(1)
    nv, smin = R[gs][ar, :, axis], s[gs][ar, axis]
    e = (delta[ar, best] * nv).sum(1)
    sg = torch.where(e.detach() < 0, -1.0, 1.0)
    fbar = smin * (sg * e / smin) ** (0.5 * lsb[gs, 3])
    pl = -2.0 * torch.log(d)
    f = torch.where(pl > 0, smin * torch.sqrt(pl.clamp(min=1e-300)), torch.zeros_like(pl))
    return (fbar - f).abs().sum(), ((u - sg[:, None] * nv) ** 2).sum()


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    if kind == "loss":
        st = prepare(case, seed)
        losses, grads, b = [], [], 0
        for w, h in st["sizes"]:
            k = 3 * w * h
            c, t = (st[q][b:b + k].double().reshape(3, h, w) for q in ("color", "target"))
            l, g = _ssim_loss(c, t)
            losses.append(l)
            grads.append(g.reshape(-1))
            b += k
        return dict(loss=torch.stack(losses), g=torch.cat(grads))
    if kind == "gsr":
        if n > 100_000 or n < 16:  # neighbour lists by brute force: too slow beyond
            return None
        raw = _scene(case, seed)
        nbr = _nearest(raw[0])
        splat, z = _samples(case, seed)
        splat, z = splat.long(), z.double()
        x = [t.double().requires_grad_(case["grads"]) for t in raw[:3]]
        sdf, nor, grads = 0.0, 0.0, [torch.zeros_like(t) for t in x]
        for i in range(0, n, 25_000):
            with torch.set_grad_enabled(case["grads"]):
                a, b = _gsr_sum(x, nbr, splat[i:i + 25_000], z[i:i + 25_000])
            if case["grads"]:
                for acc, g in zip(grads, torch.autograd.grad((a + b) / n, x)):
                    acc += torch.nan_to_num(g)
            sdf, nor = sdf + a.detach() / n, nor + b.detach() / n
        r = dict(losses=torch.stack([sdf, nor, sdf + nor]))
        return r | dict(zip(("g_pos_op", "g_lscale_beta", "g_quat"), grads)) if case["grads"] else r
    # several views of large scenes take too long; the lists are whole numbers, and a level-set point
    # is found from them
    if kind in ("knn", "levelset") or n * case["views"] > 1_600_000 or (case["scene"] == "uniform" and case["w"] > 1000):
        return None
    cams = _cameras(case, seed)
    x = [t.double().requires_grad_(kind != "render") for t in _scene(case, seed)]
    pix = [c.width * c.height for c in cams]
    base = [sum(pix[:k]) for k in range(len(pix))]
    up_all = _upstream(case, seed, sum(pix)) if kind in ("step", "autograd") else None
    target = _images(case, seed, [(c.width, c.height) for c in cams], 6) if kind == "train" else None
    imgs, losses, grads = [], [], [torch.zeros_like(t) for t in x]
    for v, cam in enumerate(cams):
        h, w, b, k = cam.height, cam.width, base[v], pix[v]
        if kind == "render":
            imgs.append(_render(x, case, cam))
            continue
        if kind == "train":
            img = _render([t.detach() for t in x], case, cam)
            l, g = _ssim_loss(img[:3], target[3 * b:3 * b + 3 * k].double().reshape(3, h, w))
            losses.append(l)
            up = torch.cat([g, torch.zeros(5, h, w, dtype=torch.float64, device=DEV)])
        else:
            gc, gd, ga, gn = (t.double() for t in up_all)
            up = torch.cat([gc[3 * b:3 * b + 3 * k].reshape(3, h, w), gd[b:b + k].reshape(1, h, w),
                            ga[b:b + k].reshape(1, h, w), gn[3 * b:3 * b + 3 * k].reshape(3, h, w)])
        img, gx = _render(x, case, cam, up)
        imgs.append(img)
        for acc, g in zip(grads, gx):
            if g is not None:
                acc += g
    part = lambda a, b: torch.cat([i[a:b].reshape(-1) for i in imgs])
    color, depth, alpha, normal = part(0, 3), part(3, 4), part(4, 5), part(5, 8)
    named = dict(zip(("g_pos_op", "g_lscale_beta", "g_quat", "g_color"), grads))
    if kind == "render":
        return dict(color=color, depth=depth, alpha=alpha, normal=normal, t_final=1.0 - alpha, last=None, n_contrib=None)
    if kind == "autograd":
        return dict(out=[color, depth, alpha, normal], grads=grads)
    if kind == "train":
        return dict(loss=torch.stack(losses), color=color, grads=named)
    return dict(out=dict(color=color, depth=depth, alpha=alpha, normal=normal), grads=named)
