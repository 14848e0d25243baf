"""The work a fitting or viewing program has this framework do, as measurable cases.

A program that fits PackUV atlases runs one L1 (or L1 + D-SSIM) step per
iteration over every camera of its rig, refreshes its low-precision proxy
and its dynamic mask now and then, prunes its UV cells after a densification
step, and renders single views to look at.  ``listed()`` holds these calls at
the sizes of the repository's own configurations (a 64^2 atlas with one
256^2 view up to the 208-view sequence), together with one odd-sized step;
``draw()`` spreads the sizes over the whole range between them.

Every input is made on the GPU from the seed alone, with the distributions
of the synthetic scenes: eight anisotropic clusters of means laid into the
live texels in the order of their spherical UV cells, log-scales N(-4, 0.5),
random quaternions, opacity logits N(0, 1), SH DC N(0, 0.5) and N(0, 0.1)
above, cameras on rings of radius 4 that look inward, U[0, 1] targets.
"""

import math
import types

import numpy as np
import torch

import paper_2602_23040_gb300 as pk

F64 = torch.float64


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------

def _case(name, kind, side, occupancy, sh, views, sizes, **more):
    c = {"kind": kind, "atlas_w": side, "atlas_h": side, "levels": 1, "occupancy": occupancy, "sh": sh, "frames": 1,
         "dynamic": 0.0, "views": views, "sizes": sizes}
    if name:
        c = {"name": name, **c}
    c.update(more)
    return c


def listed():
    rig = "1920x1080,1280x720"   # the mixed resolutions of a 360-degree capture
    return [
        # one step of a small atlas seen by one small camera: launches and latency count
        _case("step_64sq_1view", "step", 64, 1.0, 0, 1, "256x256"),
        # one iteration with the full photometric objective on odd sizes everywhere (atlas, views, SH degree 2)
        _case("photo_step_ragged_3view", "photo_step", 301, 0.57, 2, 3, "641x479,333x517,97x403", atlas_h=203),
        # a viewer's frame: forward only, one 1080p camera, SH degree 3
        _case("render_1080p", "forward", 512, 0.6, 3, 1, "1920x1080"),
        # one fitting iteration over the whole 52-camera rig
        _case("step_rig_52view", "step", 1024, 0.6, 3, 52, rig),
        # the differentiable render of a three-level FP16 atlas by 16 cameras of uneven sizes, and its backward
        _case("autograd_fp16_3level_16view", "autograd", 1024, 0.6, 3, 16, "640x480,1920x1080,960x540,1280x720,1600x900",
              levels=3),
        # the largest: four frames x 52 cameras in one launch, gradients only to the 30 % dynamic texels
        _case("step_sequence_4x52view", "step", 1024, 0.6, 3, 52, rig, frames=4, dynamic=0.3),
        # atlas -> attributes -> projected records of every camera (gather, projection and colour)
        _case("gather_project_rig", "front", 1024, 0.6, 3, 52, rig),
        # 2D gradients of every camera -> texel gradients, frozen texels kept at zero
        _case("scatter_grad_rig", "scatter", 1024, 0.6, 3, 52, rig, dynamic=0.3),
        # the L1 + D-SSIM objective and its gradient on the rig's images
        _case("photo_loss_rig", "photo_loss", 64, 1.0, 0, 52, rig),
        # a proxy refresh: channel ranges, 8-bit code planes, and the attributes read back from them
        _case("lpo_refresh_1024sq", "lpo", 1024, 0.6, 3, 1, "1280x720"),
        # motion masks of the rig's flow fields, and the dynamic mask of the Gaussians they touch
        _case("dynamic_mask_rig", "masks", 1024, 0.6, 0, 52, rig),
        # UV cells and Max-K pruning of the live set of a 1024^2 map
        _case("uv_max_k_1024sq", "uv", 1024, 0.6, 0, 1, "256x256", max_k=4),
    ]


def draw(rng):
    def logu(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def sizes(lo, hi, k):
        out = []
        for _ in range(k):
            w = logu(lo, hi)
            out.append("%dx%d" % (w, max(16, int(w * rng.choice((0.5625, 0.75, 0.62, 1.0))))))
        return ",".join(out)

    kind = rng.choice(("step", "step", "forward", "autograd", "photo_step", "front", "scatter", "photo_loss", "lpo",
                       "masks", "uv"))
    side = logu(64, 1024)
    occ = round(rng.uniform(0.4, 1.0 if side < 512 else 0.8), 3)
    sh = rng.choice((0, 1, 2, 3, 3, 3))
    more = {"atlas_h": max(32, int(side * rng.uniform(0.6, 1.0)))}
    if kind in ("step", "photo_step", "autograd"):
        views, hi = logu(1, 52), 1920
        if kind == "autograd" and rng.random() < 0.5 and side >= 64:
            more = {"levels": 3}
        if kind == "step" and rng.random() < 0.4:
            more["frames"], more["dynamic"] = rng.choice((2, 3, 4)), round(rng.uniform(0.1, 0.6), 2)
            views, hi = logu(1, 26), 1280
        return _case("", kind, side, occ, sh, views, sizes(160, hi, rng.choice((1, 2, 3))), **more)
    if kind == "forward":
        return _case("", kind, side, occ, sh, 1, sizes(256, 2560, 1), **more)
    if kind == "photo_loss":
        return _case("", kind, 64, 1.0, 0, logu(1, 52), sizes(160, 1920, 2))
    if kind in ("front", "scatter"):
        if kind == "scatter":
            more["dynamic"] = rng.choice((0.0, 0.3))
        return _case("", kind, side, occ, sh, logu(1, 52), "1280x720", **more)
    if kind == "lpo":
        more["frames"] = rng.choice((1, 1, 2, 4))
        return _case("", kind, side, occ, sh, 1, "640x480", **more)
    if kind == "masks":
        return _case("", kind, side, occ, 0, logu(1, 52), sizes(320, 1920, 2), **more)
    return _case("", "uv", logu(64, 1400), occ, 0, 1, "256x256", max_k=rng.choice((1, 2, 4, 8)))


# ---------------------------------------------------------------------------
# Scenes
# ---------------------------------------------------------------------------

def _levels(case):
    """(w, h, x0, y0, rotated) of each level, and the atlas size."""
    if case["levels"] == 1:
        return [(case["atlas_w"], case["atlas_h"], 0, 0, 0)], (case["atlas_w"], case["atlas_h"])
    s = case["atlas_w"]
    half, quarter = s // 2, s // 4
    return [(s, s, half, 0, 0), (half, half, 0, 0, 0), (quarter, quarter, 0, half, 0)], (s + half, s)


def _n_live(case):
    return sum(int(math.floor(case["occupancy"] * w * h + 1e-9)) for w, h, *_ in _levels(case)[0])


def _channels(case):
    return 11 + 3 * (case["sh"] + 1) ** 2


def _views(case):
    """Cameras on three rings (heights -1, 0, 1) of radius 4, looking at the
    origin, their sizes taken in turn; every frame sees the same rig."""
    sizes = [tuple(int(x) for x in s.split("x")) for s in case["sizes"].split(",")]
    n = case["views"]
    ring = []
    per = [n // 3 + (1 if k < n % 3 else 0) for k in range(3)] if n >= 3 else [0, n, 0]
    for count, height in zip(per, (-1.0, 0.0, 1.0)):
        for k in range(count):
            phi = 2.0 * math.pi * (k + 0.5 * (height != 0.0) + 0.137) / count
            ring.append((4.0 * math.cos(phi), height, 4.0 * math.sin(phi)))
    views = []
    for f in range(case["frames"]):
        for i, eye in enumerate(ring):
            w, h = sizes[i % len(sizes)]
            eye64 = np.asarray(eye, np.float64)
            fwd = -eye64 / np.linalg.norm(eye64)
            right = np.cross(fwd, (0.0, 1.0, 0.0))
            right /= np.linalg.norm(right)
            R = np.stack([right, np.cross(fwd, right), fwd])
            fx = float(np.float32(w / 2.0 / math.tan(math.radians(30.0))))
            views.append(types.SimpleNamespace(
                R=R.astype(np.float32).astype(np.float64), t=(-R @ eye64).astype(np.float32).astype(np.float64), fx=fx,
                fy=fx, cx=w / 2.0, cy=h / 2.0, width=w, height=h, frame=f))
    return views


def _pack_bits(mask):
    """Bool [H][W] -> int32 [H][ceil(W / 32)], texel x in bit x & 31."""
    h, w = mask.shape
    wp = (w + 31) // 32
    m = torch.zeros((h, wp * 32), dtype=torch.int64, device=mask.device)
    m[:, :w] = mask
    words = (m.view(h, wp, 32) << torch.arange(32, device=mask.device)).sum(-1)
    return torch.where(words >= 1 << 31, words - (1 << 32), words).to(torch.int32).contiguous()


def _means(n, seed, gen):
    rng = np.random.default_rng(seed)
    out = torch.empty((n, 3), dtype=F64, device="cuda")
    label = torch.randint(0, 8, (n,), generator=gen, device="cuda")
    z = torch.randn((n, 3), generator=gen, device="cuda", dtype=F64)
    for c in range(8):
        centre, sig = rng.uniform(-0.8, 0.8, 3), rng.uniform(0.05, 0.3, 3)
        q, _ = np.linalg.qr(rng.standard_normal((3, 3)))
        sel = label == c
        out[sel] = z[sel] @ torch.from_numpy(sig[:, None] * q.T).cuda() + torch.from_numpy(centre).cuda()
    return out


def _scene(case, seed):
    """atlas [F][D][H][W] float32, occupancy and dynamic bit rows, live texel ids."""
    levels, (W, H) = _levels(case)
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    occ = torch.zeros((H, W), dtype=torch.bool, device="cuda")
    for w, h, x0, y0, _ in levels:
        m = torch.zeros(w * h, dtype=torch.bool, device="cuda")
        m[torch.randperm(w * h, generator=gen, device="cuda")[: int(math.floor(case["occupancy"] * w * h + 1e-9))]] = True
        occ[y0:y0 + h, x0:x0 + w] = m.view(h, w)
    live = occ.view(-1).nonzero().view(-1)
    n, D, F = live.numel(), _channels(case), case["frames"]
    mu = _means(n, int(seed), gen)
    w0, h0 = levels[0][:2]
    theta, phi = torch.atan2(mu[:, 1], mu[:, 0]), torch.acos((mu[:, 2] / mu.norm(dim=1)).clamp(-1, 1))
    u = ((math.pi + theta) / (2 * math.pi) * w0).floor().clamp(max=w0 - 1).long()
    v = (phi / math.pi * h0).floor().clamp(max=h0 - 1).long()
    mu = mu[torch.argsort(v * w0 + u, stable=True)]

    def normal(*shape):
        return torch.randn(shape, generator=gen, device="cuda")

    attr = torch.empty((D, n), device="cuda")
    attr[3:6] = -4.0 + 0.5 * normal(3, n)
    q = normal(4, n)
    attr[6:10] = q / q.norm(dim=0)
    attr[10] = normal(n)
    attr[11:14] = 0.5 * normal(3, n)
    if D > 14:
        attr[14:] = 0.1 * normal(D - 14, n)
    dyn = None
    moving = torch.ones(n, dtype=torch.bool, device="cuda")
    rng = np.random.default_rng(int(seed) + 1)
    if case["dynamic"] > 0:
        actor = torch.from_numpy(rng.uniform(-0.5, 0.5, 3)).cuda()
        moving = torch.zeros(n, dtype=torch.bool, device="cuda")
        moving[torch.argsort((mu - actor).norm(dim=1))[: int(round(case["dynamic"] * n))]] = True
        dm = torch.zeros(H * W, dtype=torch.bool, device="cuda")
        dm[live[moving]] = True
        dyn = _pack_bits(dm.view(H, W))
    a = rng.standard_normal((4, 3))
    a = torch.from_numpy(a / np.linalg.norm(a, axis=1).sum()).cuda()
    freq, rate, ph = rng.normal(0.0, 2.0, (3, 4)), rng.uniform(0.05, 0.2, 4), rng.uniform(0, 2 * math.pi, 4)
    atlas = torch.zeros((F, D, H * W), device="cuda")
    for f in range(F):
        at = mu + 0.0
        if case["dynamic"] > 0:   # per-frame displacement of the dynamic means by a smooth flow of amplitude 0.05
            arg = mu @ torch.from_numpy(freq).cuda() + torch.from_numpy(rate * f + ph).cuda()
            at = torch.where(moving[:, None], mu + 0.05 * torch.sin(arg) @ a, mu)
        attr[0:3] = at.T.float()
        atlas[f][:, live] = attr
    return atlas.view(F, D, H, W), _pack_bits(occ), dyn, live


def _plan(case, texel="f32"):
    levels, wh = _levels(case)
    views, n = _views(case), _n_live(case)
    return pk.Plan(levels, wh, case["sh"], case["frames"], texel, views, n, max_dups=8 * n * len(views) + 65536)


def _uniform(n, seed):
    return torch.rand(n, generator=torch.Generator(device="cuda").manual_seed(int(seed) + 7), device="cuda")


def _flow(views, seed):
    """Optical flow [2 P]: a moving sphere's silhouette in every camera (magnitude up to 4 px) over N(0, 0.2) noise."""
    rng = np.random.default_rng(int(seed) + 3)
    centre, radius = rng.uniform(-0.5, 0.5, 3), 0.25
    gen = torch.Generator(device="cuda").manual_seed(int(seed) + 3)
    out = torch.empty(2 * sum(v.width * v.height for v in views), device="cuda").normal_(0.0, 0.2, generator=gen)
    at = 0
    for v in views:
        W, H = v.width, v.height
        R = torch.from_numpy(v.R).cuda().float()
        to = torch.from_numpy(centre + v.R.T @ v.t).cuda().float()   # eye = -R^T t
        xs = (torch.arange(W, device="cuda") + 0.5 - v.cx) / v.fx
        ys = (torch.arange(H, device="cuda") + 0.5 - v.cy) / v.fy
        d = torch.stack([xs.expand(H, W), ys[:, None].expand(H, W), torch.ones((H, W), device="cuda")], -1) @ R
        along = (d @ to) / d.norm(dim=-1)
        dist2 = (to @ to) - along * along
        mag = 4.0 * torch.sqrt((1.0 - dist2 / (radius * radius)).clamp(0.0, 1.0)) * (along > 0)
        ang = rng.uniform(0.0, 2.0 * math.pi)
        out[at:at + H * W] += (mag * math.cos(ang)).view(-1)
        out[at + H * W:at + 2 * H * W] += (mag * math.sin(ang)).view(-1)
        at += 2 * H * W
    return out


# ---------------------------------------------------------------------------
# What a program holds before the call, and the call
# ---------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    s = types.SimpleNamespace(kind=kind)
    if kind == "uv":
        atlas, _, _, live = _scene(case, seed)
        s.soa = atlas[0].view(14, -1)[:, live].contiguous()
        s.n, s.M, s.N, s.K = live.numel(), case["atlas_w"], case["atlas_h"], case["max_k"]
        s.cell, s.rank = (torch.empty(s.n, dtype=torch.int32, device="cuda") for _ in range(2))
        s.keep = torch.empty(s.n, dtype=torch.uint8, device="cuda")
        s.count = torch.empty(s.M * s.N, dtype=torch.int32, device="cuda")
        s.scratch = pk.uv_max_k(s.soa, s.n, s.M, s.N, s.K, s.cell, s.rank, s.keep, s.count)
        return s
    if kind == "photo_loss":
        s.plan = _plan(case)
        s.ws = pk.make_workspace(s.plan)
        pk.workspace_init(s.plan, s.ws)
        s.target = _uniform(3 * s.plan.P, seed)
        # a render part of the way to its target
        s.image = 0.7 * s.target + 0.3 * _uniform(3 * s.plan.P, seed + 1000)
        s.dimage = torch.empty_like(s.image)
        pk.photo_loss_grad(s.plan, s.image, s.target, s.dimage, s.ws, 0.2)
        return s
    s.atlas, s.occ, s.dyn, _ = _scene(case, seed)
    if kind in ("step", "photo_step", "forward", "autograd"):
        s.src = s.atlas.half() if kind == "autograd" else s.atlas
        s.r = pk.Renderer(_plan(case, "f16" if kind == "autograd" else "f32"))
        s.r.ensure_capacity(s.src, s.occ, s.dyn)
        if kind == "autograd":
            s.master = s.atlas.requires_grad_(True)
            s.dimage = (_uniform(3 * s.r.plan.P, seed) - 0.5) / (3 * s.r.plan.P)
        elif kind != "forward":
            s.target = _uniform(3 * s.r.plan.P, seed)
            s.grad = torch.zeros_like(s.atlas)
        if kind == "photo_step":
            s.r.photo_step(s.atlas, s.occ, s.dyn, s.target, s.grad)
        return s
    s.plan = p = _plan(case)
    s.ws = pk.make_workspace(p)
    pk.workspace_init(p, s.ws)
    s.soa = torch.empty(p.D * p.G, device="cuda")
    s.texel = torch.empty(p.N, dtype=torch.int32, device="cuda")
    s.dynflag = torch.empty(p.N, dtype=torch.uint8, device="cuda")
    if kind == "lpo":
        s.lohi = torch.empty(2 * p.D, device="cuda")
        levels, (W, H) = _levels(case)
        s.codes = torch.empty(case["frames"] * (p.D + 3) * H * W, dtype=torch.uint8, device="cuda")
        return s
    pk.atlas_gather(p, s.atlas, s.occ, s.dyn, s.soa, s.texel, s.dynflag, s.ws)
    s.records = torch.empty(12 * p.pairs, device="cuda")
    if kind in ("masks", "scatter"):
        pk.project_and_sh(p, s.soa, s.records, s.ws)
    if kind == "masks":
        s.flow = _flow(p.views, seed)
        s.bits = torch.empty(p.mask_words, dtype=torch.int32, device="cuda")
        s.dynbits = torch.empty(s.occ.numel(), dtype=torch.int32, device="cuda")
    elif kind == "scatter":
        # 2D gradients of the pairs a backward reaches: three in four of the visible ones
        gen = torch.Generator(device="cuda").manual_seed(int(seed) + 5)
        s.g2d = torch.randn((p.pairs, 12), generator=gen, device="cuda")
        s.g2d *= 1e-7 * (torch.rand(p.pairs, 1, generator=gen, device="cuda") < 0.75)
        s.g2d *= s.records.view(-1, 12)[:, 7:8] > 0
        s.g2d[:, 9:] = 0.0
        s.g2d = s.g2d.view(-1)
        s.records = None
        s.grad = torch.zeros_like(s.atlas)
    return s


def run(s):
    k = s.kind
    if k == "step":
        s.r.l1_step(s.atlas, s.occ, s.dyn, s.target, s.grad)
        return [s.r.image, s.grad]
    if k == "photo_step":
        s.r.photo_step(s.atlas, s.occ, s.dyn, s.target, s.grad)
        return [s.r.image, s.grad]
    if k == "forward":
        return [s.r.forward(s.atlas, s.occ)]
    if k == "autograd":
        image = pk.render(s.master, s.r, s.occ, proxy=s.src)
        (grad,) = torch.autograd.grad(image, s.master, s.dimage)
        return [image.detach(), grad]
    if k == "front":
        pk.atlas_gather(s.plan, s.atlas, s.occ, s.dyn, s.soa, s.texel, s.dynflag, s.ws)
        pk.project_and_sh(s.plan, s.soa, s.records, s.ws)
        return [s.soa, s.texel, s.records]
    if k == "scatter":
        pk.atlas_scatter_grad(s.plan, s.soa, s.g2d, None if s.dyn is None else s.dynflag, s.texel, s.grad, False, s.ws)
        return [s.grad]
    if k == "photo_loss":
        pk.photo_loss_grad(s.plan, s.image, s.target, s.dimage, s.ws, 0.2)
        return [s.dimage]
    if k == "lpo":
        pk.lpo_minmax(s.plan, s.atlas, s.occ, s.lohi, s.ws)
        pk.lpo_encode(s.plan, s.atlas, s.occ, s.lohi, s.codes, s.ws)
        pk.atlas_gather_lpo(s.plan, s.codes, 0, s.lohi, s.occ, s.dyn, s.soa, s.texel, s.dynflag, s.ws)
        return [s.lohi, s.codes, s.soa, s.texel]
    if k == "masks":
        pk.motion_mask(s.plan, s.flow, 1.0, 2, s.bits, s.ws)
        pk.dynamic_mask(s.plan, s.records, s.texel, s.bits, s.dynbits, s.ws)
        return [s.bits, s.dynbits]
    pk.uv_max_k(s.soa, s.n, s.M, s.N, s.K, s.cell, s.rank, s.keep, s.count, scratch=s.scratch)
    return [s.cell, s.rank, s.keep, s.count]


# ---------------------------------------------------------------------------
# The work of one pass
# ---------------------------------------------------------------------------

def work(case):
    """Inputs read once and outputs written once; operations of the method
    itself (a lit pixel composites about 40 splats before its transmittance
    is spent: 13 operations each forward and 26 backward)."""
    levels, (W, H) = _levels(case)
    views = _views(case)
    n, D, F, nb = _n_live(case), _channels(case), case["frames"], (case["sh"] + 1) ** 2
    P = sum(v.width * v.height for v in views)
    pairs = n * len(views)
    words = H * ((W + 31) // 32)
    k = case["kind"]
    if k == "uv":
        return {"bytes": n * 25 + 4 * case["atlas_w"] * case["atlas_h"], "flops": 60 * n}
    if k == "photo_loss":
        return {"bytes": 36 * P, "flops": 3 * P * 2 * (5 * 22 + 3 * 22)}
    if k == "lpo":
        return {"bytes": F * D * n * 8 + F * (D + 3) * W * H + 4 * words, "flops": 6 * F * D * n}
    if k == "masks":
        return {"bytes": 8 * P + P // 8 + 36 * pairs // 2 + 8 * words, "flops": 6 * P + 30 * pairs}
    project = pairs * (150 + 6 * nb)
    if k == "front":
        return {"bytes": F * D * n * 8 + 5 * n + 48 * pairs, "flops": project}
    if k == "scatter":
        return {"bytes": F * D * n * 8 + 36 * pairs, "flops": 3 * project}
    texel = 2 if k == "autograd" else 4
    forward = {"bytes": F * D * n * texel + 4 * words + 12 * P, "flops": project + 40 * 13 * P}
    if k == "forward":
        return forward
    return {"bytes": forward["bytes"] + 12 * P + F * D * n * 4,
            "flops": forward["flops"] + 3 * project + 40 * 26 * P + (3 * P * 400 if k == "photo_step" else 0)}


# ---------------------------------------------------------------------------
# 64-bit values of the same outputs, by plain torch
# ---------------------------------------------------------------------------

def _sh64(d, nb):
    x, y, z = d
    xx, yy, zz = x * x, y * y, z * z
    pi = math.pi
    Y = [torch.full_like(x, 0.5 / math.sqrt(pi))]
    if nb > 1:
        c = math.sqrt(3 / (4 * pi))
        Y += [-c * y, c * z, -c * x]
    if nb > 4:
        a, b, e = math.sqrt(15 / pi) / 2, math.sqrt(5 / pi) / 4, math.sqrt(15 / pi) / 4
        Y += [a * x * y, -a * y * z, b * (2 * zz - xx - yy), -a * x * z, e * (xx - yy)]
    if nb > 9:
        a, b, c = math.sqrt(35 / (32 * pi)), math.sqrt(105 / pi) / 2, math.sqrt(42 / pi) / 8
        e, f = math.sqrt(7 / pi) / 4, math.sqrt(105 / pi) / 4
        Y += [-a * y * (3 * xx - yy), b * x * y * z, -c * y * (4 * zz - xx - yy), e * z * (2 * zz - 3 * xx - 3 * yy),
              -c * x * (4 * zz - xx - yy), f * z * (xx - yy), -a * x * (xx - 3 * yy)]
    return Y


def _project64(attr, v, nb):
    """Record fields [11][n] (m, conic, opacity, z, radius, rgb) of one view, and which pairs it keeps."""
    mu, ls, q, logit = attr[0:3], attr[3:6], attr[6:10], attr[10]
    w, x, y, z = q / q.norm(dim=0)
    R = [[1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)],
         [2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)],
         [2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]]
    s2 = torch.exp(2 * ls)
    S = [[sum(R[i][k] * R[j][k] * s2[k] for k in range(3)) for j in range(3)] for i in range(3)]
    Wc = v.R
    X = [sum(Wc[i, k] * mu[k] for k in range(3)) + v.t[i] for i in range(3)]
    front = X[2] > 0.01
    iz = 1.0 / torch.where(front, X[2], torch.ones_like(X[2]))
    t0 = [v.fx * iz * Wc[0, k] - v.fx * X[0] * iz * iz * Wc[2, k] for k in range(3)]
    t1 = [v.fy * iz * Wc[1, k] - v.fy * X[1] * iz * iz * Wc[2, k] for k in range(3)]

    def form(a, b):
        return sum(a[i] * S[i][j] * b[j] for i in range(3) for j in range(3))

    A, B, C = form(t0, t0) + 0.3, form(t0, t1), form(t1, t1) + 0.3
    det = A * C - B * B
    keep = front & (det > 1e-7)
    eye = -(v.R.T @ v.t)
    d = torch.stack([mu[k] - eye[k] for k in range(3)])
    Y = _sh64(list(d / d.norm(dim=0)), nb)
    sh = attr[11:].view(nb, 3, -1)
    rgb = [(sum(sh[j, c] * Y[j] for j in range(nb)) + 0.5).clamp(min=0) for c in range(3)]
    with torch.no_grad():
        tr = A + C
        radius = torch.ceil(3 * torch.sqrt(0.5 * (tr + torch.sqrt((tr * tr - 4 * det).clamp(min=0)))))
    rec = [v.fx * X[0] * iz + v.cx, v.fy * X[1] * iz + v.cy, C / det, -B / det, A / det, torch.sigmoid(logit), X[2],
           radius, *rgb]
    return torch.stack(rec), keep


def _exact_front(case, seed):
    atlas, _, _, live = _scene(case, seed)
    nb, n = (case["sh"] + 1) ** 2, live.numel()
    attr = atlas[0].view(atlas.shape[1], -1)[:, live].double()
    views = _views(case)
    out = torch.zeros((len(views), n, 12), dtype=F64, device="cuda")
    for i, v in enumerate(views):
        rec, keep = _project64(attr, v, nb)
        out[i, :, :11] = (rec * keep).T
    return [attr.reshape(-1), None, out.view(-1)]


def _exact_scatter(case, seed):
    s = prepare(case, seed)
    p = s.plan
    nb = (case["sh"] + 1) ** 2
    attr = s.soa.view(p.D, p.N).double()
    g2d = s.g2d.view(p.V, p.N, 12)
    total = torch.zeros_like(attr)
    for i, v in enumerate(p.views):
        leaf = attr.clone().requires_grad_(True)
        rec, keep = _project64(leaf, v, nb)
        g = g2d[i].double().T * keep
        (d,) = torch.autograd.grad(rec[[0, 1, 2, 3, 4, 5, 8, 9, 10]], leaf, g[:9])
        total += d
    if s.dyn is not None:
        total *= s.dynflag.double()
    out = torch.zeros(s.grad.shape, dtype=F64, device="cuda").view(p.D, -1)
    out[:, s.texel.long()] = total
    return [out.view(s.grad.shape)]


def _exact_step(case, seed):
    """One small view: every pixel against every splat in depth order, and autograd."""
    s = prepare(case, seed)
    p, v = s.r.plan, s.r.plan.views[0]
    nb = (case["sh"] + 1) ** 2
    live = s.r.texel.long()
    attr = s.atlas[0].view(p.D, -1)[:, live].double().requires_grad_(True)
    rec, keep = _project64(attr, v, nb)
    order = torch.argsort(rec[6].detach())
    order = order[keep[order]]
    leaf = rec.detach()[:, order].clone().requires_grad_(True)
    W, H = v.width, v.height
    image = torch.zeros((3, H * W), dtype=F64, device="cuda")
    target = s.target.double().view(3, -1)
    step = max(1, (1 << 25) // max(1, order.numel()))
    for a in range(0, H * W, step):
        pix = torch.arange(a, min(H * W, a + step), device="cuda")
        dx, dy = (pix % W + 0.5) - leaf[0][:, None], (pix // W + 0.5) - leaf[1][:, None]
        q = leaf[2][:, None] * dx * dx + 2 * leaf[3][:, None] * dx * dy + leaf[4][:, None] * dy * dy
        alpha = (leaf[5][:, None] * torch.exp(-0.5 * q)).clamp(max=0.99)
        alpha = alpha * ((q <= 9) & (alpha >= 1 / 255)).detach()
        T = torch.cumprod(1 - alpha, 0)
        before = torch.cat([torch.ones_like(T[:1]), T[:-1]])
        wt = before * alpha * (T >= 1e-4).detach()
        img = leaf[8:11] @ wt
        (img - target[:, pix]).abs().sum().div(3 * H * W).backward()
        image[:, pix] = img.detach()
    full = torch.zeros_like(rec)
    full[:, order] = leaf.grad
    (d,) = torch.autograd.grad(rec, attr, full)
    grad = torch.zeros(s.grad.shape, dtype=F64, device="cuda").view(p.D, -1)
    grad[:, live] = d
    return [image.view(-1), grad.view(s.grad.shape)]


def _blur64(x, w):
    for dim in (-1, -2):
        pad = torch.nn.functional.pad(x, (5, 5, 0, 0) if dim == -1 else (0, 0, 5, 5))
        n = x.shape[dim]
        x = sum(w[k] * pad.narrow(dim, k, n) for k in range(11))
    return x


def _exact_photo_loss(case, seed):
    s = prepare(case, seed)
    P = s.plan.P
    w = [math.exp(-(k * k) / 4.5) for k in range(-5, 6)]
    w = [x / sum(w) for x in w]
    out = torch.empty(3 * P, dtype=F64, device="cuda")
    at = 0
    for v in s.plan.views:
        m = 3 * v.width * v.height
        x = s.image[at:at + m].double().view(3, v.height, v.width).requires_grad_(True)
        y = s.target[at:at + m].double().view(3, v.height, v.width)
        m1, m2 = _blur64(x, w), _blur64(y, w)
        e11, e22, e12 = _blur64(x * x, w), _blur64(y * y, w), _blur64(x * y, w)
        ssim = (2 * m1 * m2 + 1e-4) * (2 * (e12 - m1 * m2) + 9e-4) / (
            (m1 * m1 + m2 * m2 + 1e-4) * ((e11 - m1 * m1) + (e22 - m2 * m2) + 9e-4))
        loss = (0.8 * (x - y).abs().sum() - 0.2 * ssim.sum()) / (3 * P)
        out[at:at + m] = torch.autograd.grad(loss, x)[0].view(-1)
        at += m
    return [out]


def _exact_lpo(case, seed):
    atlas, _, _, live = _scene(case, seed)
    F, D = atlas.shape[:2]
    x = atlas.view(F, D, -1)[:, :, live].double()
    lo, hi = x.amin(dim=(0, 2)), x.amax(dim=(0, 2))
    most = torch.tensor([65535.0] * 3 + [255.0] * (D - 3), dtype=F64, device="cuda")
    delta = ((hi - lo) / most)[None, :, None]
    code = ((x - lo[None, :, None]) / delta + 0.5).floor().clamp(min=0)
    code = torch.minimum(code, most[None, :, None])
    return [torch.stack([lo, hi], 1).view(-1), None, (lo[None, :, None] + code * delta).transpose(0, 1).reshape(-1),
            None]


def exact(case, seed):
    kind = case["kind"]
    if kind == "front" and case["frames"] == 1:
        return _exact_front(case, seed)
    if kind == "scatter" and case["frames"] == 1:
        return _exact_scatter(case, seed)
    if kind == "photo_loss":
        return _exact_photo_loss(case, seed)
    if kind == "lpo":
        return _exact_lpo(case, seed)
    if kind == "step" and case["frames"] == 1 and case["views"] == 1 and case["dynamic"] == 0:
        pixels = sum(v.width * v.height for v in _views(case))
        if _n_live(case) * pixels <= 1 << 29:   # beyond that every-pixel-by-every-splat takes too long
            return _exact_step(case, seed)
    return None   # tile lists and masks are whole numbers; the large images have no quick 64-bit value
