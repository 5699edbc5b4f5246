"""The renders and training steps this package is used for, as measurable cases.

Scenes follow the workload recipe of the tests and the benchmark (surfels on
spheres and squares, Gaussians scattered around them), made on the GPU from a
seed.  ``exact`` restates the render in plain float64 tensor code: it expands
every (primitive, pixel) pair of a conservative footprint, with no tiles, no
culling and none of this package's code.
"""
import math

import torch

from paper_2504_17545_gb300 import render as R

DTYPES = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
ATTRS = ("s_rot", "s_scale", "g_rot", "g_scale", "g_opac")
R2 = 2.0 * math.log(255.0)          # opaque disc radius squared
ALPHA_MIN = 1.0 / 255.0
ZNEAR = 0.01


def _case(name, kind, width, height, surfels, gaussians, dtype="f32", degree=3, dim=3, samples=1, mip=False,
          aux=True, views=1, front=False):
    c = dict(kind=kind, width=width, height=height, surfels=surfels, gaussians=gaussians, dtype=dtype, degree=degree,
             dim=dim, samples=samples, mip=mip, aux=aux, views=views, front=front)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a thumbnail or a preview of one object: nothing but latency
        _case("tiny_view", "view", 128, 128, 1000, 4000),
        # joint-stage training on a small crop with 2D Gaussians (2D-GES), odd sizes
        _case("small_train_2d", "train", 161, 117, 5003, 7001, dim=2),
        # one frame of the full-HD scene, with the id map and W_G
        _case("view_1080p", "view", 1920, 1080, 1_000_000, 300_000),
        # a window of an odd size over a compact scene: BF16 storage, SH degree 2, colour and depth only
        _case("view_ragged_bf16", "view", 1237, 823, 333_333, 120_001, dtype="bf16", degree=2, aux=False),
        # one frame with the primitive counts of the paper's outdoor scenes (mostly Gaussians)
        _case("view_gaussian_heavy", "view", 1920, 1080, 200_000, 2_500_000, aux=False),
        # an anti-aliased still: 4 samples per pixel, Mip-GES filters, FP16 storage
        _case("view_msaa_mip_f16", "view", 1264, 832, 500_000, 250_000, dtype="f16", samples=4, mip=True),
        # one frame of the largest scene at 4K
        _case("view_4k_f16", "view", 3840, 2160, 2_250_000, 750_000, dtype="f16", aux=False),
        # depth and normal maps for meshing, 2D Gaussians
        _case("geometry_2d", "geom", 1600, 1060, 500_000, 300_000, dim=2),
        # one step of the joint optimisation stage: forward, L1 loss, backward
        _case("train_1600x1060", "train", 1600, 1060, 500_000, 500_000),
        # one step of the coarse stage: translucent surfels, forward and backward
        _case("translucent_train", "translucent", 1920, 1080, 1_000_000, 1),
        # a camera path rendered by one captured graph
        _case("orbit_batch_16", "batch", 1920, 1080, 1_000_000, 300_000, aux=False, views=16),
        # eight scenes of uneven sizes for as many clients in one call, FP16 storage
        _case("uneven_batch_8", "uneven", 3840, 2160, 2_250_000, 750_000, dtype="f16", aux=False, views=8),
    ]


def draw(rng):
    def log(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(("view", "view", "view", "geom", "train", "train", "translucent", "batch", "uneven"))
    w, h = log(64, 3840), 0
    h = max(48, min(2160, int(w * rng.uniform(0.5, 1.0))))
    n, m = log(1000, 2_000_000), log(1000, 1_500_000)
    views = 1
    if kind == "batch":
        views, w, h, n, m = rng.randint(2, 12), min(w, 1920), min(h, 1080), min(n, 1_000_000), min(m, 300_000)
    if kind == "uneven":
        views = rng.randint(2, 7)
    if kind == "translucent":
        w, h, n, m = min(w, 1920), min(h, 1080), min(n, 900_000), 1
    if kind == "train":
        w, h, n, m = min(w, 1920), min(h, 1080), min(n, 1_000_000), min(m, 600_000)
    train = kind in ("train", "translucent")
    dim = rng.choice((3, 3, 2)) if kind != "translucent" else 3
    return _case(None, kind, w, h, n, m, dtype="f32" if train else rng.choice(("f32", "f16", "bf16")),
                 degree=rng.choice((3, 3, 3, 2, 1, 0)), dim=dim,
                 samples=rng.choice((1, 1, 4)) if kind in ("view", "geom", "train") else 1,
                 mip=dim == 3 and rng.random() < 0.3, aux=rng.random() < 0.5, views=views,
                 front=rng.random() < 0.5 if kind == "translucent" else False)


# ---------------------------------------------------------------------------
# inputs

def _f32(x):
    return float(torch.tensor(x, dtype=torch.float64).to(torch.float32))


def _look_at(eye, target, up, width, height):
    eye, target, up = (torch.tensor(v, dtype=torch.float64) for v in (eye, target, up))
    z = (target - eye) / (target - eye).norm()
    x = torch.linalg.cross(z, up)
    x = x / x.norm()
    y = torch.linalg.cross(z, x)
    rot = torch.stack([x, y, z])
    w2c = torch.cat([rot, -(rot @ eye)[:, None]], 1)
    f = _f32(0.5 * height / math.tan(math.radians(30.0)))
    return dict(width=width, height=height, fx=f, fy=f, cx=0.5 * width, cy=0.5 * height,
                world_to_cam=[[_f32(float(v)) for v in row] for row in w2c], znear=_f32(ZNEAR), bg=[0.0, 0.0, 0.0])


def _small(n):
    """Small scenes are one object close by; large ones fill a 20 m box."""
    return n < 50_000


def _cameras(case, n, width, height, count, gen):
    phase = float(torch.rand((), generator=gen, device=gen.device))
    cams = []
    for k in range(count):
        th = 2.0 * math.pi * (k + phase) / count
        if _small(n):
            cams.append(_look_at((3.0 * math.sin(th), 0.0, -3.0 * math.cos(th)), (0, 0, 0), (0, 1, 0), width, height))
        else:
            cams.append(_look_at((15.0 * math.cos(th), 15.0 * math.sin(th), 5.0), (0, 0, 0), (0, 0, 1), width, height))
    return cams


def _quat_mul(a, b):
    aw, ax, ay, az = a.unbind(-1)
    bw, bx, by, bz = b.unbind(-1)
    return torch.stack([aw * bw - ax * bx - ay * by - az * bz, aw * bx + ax * bw + ay * bz - az * by,
                        aw * by - ax * bz + ay * bw + az * bx, aw * bz + ax * by - ay * bx + az * bw], -1)


def _tensors(case, n, m, gen):
    """The scene's attribute tensors (n surfels, m Gaussians) in storage types."""
    dev = gen.device
    u = lambda *s: torch.rand(s, generator=gen, device=dev)  # noqa: E731
    g = lambda *s: torch.randn(s, generator=gen, device=dev)  # noqa: E731
    small = _small(n)
    no = 3 if small else 200
    box = 0.7 if small else 10.0
    sphere = torch.ones(no, dtype=torch.bool, device=dev) if small else u(no) < 0.5
    centre = (2 * u(no, 3) - 1) * box
    radius, side = 0.5 + 0.5 * u(no), 1.0 + 3.0 * u(no)
    normal = torch.nn.functional.normalize(g(no, 3), dim=1)
    area = torch.where(sphere, 4 * math.pi * radius ** 2, side ** 2)
    edge = torch.cumsum(area / area.sum(), 0)
    which = torch.searchsorted(edge, u(n)).clamp(max=no - 1)
    dirs = torch.nn.functional.normalize(g(n, 3), dim=1)
    pn = normal[which]
    ref = torch.where(pn[:, :1].abs() < 0.8, torch.tensor([[1.0, 0, 0]], device=dev), torch.tensor([[0, 1.0, 0]], device=dev))
    b1 = torch.nn.functional.normalize(torch.linalg.cross(pn, ref), dim=1)
    b2 = torch.linalg.cross(pn, b1)
    uv = (u(n, 2) - 0.5) * side[which, None]
    plane = centre[which] + uv[:, :1] * b1 + uv[:, 1:] * b2 + 0.002 * g(n, 1) * pn
    on = sphere[which, None]
    s_pos = torch.where(on, centre[which] + radius[which, None] * dirs, plane)
    nrm = torch.where(on, dirs, pn)
    # rotation taking z to the normal, after a uniform angle about z
    al = torch.stack([1 + nrm[:, 2], -nrm[:, 1], nrm[:, 0], torch.zeros(n, device=dev)], 1)
    al[nrm[:, 2] < -0.9999] = torch.tensor([0.0, 1.0, 0.0, 0.0], device=dev)
    ph = math.pi * u(n)
    zero = torch.zeros(n, device=dev)
    s_rot = _quat_mul(torch.nn.functional.normalize(al, dim=1), torch.stack([ph.cos(), zero, zero, ph.sin()], 1))
    k = (case["degree"] + 1) ** 2

    def sh(c):
        t = 0.05 * g(c, k, 3)
        t[:, 0] = u(c, 3)
        return t

    anchor = torch.randint(0, n, (m,), generator=gen, device=dev)
    t = dict(s_pos=s_pos, s_rot=s_rot, s_scale=0.01 + 0.04 * u(n, 2), s_sh=sh(n),
             g_pos=s_pos[anchor] + 0.02 * g(m, 3), g_rot=torch.nn.functional.normalize(g(m, 4), dim=1),
             g_scale=torch.exp(-5.0 + 0.5 * g(m, case["dim"])), g_opac=0.05 + 0.85 * u(m), g_sh=sh(m))
    dt = DTYPES[case["dtype"]]
    return {key: v.to(dt if key in ATTRS or key.endswith("_sh") else torch.float32).contiguous() for key, v in t.items()}


def _generator(seed):
    gen = torch.Generator(device="cuda" if torch.cuda.is_available() else "cpu")
    gen.manual_seed(int(seed))
    return gen


def _inputs(case, seed):
    """Everything a case is made of: the parts (tensors, 3D filter, cameras) and the step's own inputs."""
    gen = _generator(seed)
    c = case
    parts = []
    count = c["views"] if c["kind"] == "uneven" else 1
    for k in range(count):
        # uneven batch: from a thirtieth of the primitives at a sixth of the width up to the full scene
        f = 1.0 if count == 1 else (count - 1 - k) / (count - 1)
        f = 0.0 if count == 1 else f
        n, m = (max(1, int(round(x * 30.0 ** -f))) for x in (c["surfels"], c["gaussians"]))
        w, h = (max(16, int(round(x * 6.0 ** -f))) for x in (c["width"], c["height"]))
        t = _tensors(c, n, m, gen)
        cams = _cameras(c, n, w, h, c["views"] if c["kind"] == "batch" else 1, gen)
        filt = None
        if c["mip"]:
            # the sampling limit of a camera at the Gaussian's distance (Mip-Splatting's world filter)
            eye = torch.tensor(_eye(cams[0]), dtype=torch.float32, device=gen.device)
            filt = 0.2 * ((t["g_pos"] - eye).norm(dim=1) / cams[0]["fx"]) ** 2
        parts.append((t, filt, cams))
    extra = {}
    if c["kind"] in ("train", "translucent"):
        low = torch.rand((1, 3, 9, 16), generator=gen, device=gen.device)
        extra["target"] = torch.nn.functional.interpolate(low, (c["height"], c["width"]), mode="bilinear",
                                                          align_corners=True)[0].contiguous()
    if c["kind"] == "translucent":
        u = torch.rand((c["surfels"],), generator=gen, device=gen.device)
        extra["w"] = 30.0 + 225.0 * u if c["front"] else 0.1 + 29.9 * u
    return parts, extra


def _eye(cam):
    w = torch.tensor(cam["world_to_cam"], dtype=torch.float64)
    return [float(v) for v in -(w[:, :3].T @ w[:, 3])]


def _opts(case):
    o = {}
    if case["samples"] != 1:
        o["samples"] = case["samples"]
    if case["mip"]:
        o.update(filter=1, lowpass=0.1)
    return o or None


def prepare(case, seed):
    parts, extra = _inputs(case, seed)
    kind = case["kind"]
    st = dict(kind=kind, opts=_opts(case), aux=case["aux"], front=case["front"], cams=parts[0][2], **extra)
    st["scenes"] = [R.GESScene(case["degree"], g_filter3d=f, **t) for t, f, _ in parts]
    if kind == "train":
        t = st["scenes"][0].t
        st["params"] = [t[k] for k in ("g_pos", "g_rot", "g_scale", "g_opac", "g_sh", "s_sh")]
        for p in st["params"]:
            p.requires_grad_(True)
    if kind == "batch":
        st["batch"] = R.GESBatch(st["scenes"], st["cams"], opts=st["opts"])
    if kind == "uneven":
        st["cams"] = [cams[0] for _, _, cams in parts]
        st["out"] = [(torch.empty((3, c["height"], c["width"]), device="cuda"),
                      torch.empty((c["height"], c["width"]), device="cuda")) for c in st["cams"]]
    return st


def run(st):
    kind, scene, cam, opts = st["kind"], st["scenes"][0], st["cams"][0], st["opts"]
    if kind == "view":
        return R.render(scene, cam, opts, with_aux=st["aux"])
    if kind == "geom":
        return R.render_geom(scene, cam, opts)
    if kind == "train":
        rgb, depth, sid, aux = R.render_differentiable(scene, cam, opts)
        loss = (rgb - st["target"]).abs().mean()
        grads = torch.autograd.grad(loss, st["params"])
        return dict(rgb=rgb.detach(), depth=depth, id=sid, aux=aux, grads=list(grads))
    if kind == "translucent":
        fwd = R.render_translucent(scene, cam, st["w"], st["front"], opts, cover=True)
        dl = (fwd["rgb"] - st["target"]).sign() / st["target"].numel()
        grads = R.render_translucent_backward(scene, cam, st["w"], fwd, dl, st["front"], opts)
        return dict({k: fwd[k] for k in ("rgb", "T", "front", "last", "Tlast", "cover")}, grads=grads)
    if kind == "batch":
        b = st["batch"]
        b.launch()
        b.sync()
        return [b.rgb, b.depth]
    out = R.render_batch(st["scenes"], st["cams"], list(range(len(st["scenes"]))), opts, st["out"])
    return [list(p) for p in out]


def _sizes(case):
    """(surfels, Gaussians, width, height, views of it) of each scene of a case."""
    c = case
    if c["kind"] != "uneven":
        return [(c["surfels"], c["gaussians"], c["width"], c["height"], c["views"])]
    out = []
    for k in range(c["views"]):
        f = (c["views"] - 1 - k) / (c["views"] - 1)
        out.append(tuple(max(1, int(round(x * 30.0 ** -f))) for x in (c["surfels"], c["gaussians"])) +
                   tuple(max(16, int(round(x * 6.0 ** -f))) for x in (c["width"], c["height"])) + (1,))
    return out


def work(case):
    c = case
    e = 4 if c["dtype"] == "f32" else 2
    k = (c["degree"] + 1) ** 2
    bs, bg = 12 + e * (6 + 3 * k), 12 + e * (5 + c["dim"] + 3 * k)
    out = {"view": 16 + (8 if c["aux"] else 0) + (12 if c["aux"] and c["samples"] == 4 else 0), "geom": 60, "train": 24,
           "translucent": 28, "batch": 16, "uneven": 16}[c["kind"]]
    total, flops = 0, 0
    for n, m, w, h, v in _sizes(c):
        if c["kind"] == "translucent":
            m = 0
        total += n * bs + m * bg + out * w * h * v
        # set-up and SH colour of each primitive in each view, and the winning fragment of each sample
        flops += v * ((n + m) * (300 + 6 * k) + 40 * w * h * c["samples"])
        if c["kind"] in ("train", "translucent"):
            # target and dL in, gradients out
            total += 24 * w * h + (m * bg + n * 12 * k if c["kind"] == "train" else n * (bs + 4) + 4 * n)
            flops *= 3
    return {"bytes": float(total), "flops": float(flops)}


# ---------------------------------------------------------------------------
# the same in 64 bits

PAIRS = 6_000_000        # (primitive, pixel) pairs expanded at a time


def _rot(q):
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y), 2 * (x * y + w * z),
                        1 - 2 * (x * x + z * z), 2 * (y * z - w * x), 2 * (x * z - w * y), 2 * (y * z + w * x),
                        1 - 2 * (x * x + y * y)], 1).reshape(-1, 3, 3)


def _colour(sh, pos, eye):
    """max(0, 0.5 + sum_k SH_k Y_k) at the unit vector from the primitive to the camera."""
    d = eye - pos
    x, y, z = (d / d.norm(dim=1, keepdim=True)).unbind(1)
    pi = math.pi
    Y = [torch.full_like(x, 0.5 / math.sqrt(pi))]
    if sh.shape[1] > 1:
        c = math.sqrt(3 / (4 * pi))
        Y += [-c * y, c * z, -c * x]
    if sh.shape[1] > 4:
        a, b = math.sqrt(15 / pi) / 2, math.sqrt(5 / pi) / 4
        Y += [a * x * y, -a * y * z, b * (3 * z * z - 1), -a * x * z, a / 2 * (x * x - y * y)]
    if sh.shape[1] > 9:
        a, b, c, e = math.sqrt(35 / (2 * pi)) / 4, math.sqrt(105 / pi) / 2, math.sqrt(21 / (2 * pi)) / 4, math.sqrt(7 / pi) / 4
        Y += [-a * y * (3 * x * x - y * y), b * x * y * z, -c * y * (5 * z * z - 1), e * z * (5 * z * z - 3),
              -c * x * (5 * z * z - 1), b / 2 * z * (x * x - y * y), -a * x * (x * x - 3 * y * y)]
    return (0.5 + (sh * torch.stack(Y, 1)[:, :, None]).sum(1)).clamp(min=0)


class _Cam:
    def __init__(self, cam, dev):
        w = torch.tensor(cam["world_to_cam"], dtype=torch.float64, device=dev)
        self.R, self.t = w[:, :3], w[:, 3]
        self.eye = -(self.R.T @ self.t)
        self.f, self.cx, self.cy = cam["fx"], cam["cx"], cam["cy"]
        self.W, self.H, self.zn = cam["width"], cam["height"], cam["znear"]


def _boxes(cam, u, v, ok):
    """Pixel ranges of pixel-coordinate extents u, v ([n,2] lo/hi), a pixel wider; empty where not ok."""
    lim = lambda t, n: t.nan_to_num(0.0, 1e9, -1e9).clamp(-10, n + 10)  # noqa: E731
    x0, x1 = lim(u[:, 0], cam.W).floor().long() - 1, lim(u[:, 1], cam.W).ceil().long() + 1
    y0, y1 = lim(v[:, 0], cam.H).floor().long() - 1, lim(v[:, 1], cam.H).ceil().long() + 1
    x0, y0, x1, y1 = x0.clamp(min=0), y0.clamp(min=0), x1.clamp(max=cam.W - 1), y1.clamp(max=cam.H - 1)
    w, h = (x1 - x0 + 1).clamp(min=0), (y1 - y0 + 1).clamp(min=0)
    return x0, y0, w, torch.where(ok, w * h, torch.zeros_like(w))


def _pairs(box, cam):
    """(primitive, x, y) of every footprint, in chunks."""
    x0, y0, w, count = box
    live = count.nonzero()[:, 0]
    if not live.numel():
        return
    end = torch.cumsum(count[live], 0)
    total, at, base = int(end[-1]), 0, 0
    while base < total:
        stop = max(at + 1, int(torch.searchsorted(end, base + PAIRS, right=True)))
        ids = live[at:stop]
        c = count[ids]
        p = torch.repeat_interleave(ids, c)
        k = torch.arange(p.numel(), device=p.device) - torch.repeat_interleave(torch.cumsum(c, 0) - c, c)
        yield p, x0[p] + k % w[p], y0[p] + k // w[p]
        base, at = int(end[stop - 1]), stop


def _discs(cam, pos, rot, scale, radius):
    """Camera-space discs and their footprints: corners of the enclosing rectangle, or the image where it nears the camera."""
    P = pos @ cam.R.T + cam.t
    F = cam.R @ _rot(rot)
    U, V, N = F[:, :, 0], F[:, :, 1], F[:, :, 2]
    a, b = (radius * scale[:, 0])[:, None] * U, (radius * scale[:, 1])[:, None] * V
    cor = torch.stack([P + a + b, P - a + b, P + a - b, P - a - b], 1)
    near = cor[:, :, 2].amin(1) <= cam.zn * 1.01
    u, v = (cam.f * cor[:, :, k] / cor[:, :, 2] + o for k, o in ((0, cam.cx), (1, cam.cy)))
    u = torch.stack([torch.where(near, -1e9, u.amin(1)), torch.where(near, 1e9, u.amax(1))], 1)
    v = torch.stack([torch.where(near, -1e9, v.amin(1)), torch.where(near, 1e9, v.amax(1))], 1)
    ok = cor[:, :, 2].amax(1) > cam.zn
    return dict(P=P, U=U, V=V, N=N, s=scale, box=_boxes(cam, u.detach(), v.detach(), ok))


def _hit(D, p, cam, u, v):
    """1/z of the ray-plane hit and its disc coordinates in scale units."""
    d = torch.stack([(u - cam.cx) / cam.f, (v - cam.cy) / cam.f, torch.ones_like(u)], 1)
    N, P = D["N"][p], D["P"][p]
    iz = (N * d).sum(1) / (N * P).sum(1)
    X = d / iz[:, None] - P
    return iz, (X * D["U"][p]).sum(1) / D["s"][p, 0], (X * D["V"][p]).sum(1) / D["s"][p, 1]


def _surfels(cam, t, samples):
    """Per sample 1/z and surfel of the nearest fragment (-1: none), and the discs."""
    n, dev = t["s_pos"].shape[0], t["s_pos"].device
    D = _discs(cam, t["s_pos"], t["s_rot"], t["s_scale"], torch.full((n,), math.sqrt(R2), dtype=torch.float64, device=dev))
    grid = [(0.5, 0.5)] if samples == 1 else [(0.25 + 0.5 * (k & 1), 0.25 + 0.5 * (k >> 1)) for k in range(4)]
    best = torch.zeros((len(grid), cam.H * cam.W), dtype=torch.float64, device=dev)
    win = torch.full_like(best, n, dtype=torch.int64)
    for phase in (0, 1):
        for p, x, y in _pairs(D["box"], cam):
            for k, (ox, oy) in enumerate(grid):
                iz, a, b = _hit(D, p, cam, x + ox, y + oy)
                ok = (iz > 0) & (iz < 1 / cam.zn) & (a * a + b * b <= R2)
                pix = y * cam.W + x
                if phase == 0:
                    best[k].scatter_reduce_(0, pix[ok], iz[ok], "amax")
                else:
                    ok &= iz == best[k][pix]
                    win[k].scatter_reduce_(0, pix[ok], p[ok], "amin")
    return best, torch.where(win == n, -1, win), D


def _gauss(cam, t, case, filt):
    """Per-Gaussian projected quantities: footprint, alpha arguments, depth test."""
    low = 0.1 if case["mip"] else 0.3
    pos, sc, op = t["g_pos"], t["g_scale"], t["g_opac"]
    P = pos @ cam.R.T + cam.t
    x, y, z = P.unbind(1)
    zs = torch.where(z > cam.zn, z, torch.ones_like(z))
    zero = torch.zeros_like(z)
    J = torch.stack([cam.f / zs, zero, -cam.f * x / zs ** 2, zero, cam.f / zs, -cam.f * y / zs ** 2], 1).reshape(-1, 2, 3)
    Rm = _rot(t["g_rot"])
    G = dict(P=P, col=_colour(t["g_sh"], pos, cam.eye))
    if case["dim"] == 2:
        F = cam.R @ Rm
        Jl = J @ (F[:, :, :2] * sc[:, None, :])
        M = Jl.transpose(1, 2) @ Jl
        det = M[:, 0, 0] * M[:, 1, 1] - M[:, 0, 1] ** 2
        S1, S2 = (1 + low * M[:, 1, 1] / det).sqrt(), (1 + low * M[:, 0, 0] / det).sqrt()
        sig = op / (S1 * S2)
        ok = (z > cam.zn) & (sig >= ALPHA_MIN) & (det > 0)
        rad = (2 * (sig / ALPHA_MIN).clamp(min=1).log()).sqrt()
        D = _discs(cam, pos, t["g_rot"], torch.stack([sc[:, 0] * S1, sc[:, 1] * S2], 1), rad.detach())
        G.update(D=D, sig=sig, box=D["box"][:3] + (torch.where(ok, D["box"][3], 0),), eps=2.5 * sc.sum(1), n=F[:, :, 2])
        return G
    se = sc if filt is None else (sc ** 2 + filt[:, None]).sqrt()
    if filt is not None:
        op = op * (sc / se).prod(1)
    T = J @ cam.R @ (Rm * se[:, None, :])
    S = T @ T.transpose(1, 2)
    A, B, C = S[:, 0, 0] + low, S[:, 0, 1], S[:, 1, 1] + low
    x0 = torch.linalg.cross(T[:, 0], T[:, 1])
    det0 = (x0 * x0).sum(1)
    det = det0 + low * (S[:, 0, 0] + S[:, 1, 1]) + low * low
    if case["mip"]:
        op = op * (det0 / det).sqrt()
    ok = (z > cam.zn) & (op >= ALPHA_MIN)
    px, py = cam.f * x / zs + cam.cx, cam.f * y / zs + cam.cy
    q = (2 * (op / ALPHA_MIN).clamp(min=1).log()).detach()
    hx, hy = (q * A).detach().sqrt(), (q * C).detach().sqrt()
    box = _boxes(cam, torch.stack([px - hx, px + hx], 1).detach(), torch.stack([py - hy, py + hy], 1).detach(), ok)
    k = sc.abs().argmin(1)
    nrm = (Rm.gather(2, k[:, None, None].expand(-1, 3, 1))[:, :, 0]) @ cam.R.T
    G.update(px=px, py=py, ia=C / det, ib=-B / det, ic=A / det, sig=op, box=box, eps=5.0 / 3.0 * sc.sum(1), n=nrm)
    return G


def _gauss_alpha(G, p, x, y, cam, dim):
    """alpha, and whether the pair passes the near plane; its depth less eps."""
    if dim == 2:
        iz, a, b = _hit(G["D"], p, cam, x + 0.5, y + 0.5)
        z = 1 / iz
        return G["sig"][p] * torch.exp(-0.5 * (a * a + b * b)), (iz > 0) & (iz < 1 / cam.zn), z
    dx, dy = x + 0.5 - G["px"][p], y + 0.5 - G["py"][p]
    q = G["ia"][p] * dx * dx + 2 * G["ib"][p] * dx * dy + G["ic"][p] * dy * dy
    return G["sig"][p] * torch.exp(-0.5 * q), torch.ones_like(p, dtype=torch.bool), G["P"][p, 2]


def _render64(cam, t, case, filt, geo=False):
    best, win, D = _surfels(cam, t, case["samples"])
    col = torch.cat([_colour(t["s_sh"], t["s_pos"], cam.eye), torch.zeros((1, 3), dtype=torch.float64, device=best.device)])
    Cs = col[win].mean(0)                                    # [HW,3]; -1 picks the background row
    bmax = best.amax(0)
    Ds = torch.where(bmax > 0, 1 / bmax, math.inf)
    G = _gauss(cam, t, case, filt)
    HW = cam.W * cam.H
    sums = torch.zeros((HW, 8), dtype=torch.float64, device=best.device)   # W_G, C_G, D_G, N_G
    side = torch.where((G["n"] * G["P"]).sum(1) > 0, -1.0, 1.0)[:, None] * G["n"]
    for p, x, y in _pairs(G["box"], cam):
        a, ok, z = _gauss_alpha(G, p, x, y, cam, case["dim"])
        pix = y * cam.W + x
        ok &= (a >= ALPHA_MIN) & (z - G["eps"][p] < Ds[pix])
        p, a, z, pix = p[ok], a[ok], z[ok], pix[ok]
        sums.index_add_(0, pix, a[:, None] * torch.cat([torch.ones_like(z)[:, None], G["col"][p], z[:, None], side[p]], 1))
    W = sums[:, 0]
    rgb = (Cs + sums[:, 1:4]) / (1 + W)[:, None]
    plane = lambda v: v.T.reshape(-1, cam.H, cam.W) if v.dim() == 2 else v.reshape(cam.H, cam.W)  # noqa: E731
    out = dict(rgb=plane(rgb), depth=plane(Ds), id=None, aux=plane(W))
    if geo:
        ws = (bmax > 0).double()
        near = win.gather(0, best.argmax(0, keepdim=True))[0].clamp(min=0)
        ns = torch.where((D["N"] * D["P"]).sum(1) > 0, -1.0, 1.0)[:, None] * D["N"]
        ns = ns[near] * ws[:, None]
        wt = ws + W
        out.update(ns=plane(ns), dg=plane(sums[:, 4]), ng=plane(sums[:, 5:8]),
                   dsmooth=plane(torch.where(wt > 0, (torch.where(ws > 0, Ds, 0.0) + sums[:, 4]) / wt, math.inf)),
                   nsmooth=plane(torch.where(wt[:, None] > 0, (ns + sums[:, 5:8]) / wt[:, None].clamp(min=1e-300), 0.0)))
    return out, dict(win=win, Ds=Ds, W=W, C=rgb)


def _train64(cam, t, case, filt, target):
    out, st = _render64(cam, t, case, filt)
    g = ((out["rgb"] - target).sign() / target.numel()).reshape(3, -1).T     # dL/dC [HW,3]
    kg = g / (1 + st["W"])[:, None]
    kgC = (kg * st["C"]).sum(1)
    names = ("g_pos", "g_rot", "g_scale", "g_opac", "g_sh")
    leaf = {k: t[k].clone().requires_grad_(True) for k in names}
    G = _gauss(cam, dict(t, **leaf), case, filt)
    D = G.get("D", {})
    keys = [(G, k) for k in ("col", "sig") + (() if D else ("px", "py", "ia", "ib", "ic"))] + \
           [(D, k) for k in (("P", "U", "V", "N", "s") if D else ())]
    whole = [d[k] for d, k in keys]
    for (d, k), v in zip(keys, whole):
        d[k] = v.detach().requires_grad_(True)
    G["P"] = G["P"].detach()
    for p, x, y in _pairs(G["box"], cam):
        pix = y * cam.W + x
        with torch.no_grad():
            a, ok, z = _gauss_alpha(G, p, x, y, cam, case["dim"])
            ok &= (a >= ALPHA_MIN) & (z - G["eps"][p] < st["Ds"][pix])
        if bool(ok.any()):
            p, x, y, pix = p[ok], x[ok], y[ok], pix[ok]
            a = _gauss_alpha(G, p, x, y, cam, case["dim"])[0]
            (a * ((kg[pix] * G["col"][p]).sum(1) - kgC[pix])).sum().backward()
    got = [d[k].grad if d[k].grad is not None else torch.zeros_like(d[k]) for d, k in keys]
    grads = torch.autograd.grad(whole, [leaf[k] for k in names], got, allow_unused=True)
    grads = [v if v is not None else torch.zeros_like(leaf[k]) for k, v in zip(names, grads)]
    sh = t["s_sh"].clone().requires_grad_(True)
    acc = torch.zeros_like(t["s_pos"])
    for w in st["win"]:
        on = w >= 0
        acc.index_add_(0, w[on], kg[on] / st["win"].shape[0])
    grads += torch.autograd.grad(_colour(sh, t["s_pos"], cam.eye), [sh], acc)
    return dict(rgb=out["rgb"], depth=out["depth"], id=None, aux=out["aux"], grads=grads)


def _translucent64(cam, t, case, w, target):
    """Sorted blending by bands of rows: pairs ordered by (pixel, order), transmittance by a running sum of logs."""
    names = ("s_pos", "s_rot", "s_scale")
    n, dev = t["s_pos"].shape[0], t["s_pos"].device
    leaf = {k: t[k].clone().requires_grad_(True) for k in names + ("s_sh",)}
    D = _discs(cam, leaf["s_pos"], leaf["s_rot"], leaf["s_scale"], torch.full((n,), math.sqrt(R2), dtype=torch.float64, device=dev))
    keys = ("P", "U", "V", "N", "s")
    whole = [D[k] for k in keys] + [_colour(leaf["s_sh"], leaf["s_pos"], cam.eye)]
    for k in keys:
        D[k] = D[k].detach().requires_grad_(True)
    col, wl = whole[-1].detach().requires_grad_(True), w.clone().requires_grad_(True)
    rank = torch.empty(n, dtype=torch.int64, device=dev)
    rank[torch.sort(D["P"].detach()[:, 2].float(), stable=True).indices] = torch.arange(n, device=dev)
    HW = cam.W * cam.H
    rgb, T, Tl = (torch.zeros((HW, 3), dtype=torch.float64, device=dev), torch.ones(HW, dtype=torch.float64, device=dev),
                  torch.ones(HW, dtype=torch.float64, device=dev))
    x0, y0, bw, count = D["box"]
    rows = torch.where(bw > 0, count // bw.clamp(min=1), 0)

    def opacity(p, x, y):
        iz, a, b = _hit(D, p, cam, x + 0.5, y + 0.5)
        Gs = torch.exp(-0.5 * (a * a + b * b))
        al = (wl[p] * Gs).clamp(max=1)
        return iz, al, (iz > 0) & (iz < 1 / cam.zn) & (torch.minimum(al, Gs) >= ALPHA_MIN)

    step = max(1, min(cam.H, int(cam.H * 16 * PAIRS // max(1, int(count.sum())))))
    for r0 in range(0, cam.H, step):
        lo, hi = y0.clamp(min=r0), (y0 + rows).clamp(max=min(cam.H, r0 + step))
        band = (x0, lo, bw, bw * (hi - lo).clamp(min=0))
        found = []
        with torch.no_grad():
            for p, x, y in _pairs(band, cam):
                iz, al, ok = opacity(p, x, y)
                found.append((p[ok], x[ok], y[ok], iz[ok]))
        if not found or not sum(f[0].numel() for f in found):
            continue
        p, x, y, iz = (torch.cat(v) for v in zip(*found))
        pix = y * cam.W + x
        key = rank[p]
        if case["front"]:
            best = torch.zeros(HW, dtype=torch.float64, device=dev).scatter_reduce_(0, pix, iz, "amax")
            first = torch.full((HW,), n, dtype=torch.int64, device=dev)
            lead = iz == best[pix]
            first.scatter_reduce_(0, pix[lead], p[lead], "amin")
            key = torch.where(first[pix] == p, torch.full_like(key, -1), key)
        order = torch.argsort(pix * (n + 1) + key + 1)
        p, x, y, pix = p[order], x[order], y[order], pix[order]
        al = opacity(p, x, y)[1]
        start = torch.ones_like(pix, dtype=torch.bool)
        start[1:] = pix[1:] != pix[:-1]
        at = torch.cummax(torch.where(start, torch.arange(pix.numel(), device=dev), 0), 0).values
        lg = torch.log1p(-al.clamp(max=1 - 1e-12))
        cs = torch.cumsum(lg, 0)
        before = torch.exp(cs - lg - (cs - lg)[at])          # transmittance before each entry
        with torch.no_grad():
            on = before >= 1e-4                              # blending stops once it is below
        before = torch.where(on, before, 0.0)
        al = torch.where(on, al, 0.0)
        band_rgb = torch.zeros((HW, 3), dtype=torch.float64, device=dev).index_add_(0, pix, (al * before)[:, None] * col[p])
        ys = slice(r0 * cam.W, min(cam.H, r0 + step) * cam.W)
        with torch.no_grad():
            rgb[ys] = band_rgb[ys]
            last = on.clone()
            last[:-1] = on[:-1] & ((~on)[1:] | start[1:])
            Tl[pix[last]] = before[last]
            T[pix[last]] = before[last] * (1 - al[last])
            g = ((band_rgb.T.reshape(3, cam.H, cam.W) - target).sign() / target.numel()).reshape(3, -1).T
        (band_rgb * g)[ys].sum().backward()
    got = [D[k].grad for k in keys] + [col.grad]
    got = [v if v is not None else torch.zeros_like(x) for v, x in zip(got, whole)]
    grads = torch.autograd.grad(whole, [leaf[k] for k in names + ("s_sh",)], got, allow_unused=True)
    grads = dict(zip(names + ("s_sh",), grads), s_w=wl.grad if wl.grad is not None else torch.zeros_like(w))
    plane = lambda v: v.T.reshape(-1, cam.H, cam.W) if v.dim() == 2 else v.reshape(cam.H, cam.W)  # noqa: E731
    return dict(rgb=plane(rgb), T=plane(T), front=None, last=None, Tlast=plane(Tl), cover=None, grads=grads)


def exact(case, seed):
    parts, extra = _inputs(case, seed)
    up = lambda v: None if v is None else v.double()  # noqa: E731
    parts = [({k: up(v) for k, v in t.items()}, up(f), [_Cam(c, v.device) for c in cams])
             for t, f, cams in parts for v in (t["s_pos"],)]
    t, filt, cams = parts[0]
    if case["kind"] == "view":
        out = _render64(cams[0], t, case, filt)[0]
        return out if case["aux"] else dict(rgb=out["rgb"], depth=out["depth"])
    if case["kind"] == "geom":
        out = _render64(cams[0], t, case, filt, geo=True)[0]
        return {k: out[k] for k in ("rgb", "depth", "ns", "dsmooth", "nsmooth", "dg", "ng")}
    if case["kind"] == "train":
        return _train64(cams[0], t, case, filt, up(extra["target"]))
    if case["kind"] == "translucent":
        return _translucent64(cams[0], t, case, up(extra["w"]), up(extra["target"]))
    if case["kind"] == "batch":
        outs = [_render64(c, t, case, filt)[0] for c in cams]
        return [[o["rgb"] for o in outs], [o["depth"] for o in outs]]
    outs = [_render64(c[0], tt, case, f)[0] for tt, f, c in parts]
    return [[o["rgb"], o["depth"]] for o in outs]
