"""Performance cases of the k-shell renderer and its neural textures.

Each case is a dict of plain sizes and options; `prepare` makes its inputs on
the GPU from a seed (geometry, textures, cameras, targets, parameters), `run`
is one pass through the package's public entry points, `work` the bytes and
operations that pass cannot do without, and `exact` its floating outputs in
64 bits from a plain torch statement of the method, which shares no code with
the package.  The workloads are the repository's own configurations (nested
noise-displaced spheres seen from a hemisphere, spherical-harmonic, RGBA and
baked byte textures, the fitting step and the networks that produce the
textures), at their full texture and image sizes with fewer views.
"""

from __future__ import annotations

import dataclasses
import math

import torch

import paper_2409_02482_gb300 as vs

RGBA, SH, BAKED = 0, 1, 2                 # texel formats (the values of vs.VS_TEX_*)
BAKED_STRIDE = (4, 16, 32, 32)            # bytes per texel of band l
BACKGROUND = (1.0, 0.9, 0.8)
ADAM_STEP = 100                           # steps taken before the timed one
LR, BETA1, BETA2, EPS = 1e-3, 0.9, 0.99, 1e-15
RESOLUTIONS = ((512, 512), (800, 800), (1024, 1024), (1920, 1080))
PRIME = 2654435761


# ----------------------------------------------------------------------------
# the cases
# ----------------------------------------------------------------------------

def listed():
    net = dict(levels=16, features=2, log2_table=19, base_res=16, growth=1.447, hidden=64, out_ch=27,
               tex_w=2048, tex_h=2048)
    return [
        # a small asset in a small window: latency and launches
        dict(name="frame_rgba_256", op="frame", k=3, tris=1280, fmt=RGBA, degree=0, pad=False, tex_w=256, tex_h=256,
             width=256, height=256, distance=3.0, atten=False),
        # the viewer's frame at the paper's evaluation size, continuous textures
        dict(name="frame_sh2_800", op="frame", k=7, tris=200000, fmt=SH, degree=2, pad=True, tex_w=2048, tex_h=2048,
             width=800, height=800, distance=4.0, atten=False),
        # the deployed asset (bytes, band images) in a full-HD window
        dict(name="frame_baked_1080p", op="frame", k=7, tris=200000, fmt=BAKED, degree=3, pad=True, tex_w=2048,
             tex_h=2048, width=1920, height=1080, distance=4.0, atten=False),
        # one differentiable render in a training script (autograd), odd sizes, attenuated opacity
        dict(name="autograd_sh1_odd", op="autograd", k=5, tris=50000, fmt=SH, degree=1, pad=True, tex_w=1000,
             tex_h=720, width=1001, height=751, distance=4.0, atten=True),
        # evaluation: many views of one asset in one call
        dict(name="views_sh2_800", op="views", k=7, tris=200000, fmt=SH, degree=2, pad=True, tex_w=2048, tex_h=2048,
             width=800, height=800, views=32, distance=4.0, atten=False),
        # the texture-fitting step: fused forward and adjoint over a batch of views
        dict(name="fit_sh2_800", op="fit", k=7, tris=200000, fmt=SH, degree=2, pad=True, tex_w=2048, tex_h=2048,
             width=800, height=800, views=24, distance=4.0, atten=False, loss="l2"),
        # fitting several assets of uneven size together
        dict(name="fit_uneven_sh1", op="uneven", objects=8, tris_lo=10000, tris_hi=1000000, fmt=SH, degree=1,
             pad=True, tex_w=1024, tex_h=1024, views=2, distance=4.0, atten=False, loss="l1"),
        # offline rendering of a large asset in 4K
        dict(name="views_sh3_4k", op="views", k=9, tris=2000000, fmt=SH, degree=3, pad=True, tex_w=4096, tex_h=4096,
             width=3840, height=2160, views=4, distance=3.5, atten=False),
        # a colour network written to its texture (default FP32 layers)
        dict(name="net_f32_forward", op="net_forward", tensor_cores=False, half=True, **net),
        # ... and its adjoint
        dict(name="net_f32_backward", op="net_backward", tensor_cores=False, **net),
        # both, with the layers on the tensor cores
        dict(name="net_tf32_both", op="net_both", tensor_cores=True, half=True, **net),
        # the optimizer's step on that network
        dict(name="adam", op="adam", tensor_cores=False, **net),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["frame", "frame", "autograd", "views", "fit", "uneven", "net_forward", "net_backward",
                     "net_both", "adam"])
    if op.startswith("net") or op == "adam":
        hidden = rng.choice([32, 64, 64, 64, 128])
        side = 1024 if hidden > 64 else 2048
        c = dict(op=op, tensor_cores=op == "net_both", levels=rng.choice([8, 12, 16]), features=rng.choice([1, 2, 2, 4]),
                 log2_table=rng.choice([12, 15, 19]), base_res=rng.choice([4, 16]),
                 growth=rng.choice([1.3, 1.4, 1.447]), hidden=hidden, out_ch=rng.choice([1, 4, 13, 27, 28]),
                 tex_w=_log_int(rng, 60, side), tex_h=_log_int(rng, 60, side))
        if op == "net_both" or op == "net_forward":
            c["half"] = rng.random() < 0.7
        return c
    fmt = rng.choice([SH, SH, SH, RGBA, BAKED])
    if fmt == BAKED and op not in ("frame", "views"):
        fmt = SH
    if op == "uneven":
        fmt = SH
    c = dict(op=op, fmt=fmt, degree=0 if fmt == RGBA else rng.choice([0, 1, 2, 3]), pad=rng.random() < 0.7,
             tex_w=8 * _log_int(rng, 16, 256), tex_h=8 * _log_int(rng, 16, 256),
             distance=rng.choice([3.0, 3.5, 4.0]), atten=rng.random() < 0.3)
    if op == "uneven":
        return dict(c, objects=rng.randint(2, 8), tris_lo=10000, tris_hi=_log_int(rng, 20000, 1000000),
                    views=rng.randint(1, 2), loss=rng.choice(["l1", "l2"]))
    c = dict(c, k=rng.randint(2, 9), tris=_log_int(rng, 2000, 500000), width=_log_int(rng, 100, 1920),
             height=_log_int(rng, 100, 1080))
    if op in ("views", "fit"):
        c["views"] = rng.randint(2, 12)
    if op == "fit":
        c["loss"] = rng.choice(["l1", "l2"])
    return c


# ----------------------------------------------------------------------------
# inputs (plain tensors)
# ----------------------------------------------------------------------------

def _generator(seed):
    return torch.Generator("cuda").manual_seed(int(seed) & 0x7FFFFFFF)


def _channels(fmt, degree):
    return 4 if fmt == RGBA else 1 + 3 * (degree + 1) ** 2


def _pitch(case):
    """Values per texel in memory: padded texels suit the widest loads."""
    c = _channels(case["fmt"], case["degree"])
    return c if case["fmt"] == RGBA or not case["pad"] else (8, 16, 32, 64)[case["degree"]]


def _n_lat(tris):
    return max(4, int(round(math.sqrt(tris / 4.0))))


def _sphere(n_lat):
    """Directions, UVs and outward counter-clockwise triangles of a lat-long
    sphere with a UV seam and one pole vertex per pole triangle."""
    n_lon, dev, f64 = 2 * n_lat, "cuda", torch.float64
    th = math.pi * torch.arange(1, n_lat, device=dev, dtype=f64) / n_lat
    ph = 2 * math.pi * torch.arange(n_lon + 1, device=dev, dtype=f64) / n_lon
    th, ph = torch.meshgrid(th, ph, indexing="ij")
    ring = torch.stack([th.sin() * ph.cos(), th.sin() * ph.sin(), th.cos()], -1).reshape(-1, 3)
    ring_uv = torch.stack([ph / (2 * math.pi), th / math.pi], -1).reshape(-1, 2)
    cols = torch.arange(n_lon, device=dev)
    pole_u = (cols.to(f64) + 0.5) / n_lon
    z = torch.zeros_like(pole_u)
    north, south = torch.stack([z, z, z + 1], 1), torch.stack([z, z, z - 1], 1)
    dirs = torch.cat([ring, north, south])
    uv = torch.cat([ring_uv, torch.stack([pole_u, z], 1), torch.stack([pole_u, z + 1], 1)])

    def rid(i, j):
        return i * (n_lon + 1) + j

    i = torch.arange(n_lat - 2, device=dev)[:, None]
    j = cols[None, :]
    a, b, c, d = rid(i, j), rid(i, j + 1), rid(i + 1, j), rid(i + 1, j + 1)
    quads = torch.stack([torch.stack([a, c, b], -1), torch.stack([b, c, d], -1)], 2).reshape(-1, 3)
    nid, last = ring.shape[0] + cols, n_lat - 2
    sid = nid + n_lon
    caps = [torch.stack([nid, rid(0, cols), rid(0, cols + 1)], -1),
            torch.stack([rid(last, cols), sid, rid(last, cols + 1)], -1)]
    return dirs, uv.float().contiguous(), torch.cat([quads] + caps).int().contiguous()


def _geometry(tris, g):
    """Nested shells 0.02 apart of one sphere displaced by a smooth seeded
    function (24 plane waves); `tris` holds each shell's triangle count."""
    r = dict(device="cuda", dtype=torch.float64, generator=g)
    u = torch.randn(24, 3, **r)
    u = u / u.norm(dim=1, keepdim=True)
    w = 1.0 + 3.0 * torch.rand(24, **r)
    p, a = 2 * math.pi * torch.rand(24, **r), torch.randn(24, **r) / w.sqrt()
    out, made = [], {}
    for i, t in enumerate(tris):
        n = _n_lat(t)
        if n not in made:
            dirs, uv, tri = _sphere(n)
            noise = sum(torch.cos(dirs @ u[q] * w[q] + p[q]) * a[q] for q in range(24))
            made[n] = dirs, uv, tri, noise / a.abs().sum()
        dirs, uv, tri, noise = made[n]
        out.append(dict(pos=(dirs * (1.0 + 0.2 * noise - 0.02 * i)[:, None]).float().contiguous(), uv=uv, tris=tri))
    return out


def _baked_bands(w, h, degree):
    """(byte offset, width, height, stride) of each band, and all bytes."""
    bands, off = [], 0
    for band in range(degree + 1):
        bw, bh = w >> band, h >> band
        bands.append((off, bw, bh, BAKED_STRIDE[band]))
        off += -(-bw * bh * BAKED_STRIDE[band] // 256) * 256
    return bands, off


def _texture(case, g):
    """One shell's texels: SH coefficients N(0, 0.3), RGB U(0, 1) with alpha
    U(0.2, 0.8), or baked bytes of N(0, 3.5) base values, weaker in the
    higher bands."""
    w, h, fmt, degree = case["tex_w"], case["tex_h"], case["fmt"], case["degree"]
    if fmt == BAKED:
        bands, total = _baked_bands(w, h, degree)
        buf = torch.zeros(total, dtype=torch.uint8, device="cuda")
        for band, (off, bw, bh, stride) in enumerate(bands):
            n = 4 * (2 * band + 1)
            v = torch.randn(bh, bw, n, device="cuda", generator=g) * (3.5 if band == 0 else 3.5 / (2 * band))
            q = torch.round((v + 15.0) * (255.0 / 30.0)).clamp(0, 255).to(torch.uint8)
            buf[off:off + bw * bh * stride].view(bh, bw, stride)[..., :n] = q
        return buf
    if fmt == RGBA:
        t = torch.rand(h, w, 4, device="cuda", generator=g)
        t[..., 3] = 0.2 + 0.6 * t[..., 3]
        return t
    t = torch.randn(h, w, _pitch(case), device="cuda", dtype=torch.float16, generator=g) * 0.3
    t[..., _channels(fmt, degree):] = 0
    return t


@dataclasses.dataclass
class Camera:
    world_to_cam: torch.Tensor     # [3, 4] FP32 on the host
    fx: float
    fy: float
    cx: float
    cy: float
    znear: float
    width: int
    height: int


def _cameras(n, width, height, distance, g):
    """n views of the origin from a Fibonacci lattice of the upper
    hemisphere, turned by a seeded azimuth."""
    turn = float(torch.rand(1, device="cuda", generator=g, dtype=torch.float64).item()) * 2 * math.pi
    lo, hi = math.sin(math.radians(5)), math.sin(math.radians(80))
    out = []
    for i in range(n):
        z = lo + (hi - lo) * (i + 0.5) / n
        az, rxy = turn + math.pi * (3 - math.sqrt(5)) * i, math.sqrt(1 - z * z)
        eye = torch.tensor([rxy * math.cos(az), rxy * math.sin(az), z], dtype=torch.float64) * distance
        f = -eye / eye.norm()
        right = torch.linalg.cross(f, torch.tensor([0.0, 0.0, 1.0], dtype=torch.float64))
        right = right / right.norm()
        r = torch.stack([right, torch.linalg.cross(f, right), f])
        m = torch.cat([r, -(r @ eye)[:, None]], 1).float()
        focal = float(torch.tensor(height / 2.0 / math.tan(math.radians(20.0)), dtype=torch.float32))
        out.append(Camera(m, focal, focal, width / 2.0, height / 2.0, float(torch.tensor(0.1)), width, height))
    return out


def _sizes(case):
    """(triangles of each shell, view sizes) per object."""
    if case["op"] != "uneven":
        return [([case["tris"]] * case["k"], [(case["width"], case["height"])] * case.get("views", 1))]
    out = []
    for j in range(case["objects"]):
        k = (3, 5, 7, 9)[j % 4]
        span = math.log(case["tris_hi"] / case["tris_lo"])
        tris = [int(case["tris_lo"] * math.exp(span * ((5 * j + 3 * i) % 11) / 10.0)) for i in range(k)]
        out.append((tris, [RESOLUTIONS[(j + 3 * v) % 4] for v in range(case["views"])]))
    return out


def _scenes(case, seed):
    """Per object: its shells, cameras and, per view, the target image (or,
    for autograd, the gradient of the rendered image)."""
    g = _generator(seed)
    out = []
    for tris, views in _sizes(case):
        shells = _geometry(tris, g)
        for s in shells:
            s.update(tex=_texture(case, g), fmt=case["fmt"], degree=case["degree"])
            if case["fmt"] == BAKED:
                s.update(tex_w=case["tex_w"], tex_h=case["tex_h"], band_shift=1, vmin=-15.0, vmax=15.0)
        if len(set(views)) == 1:
            cams = _cameras(len(views), *views[0], case["distance"], g)
        else:
            cams = [_cameras(1, w, h, case["distance"], g)[0] for w, h in views]
        tgt = []
        if case["op"] in ("fit", "uneven"):
            tgt = [torch.rand(h, w, 3, device="cuda", generator=g) for w, h in views]
        elif case["op"] == "autograd":
            tgt = [torch.randn(h, w, 4, device="cuda", generator=g) for w, h in views]
        out.append((shells, cams, tgt))
    return out


def _net_shapes(c):
    lf, h, o = c["levels"] * c["features"], c["hidden"], c["out_ch"]
    return [(c["levels"], 1 << c["log2_table"], c["features"]), (h, lf), (h,), (h, h), (h,), (o, h), (o,)]


def _net_inputs(case, seed):
    """Parameters of a network in training (tables grown to N(0, 0.1),
    He-normal weights, small biases) and a texel gradient."""
    g = _generator(seed)
    parts = []
    for i, shp in enumerate(_net_shapes(case)):
        n = math.prod(shp)
        sigma = 0.1 if i == 0 else math.sqrt(2.0 / shp[-1]) if len(shp) == 2 else 0.05
        parts.append(torch.randn(n, device="cuda", generator=g) * sigma)
    params = torch.cat(parts)
    if case["op"] == "adam":
        m = torch.randn(params.numel(), device="cuda", generator=g) * 1e-3
        v = (torch.randn(params.numel(), device="cuda", generator=g) * 1e-3) ** 2
        return params, torch.randn(params.numel(), device="cuda", generator=g) * 1e-3, m, v
    grad = None
    if case["op"] != "net_forward":
        grad = torch.randn(case["tex_h"], case["tex_w"], _net_pitch(case), device="cuda", generator=g)
    return params, grad, None, None


def _net_pitch(case):
    return -(-case["out_ch"] // 4) * 4


# ----------------------------------------------------------------------------
# prepare and run
# ----------------------------------------------------------------------------

_context = []


def _ctx():
    if not _context:
        _context.append(vs.Context(0))
    return _context[0]


def _flags(case):
    f = vs.VS_FLAG_ALPHA_ATTEN if case["atten"] else 0
    return f | {None: 0, "l1": vs.VS_FLAG_LOSS_L1, "l2": vs.VS_FLAG_LOSS_L2}[case.get("loss")]


def prepare(case, seed):
    ctx = _ctx()
    op = case["op"]
    if op.startswith("net") or op == "adam":
        nt = vs.NeuralTexture(ctx, levels=case["levels"], features=case["features"], log2_table=case["log2_table"],
                              base_res=case["base_res"], growth=case["growth"], hidden=case["hidden"],
                              out_ch=case["out_ch"], tex_w=case["tex_w"], tex_h=case["tex_h"],
                              tensor_cores=case["tensor_cores"])
        params, grad, m, v = _net_inputs(case, seed)
        nt.params.copy_(params)
        s = dict(op=op, net=nt, grad=grad)
        if op == "adam":
            nt.grads.copy_(grad)
            nt.m.copy_(m)
            nt.v.copy_(v)
            nt.step = ADAM_STEP
        elif op != "net_backward":
            s["tex"] = torch.zeros(case["tex_h"], case["tex_w"], _net_pitch(case), device="cuda",
                                   dtype=torch.float16 if case["half"] else torch.float32)
        return s
    flags = _flags(case)
    scenes = [(vs.ShellObject(ctx, shells), cams, tgt) for shells, cams, tgt in _scenes(case, seed)]
    objs = [o for o, cams, _ in scenes for _ in cams]
    cams = [c for _, cs, _ in scenes for c in cs]
    s = dict(op=op, ctx=ctx, flags=flags, ws=vs.make_workspace(ctx, objs, cams, flags), scenes=scenes)
    if op in ("frame", "autograd"):
        s.update(obj=objs[0], cam=cams[0])
        if op == "autograd":
            s.update(up=scenes[0][2][0], textures=[t.requires_grad_() for t in objs[0].textures])
        return s
    s["outs"] = [torch.empty(c.height, c.width, 4, device="cuda") for c in cams]
    items = [dict(obj=o, cam=c, out=t) for o, c, t in zip(objs, cams, s["outs"])]
    if op == "views":
        s["hits"] = [torch.empty(o.k, c.height, c.width, dtype=torch.int32, device="cuda")
                     for o, c in zip(objs, cams)]
        for it, h in zip(items, s["hits"]):
            it["hits"] = h
    else:
        s["loss"] = torch.zeros(len(items), device="cuda")
        # one buffer for the gradients of all shells, cleared by one fill a step
        shapes = [sh for o, _, _ in scenes for sh in o.grad_shapes()]
        s["flat"] = torch.zeros(sum(math.prod(sh) for sh in shapes), device="cuda")
        s["grads"] = [p.view(sh) for p, sh in zip(s["flat"].split([math.prod(sh) for sh in shapes]), shapes)]
        first, at = {}, 0
        for o, _, _ in scenes:
            first[id(o)], at = at, at + o.k
        targets = [t for _, _, ts in scenes for t in ts]
        for j, it in enumerate(items):
            a = first[id(it["obj"])]
            it.update(grad_rgb=targets[j], grads=s["grads"][a:a + it["obj"].k], loss=s["loss"][j:j + 1])
    s["items"] = vs.BatchItems(items)
    return s


def run(state):
    s = state
    op = s["op"]
    if op == "frame":
        return vs.render(s["ctx"], s["obj"], s["cam"], s["ws"], bg=BACKGROUND, flags=s["flags"])
    if op == "autograd":
        out = vs.VSRender.apply(s["ctx"], s["obj"], s["cam"], s["ws"], BACKGROUND, s["flags"], *s["textures"])
        return [out.detach()] + list(torch.autograd.grad(out, s["textures"], s["up"]))
    if op == "views":
        vs.render_batch(s["ctx"], s["items"], s["ws"], bg=BACKGROUND, flags=s["flags"])
        return dict(rgba=s["outs"], hits=s["hits"])
    if op in ("fit", "uneven"):
        s["flat"].zero_()
        s["loss"].zero_()
        vs.render_batch(s["ctx"], s["items"], s["ws"], bg=BACKGROUND, do_backward=True, flags=s["flags"])
        return dict(rgba=s["outs"], loss=s["loss"], grads=s["flat"])
    nt = s["net"]
    if op == "adam":
        nt.adam(LR, BETA1, BETA2, EPS)
        return [nt.params, nt.m, nt.v]
    out = {}
    if op in ("net_forward", "net_both"):
        nt.forward(s["tex"])
        out["texels"] = s["tex"]
    if op in ("net_backward", "net_both"):
        nt.grads.zero_()
        nt.backward(s["grad"])
        out["grads"] = nt.grads
    return out


# ----------------------------------------------------------------------------
# the work of a pass
# ----------------------------------------------------------------------------

def _fragments(k, w, h, distance):
    """Expected (pixel, shell) hits of one view: the discs of k spheres of
    mean radius 1 - 0.01 (k - 1) in a 40 degree field of view."""
    r = 1.0 - 0.01 * (k - 1)
    radius = math.tan(math.asin(r / distance)) / (2 * math.tan(math.radians(20.0))) * h
    return k * min(math.pi * radius * radius, float(w * h))


def work(case):
    op = case["op"]
    if op.startswith("net") or op == "adam":
        n, shapes = case["tex_w"] * case["tex_h"], _net_shapes(case)
        count = sum(math.prod(s) for s in shapes)
        lf, hd, c = shapes[1][1], case["hidden"], case["out_ch"]
        if op == "adam":
            return dict(bytes=28 * count, flops=12 * count)
        layers = lf * hd + hd * hd + hd * c
        fwd, enc = n * (2 * layers + 8 * lf), n * 8 * lf
        texel = n * c * (2 if case.get("half") else 4)
        if op == "net_forward":
            return dict(bytes=4 * count + texel, flops=fwd)
        bwd = n * (2 * (lf * hd + hd * hd) + 8 * lf + 4 * layers) + enc
        back = dict(bytes=4 * count + 4 * n * c + 4 * count, flops=bwd)
        if op == "net_backward":
            return back
        return dict(bytes=back["bytes"] + 4 * count + texel, flops=back["flops"] + fwd)
    fmt, deg, texels = case["fmt"], case["degree"], case["tex_w"] * case["tex_h"]
    c = 4 * (deg + 1) ** 2 if fmt == BAKED else _channels(fmt, deg)
    size = 4 if fmt == RGBA else 2 if fmt == SH else 1
    bwd = op in ("autograd", "fit", "uneven")
    nbytes = flops = 0.0
    for tris, views in _sizes(case):
        frags = [_fragments(len(tris), w, h, case["distance"]) for w, h in views]
        pixels = sum(w * h for w, h in views)
        # texels seen: up to four per fragment, half a closed surface per view
        seen = min(texels * len(tris), sum(min(4 * f, 0.5 * texels * len(tris)) for f in frags))
        verts = sum(0.5 * t for t in tris)
        nbytes += 20 * verts + 12 * sum(tris) + seen * c * size + 16 * pixels
        flops += len(views) * (30 * verts + 60 * sum(tris)) + sum(frags) * (10 * c + 150)
        if op in ("frame", "views"):
            nbytes += 4 * len(tris) * pixels
        if bwd:
            flops += sum(frags) * (10 * c + 100)
            nbytes += 12 * pixels + texels * len(tris) * (_pitch(case) if fmt != RGBA else 4) * (
                2 if op == "autograd" and fmt == SH else 4)
    return dict(bytes=nbytes, flops=flops)


# ----------------------------------------------------------------------------
# the same in 64 bits
# ----------------------------------------------------------------------------

def _hits(s, cam):
    """Nearest front-facing triangle of one shell at every pixel, -1 = none.
    The method's own definition: a vertex transform in single roundings
    (each torch operation rounds once), positions snapped to 1/256 pixel,
    integer edge functions with the top-left rule, and an integer depth key
    whose ties go to the lower triangle."""
    m = cam.world_to_cam.reshape(-1).tolist()
    x, y, z = s["pos"].unbind(1)

    def row(a):
        return ((x * m[a] + y * m[a + 1]) + z * m[a + 2]) + m[a + 3]

    xc, yc, zc = row(0), row(4), row(8)
    iw = 1.0 / zc
    X = torch.round(((xc * cam.fx) * iw + cam.cx) * 256.0).long()
    Y = torch.round(((yc * cam.fy) * iw + cam.cy) * 256.0).long()
    scale = float(torch.tensor(cam.znear) * 1073741824.0)
    q = torch.round(iw * scale).long()
    tri = s["tris"].long()
    W, H = cam.width, cam.height
    X, Y, q = X[tri], Y[tri], q[tri]
    area = (X[:, 1] - X[:, 0]) * (Y[:, 2] - Y[:, 0]) - (X[:, 2] - X[:, 0]) * (Y[:, 1] - Y[:, 0])
    xlo = (-((128 - X.amin(1)) >> 8)).clamp(min=0)
    xhi = ((X.amax(1) - 128) >> 8).clamp(max=W - 1)
    ylo = (-((128 - Y.amin(1)) >> 8)).clamp(min=0)
    yhi = ((Y.amax(1) - 128) >> 8).clamp(max=H - 1)
    bw, bh = (xhi - xlo + 1).clamp(min=0), (yhi - ylo + 1).clamp(min=0)
    n = torch.where(area < 0, bw * bh, 0)
    ids = n.nonzero()[:, 0]
    best = torch.zeros(H * W, dtype=torch.int64, device="cuda")
    ends = n[ids].cumsum(0)
    done, total, step = 0, int(ends[-1]) if len(ids) else 0, 1 << 25
    lo = 0
    while done < total:
        hi = max(lo + 1, int(torch.searchsorted(ends, done + step, right=True)))
        t = ids[lo:hi]
        cnt = n[t]
        rep = torch.repeat_interleave(torch.arange(len(t), device="cuda"), cnt)
        local = torch.arange(len(rep), device="cuda") - (cnt.cumsum(0) - cnt)[rep]
        t = t[rep]
        px, py = xlo[t] + local % bw[t], ylo[t] + local // bw[t]
        e, inside = [], torch.ones(len(t), dtype=torch.bool, device="cuda")
        for j in range(3):
            a, b = (j + 2) % 3, (j + 1) % 3
            xa, ya = X[t, a], Y[t, a]
            dx, dy = X[t, b] - xa, Y[t, b] - ya
            ej = dx * (256 * py + 128 - ya) - dy * (256 * px + 128 - xa)
            inside &= (ej > 0) | ((ej == 0) & ((dy < 0) | ((dy == 0) & (dx > 0))))
            e.append(ej)
        t, pix = t[inside], (py * W + px)[inside]
        e = [v[inside] for v in e]
        depth = (e[0] * q[t, 0] + e[1] * q[t, 1] + e[2] * q[t, 2]) // (e[0] + e[1] + e[2])
        best.scatter_reduce_(0, pix, (depth << 32) | (0xFFFFFFFF - t), "amax")
        done, lo = int(ends[hi - 1]), hi
    return torch.where(best > 0, 0xFFFFFFFF - (best & 0xFFFFFFFF), -1), X, Y, iw[tri]


def _basis(degree, v):
    """Real orthonormal spherical harmonics up to degree 3, [n, (d + 1)^2]."""
    x, y, z = v.unbind(1)
    xx, yy, zz, pi = x * x, y * y, z * z, math.pi
    out = [torch.full_like(x, 0.5 / math.sqrt(pi))]
    if degree >= 1:
        a = math.sqrt(3 / (4 * pi))
        out += [a * y, a * z, a * x]
    if degree >= 2:
        a, b, c = math.sqrt(15 / pi) / 2, math.sqrt(5 / pi) / 4, math.sqrt(15 / pi) / 4
        out += [a * x * y, a * y * z, b * (2 * zz - xx - yy), a * x * z, c * (xx - yy)]
    if degree >= 3:
        a, b, c, d = (math.sqrt(35 / (2 * pi)) / 4, math.sqrt(105 / pi) / 2, math.sqrt(21 / (2 * pi)) / 4,
                      math.sqrt(7 / pi) / 4)
        out += [a * y * (3 * xx - yy), b * x * y * z, c * y * (4 * zz - xx - yy),
                d * z * (2 * zz - 3 * xx - 3 * yy), c * x * (4 * zz - xx - yy), b / 2 * z * (xx - yy),
                a * x * (xx - 3 * yy)]
    return torch.stack(out, 1)


def _taps(x, y, w, h):
    """Bilinear taps of texel coordinates (x, y): [(texel, weight)] * 4."""
    ix, iy = x.floor(), y.floor()
    fx, fy = x - ix, y - iy
    xs = [ix.long().clamp(0, w - 1), (ix.long() + 1).clamp(0, w - 1)]
    ys = [iy.long().clamp(0, h - 1), (iy.long() + 1).clamp(0, h - 1)]
    return [(ys[b] * w + xs[a], (fx if a else 1 - fx) * (fy if b else 1 - fy)) for b in (0, 1) for a in (0, 1)]


def _texels(s, case, x, y):
    """Bilinear values [n, channels] at texel coordinates, and their taps."""
    if case["fmt"] == BAKED:
        vals = []
        bands, _ = _baked_bands(case["tex_w"], case["tex_h"], case["degree"])
        for band, (off, bw, bh, stride) in enumerate(bands):
            img = s["tex"][off:off + bw * bh * stride].view(-1, stride)[:, :4 * (2 * band + 1)]
            taps = _taps((x + 0.5) / 2 ** band - 0.5, (y + 0.5) / 2 ** band - 0.5, bw, bh)
            vals.append(sum(img[i].double() * w[:, None] for i, w in taps) * (30.0 / 255.0) - 15.0)
        return torch.cat(vals, 1), None
    taps = _taps(x, y, case["tex_w"], case["tex_h"])
    img = s["tex"].detach().view(case["tex_w"] * case["tex_h"], -1)[:, :_channels(case["fmt"], case["degree"])]
    return sum(img[i].double() * w[:, None] for i, w in taps), taps


def _render64(case, shells, cam, up, grads):
    """(rgba [H, W, 4], loss) of one view; adds the texel gradients to
    `grads` when given (up: target image or gradient of the image)."""
    W, H, f64 = cam.width, cam.height, torch.float64
    m = cam.world_to_cam.double().cuda()
    pix = torch.arange(H * W, device="cuda")
    a, b = (pix % W + 0.5 - cam.cx) / cam.fx, (pix // W + 0.5 - cam.cy) / cam.fy
    ray = torch.stack([a, b, torch.ones_like(a)], 1).double() @ m[:, :3]
    ray = ray / ray.norm(dim=1, keepdim=True)
    layers = []
    C, T = torch.zeros(H * W, 3, device="cuda", dtype=f64), torch.ones(H * W, device="cuda", dtype=f64)
    for s in shells:
        hit, X, Y, iw = _hits(s, cam)
        p = (hit >= 0).nonzero()[:, 0]
        t = hit[p]
        px, py = 256 * (p % W) + 128, 256 * (p // W) + 128
        w = []
        for j in range(3):
            i, o = (j + 2) % 3, (j + 1) % 3
            w.append(((X[t, o] - X[t, i]) * (py - Y[t, i]) - (Y[t, o] - Y[t, i]) * (px - X[t, i])).double()
                     * iw[t, j].double())
        den = w[0] + w[1] + w[2]
        uv = s["uv"].double()[s["tris"].long()[t]]
        at = uv[:, 0] + (w[1] / den)[:, None] * (uv[:, 1] - uv[:, 0]) + (w[2] / den)[:, None] * (uv[:, 2] - uv[:, 0])
        val, taps = _texels(s, case, at[:, 0] * case["tex_w"] - 0.5, at[:, 1] * case["tex_h"] - 0.5)
        Yb = _basis(case["degree"], ray[p])
        if case["fmt"] == RGBA:
            rgb, alpha = val[:, :3], val[:, 3]
        elif case["fmt"] == SH:
            rgb = torch.sigmoid(torch.einsum("nmc,nm->nc", val[:, 1:].view(len(p), -1, 3), Yb))
            alpha = torch.sigmoid(val[:, 0])
        else:
            z = torch.sigmoid(torch.einsum("nmc,nm->nc", val.view(len(p), -1, 4), Yb))
            rgb, alpha = z[:, :3], z[:, 3]
        del val
        aw = torch.ones_like(alpha)
        if case["atten"]:
            v = s["pos"].double()[s["tris"].long()[t]]
            nrm = torch.linalg.cross(v[:, 1] - v[:, 0], v[:, 2] - v[:, 0])
            nrm = nrm / nrm.norm(dim=1, keepdim=True)
            aw = 2 * torch.sigmoid(10 * (nrm * ray[p]).sum(1).abs()) - 1
        Tp = T[p]
        C[p] += (Tp * aw * alpha)[:, None] * rgb
        T[p] = Tp * (1 - aw * alpha)
        layers.append((p, taps, Yb, rgb, alpha, aw, Tp) if grads is not None else None)
    bg = torch.tensor(BACKGROUND, dtype=torch.float32).double().cuda()
    image = C + T[:, None] * bg
    out = torch.cat([image, 1 - T[:, None]], 1).view(H, W, 4)
    if grads is None:
        return out, None
    up, loss = up.double().view(H * W, -1), None
    if case.get("loss"):
        d = image - up
        loss = (d.square() if case["loss"] == "l2" else d.abs()).mean()
        up = (2 * d if case["loss"] == "l2" else d.sign()) / (3 * H * W)
    up = up[:, :3]
    behind = (up * bg).sum(1)
    for (p, taps, Yb, rgb, alpha, aw, Tp), g in reversed(list(zip(layers, grads))):
        a, u = aw * alpha, up[p]
        seen = (rgb * u).sum(1)
        d_rgb, d_a = (Tp * a)[:, None] * u, Tp * (seen - behind[p]) * aw
        behind[p] += a * (seen - behind[p])
        if case["fmt"] == RGBA:
            d = torch.cat([d_rgb, d_a[:, None]], 1)
        else:
            d_rgb = d_rgb * rgb * (1 - rgb)
            d = torch.cat([(d_a * alpha * (1 - alpha))[:, None],
                           (Yb[:, :, None] * d_rgb[:, None, :]).reshape(len(p), -1)], 1)
        flat = g.view(case["tex_w"] * case["tex_h"], -1)
        for i, w in taps:
            add = torch.zeros(len(p), flat.shape[1], dtype=f64, device="cuda")
            add[:, :d.shape[1]] = d * w[:, None]
            flat.index_add_(0, i, add)
    return out, loss


def _encode64(case, params, n0, n1):
    """Table rows, weights and features of texels [n0, n1): per level the
    four lattice corners."""
    W, H, F, T = case["tex_w"], case["tex_h"], case["features"], 1 << case["log2_table"]
    n = torch.arange(n0, n1, device="cuda")
    tx, ty = n % W, n // W
    table = params[:case["levels"] * T * F].view(case["levels"], T, F)
    rows, feats = [], []
    for lv in range(case["levels"]):
        res = int(math.floor(case["base_res"] * float(torch.tensor(case["growth"])) ** lv))
        nx, ny = (2 * tx + 1) * res, (2 * ty + 1) * res
        cx, cy = nx // (2 * W), ny // (2 * H)
        rx, ry = (nx - cx * 2 * W).double() / (2 * W), (ny - cy * 2 * H).double() / (2 * H)
        corner = []
        for dy in (0, 1):
            for dx in (0, 1):
                c0, c1 = cx + dx, cy + dy
                row = c0 + c1 * (res + 1) if (res + 1) ** 2 <= T else (c0 ^ ((c1 * PRIME) & 0xFFFFFFFF)) & (T - 1)
                corner.append((row, (rx if dx else 1 - rx) * (ry if dy else 1 - ry)))
        rows.append(corner)
        feats.append(sum(table[lv][r] * w[:, None] for r, w in corner))
    return rows, torch.cat(feats, 1)


def _net64(case, seed):
    params, grad, m, v = _net_inputs(case, seed)
    if case["op"] == "adam":
        b1, b2, eps, lr = (float(torch.tensor(x)) for x in (BETA1, BETA2, EPS, LR))
        g, step = grad.double(), ADAM_STEP + 1
        m = b1 * m.double() + (1 - b1) * g
        v = b2 * v.double() + (1 - b2) * g * g
        return [params.double() - lr * (m / (1 - b1 ** step)) / ((v / (1 - b2 ** step)).sqrt() + eps), m, v]
    params = params.double()
    shapes = _net_shapes(case)
    parts = [p.view(s) for p, s in zip(params.split([math.prod(s) for s in shapes]), shapes)]
    _, W0, b0, W1, b1, W2, b2 = parts
    N, C, T = case["tex_w"] * case["tex_h"], case["out_ch"], 1 << case["log2_table"]
    out, total = {}, torch.zeros_like(params)
    sums = [p.view(s) for p, s in zip(total.split([math.prod(s) for s in shapes]), shapes)]
    tex = torch.zeros(N, _net_pitch(case), dtype=torch.float64, device="cuda")
    for n0 in range(0, N, 1 << 18):
        n1 = min(N, n0 + (1 << 18))
        rows, X = _encode64(case, params, n0, n1)
        H1 = torch.relu(X @ W0.T + b0)
        H2 = torch.relu(H1 @ W1.T + b1)
        if case["op"] != "net_backward":
            tex[n0:n1, :C] = H2 @ W2.T + b2
        if case["op"] == "net_forward":
            continue
        dY = grad.view(N, -1)[n0:n1, :C].double()
        d2 = (dY @ W2) * (H2 > 0)
        d1 = (d2 @ W1) * (H1 > 0)
        for q, t in ((1, d1.T @ X), (2, d1.sum(0)), (3, d2.T @ H1), (4, d2.sum(0)), (5, dY.T @ H2), (6, dY.sum(0))):
            sums[q] += t
        dX = (d1 @ W0).view(n1 - n0, case["levels"], case["features"])
        for lv, corner in enumerate(rows):
            for r, w in corner:
                sums[0][lv].index_add_(0, r, dX[:, lv] * w[:, None])
    if case["op"] != "net_backward":
        out["texels"] = tex.view(case["tex_h"], case["tex_w"], -1)
    if case["op"] != "net_forward":
        out["grads"] = total
    return out


def exact(case, seed):
    op = case["op"]
    if op.startswith("net") or op == "adam":
        return _net64(case, seed)
    scenes = _scenes(case, seed)
    bwd = op in ("autograd", "fit", "uneven")
    if op == "autograd":
        grads = [[torch.zeros(s["tex"].shape, dtype=torch.float64, device="cuda") for s in shells]
                 for shells, _, _ in scenes]
    else:
        # gradients have the texels' pitch; one buffer, as run() returns it
        shape = (case["tex_h"], case["tex_w"], _pitch(case) if case["fmt"] != BAKED else 0)
        size = math.prod(shape)
        flat = torch.zeros(sum(len(sh) for sh, _, _ in scenes) * size if bwd else 0, dtype=torch.float64, device="cuda")
        parts = iter(flat.split(size)) if bwd else None
        grads = [[next(parts).view(shape) for _ in sh] if bwd else None for sh, _, _ in scenes]
    outs, losses = [], []
    for (shells, cams, tgt), g in zip(scenes, grads):
        for i, cam in enumerate(cams):
            o, loss = _render64(case, shells, cam, tgt[i] if tgt else None, g)
            outs.append(o)
            losses.append(loss)
    if op == "frame":
        return outs[0], None
    if op == "autograd":
        return [outs[0]] + grads[0]
    if op == "views":
        return dict(rgba=outs, hits=None)
    return dict(rgba=outs, loss=torch.stack(losses), grads=flat)
