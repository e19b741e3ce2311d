"""Performance cases of the texture filtering library: what a renderer has it do.

Each case is one pass through the public entry points of ``paper_2305_05810_gb300``
on inputs made on the GPU from a seed: ray-march samples of dense and sparse density
grids, texture lookups of images and material sets, anisotropic filtering of a ground
plane, and decoding and training of a neural texture; each in the stochastic and the
deterministic form.  ``exact`` gives the same outputs in 64 bits with plain torch.
"""
import math

import torch
import torch.nn.functional as nnf

import paper_2305_05810_gb300 as stf

MAX_ANISOTROPY = 16.0
DEV = "cuda"

# ---------------------------------------------------------------- cases


def listed():
    return [
        # a volume renderer's frame: 1080p rays x 16 steps through a fog density, one texel
        # per sample (the default benchmark workload)
        dict(name="dense_march", kind="dense", grid=256, fmt="f16", filter="bspline3",
             form="stochastic", width=1920, height=1080, steps=16),
        # the same renderer's reference frame at quarter resolution: the whole 64-tap filter
        dict(name="dense_march_full", kind="dense", grid=256, fmt="f16", filter="bspline3",
             form="deterministic", width=960, height=540, steps=16),
        # a cloud in a sparse grid, most samples in empty space
        dict(name="sparse_march", kind="sparse", domain=2048, fmt="f32", filter="bspline3",
             form="stochastic", width=1024, height=1024, steps=16),
        # the same cloud with 8-bit leaves, whole filter
        dict(name="sparse_march_full", kind="sparse", domain=2048, fmt="e4m3", filter="bspline3",
             form="deterministic", width=1024, height=1024, steps=16),
        # one small batch of shading points: latency
        dict(name="image_small", kind="image", tex_w=256, tex_h=256, channels=4, fmt="f32", levels=1,
             filter="bspline3", form="stochastic", queries=65536),
        # bicubic resampling of an image, a ragged number of points
        dict(name="image_bicubic", kind="image", tex_w=256, tex_h=256, channels=4, fmt="f32", levels=1,
             filter="bspline3", form="deterministic", queries=4194301),
        # a 4K frame of a ground plane with a DCT-compressed 8-channel material set,
        # level of detail from the screen-space derivatives, trilinear
        dict(name="dct_view", kind="view", tex_w=4096, tex_h=4096, channels=8, fmt="dct", levels=13,
             filter="linear", form="deterministic", width=3840, height=2160),
        # a 4K frame of a ground plane with an RGBA image: elliptical footprints
        dict(name="ewa_view", kind="ewa", tex_w=1024, tex_h=1024, channels=4, fmt="f16", levels=11,
             form="stochastic", width=3840, height=2160),
        dict(name="ewa_view_full", kind="ewa", tex_w=1024, tex_h=1024, channels=4, fmt="f16", levels=11,
             form="deterministic", width=3840, height=2160),
        # shading points on a neural material: one decode each, or every bilinear tap
        dict(name="neural", kind="neural", size=4096, filter="linear", form="stochastic",
             queries=1 << 24),
        dict(name="neural_full", kind="neural", size=4096, filter="linear", form="deterministic",
             queries=1 << 22),
        # one training batch of the neural material: loss and gradients
        dict(name="neural_gradients", kind="gradients", size=1024, batch=65536),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["dense", "sparse", "image", "view", "ewa", "neural", "gradients"])
    form = rng.choice(["stochastic", "deterministic"])
    filt = rng.choice(["linear", "bspline3", "bspline3", "catmull_rom"])
    if kind in ("dense", "sparse"):
        # rays from a thumbnail to a full frame (a quarter of it for the whole filter)
        rays = _log(rng, 64, 1920 * 1080 if form == "stochastic" else 960 * 540)
        width = max(1, int(math.sqrt(rays * rng.uniform(0.5, 2.0))))
        c = dict(kind=kind, filter=filt, form=form, width=width, height=max(1, rays // width),
                 steps=rng.choice([8, 13, 16]))
        if kind == "dense":
            return dict(c, grid=_log(rng, 64, 256), fmt=rng.choice(["f16", "f16", "f32"]))
        return dict(c, domain=rng.choice([512, 1024, 2048]), fmt=rng.choice(["f32", "e4m3"]))
    if kind == "image":
        fmt = rng.choice(["f32", "f16", "dct"])
        channels = rng.choice([1, 2, 4, 4, 8])
        if rng.random() < 0.5:                       # any size, no pyramid
            w, h, levels = _log(rng, 63, 2048), _log(rng, 63, 2048), 1
        else:
            side = rng.choice([6, 8, 10, 11])
            w, h, levels = 1 << side, 1 << side, side + 1
        top = {1: 1 << 24, 2: 1 << 23, 4: 1 << 22, 8: 1 << 21}[channels]
        return dict(kind=kind, tex_w=w, tex_h=h, channels=channels, fmt=fmt, levels=levels, filter=filt,
                    form=form, queries=_log(rng, 4099, top))
    if kind in ("view", "ewa"):
        side = rng.choice([9, 10, 11])
        height = _log(rng, 135, 2160)
        c = dict(kind=kind, tex_w=1 << side, tex_h=1 << side, levels=side + 1, form=form,
                 width=height * 16 // 9 + rng.choice([0, 1, 3]), height=height)
        if kind == "ewa":
            return dict(c, channels=rng.choice([1, 4]), fmt=rng.choice(["f16", "f32"]))
        return dict(c, channels=rng.choice([4, 8]), fmt=rng.choice(["f16", "dct"]),
                    filter=rng.choice(["linear", "bspline3"]))
    if kind == "neural":
        filt = rng.choice(["linear", "linear", "bspline3"])
        top = 1 << 24 if form == "stochastic" else 1 << 22 if filt == "linear" else 1 << 20
        return dict(kind=kind, size=rng.choice([512, 1024, 2048]), filter=filt, form=form,
                    queries=_log(rng, 1031, top))
    return dict(kind=kind, size=rng.choice([256, 512, 1024]), batch=32 * _log(rng, 8, 2048))


# ---------------------------------------------------------------- inputs


def _generator(seed, what):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * int(seed) + what)
    return g


def _noise(shape, channels, g, octaves=4, cells=8):
    """Fractal value noise in [0, 1], (channels, *shape): `cells` lattice cells along each
    axis in the first octave, twice as many and half the amplitude in each further one."""
    mode = "bilinear" if len(shape) == 2 else "trilinear"
    out = torch.zeros((channels, *shape), device=DEV)
    for o in range(octaves):
        lattice = torch.rand((1, channels) + (cells << o,) * len(shape), generator=g, device=DEV)
        out += 0.5 ** o * nnf.interpolate(lattice, size=shape, mode=mode, align_corners=False)[0]
    flat = out.reshape(channels, -1)
    lo, hi = flat.min(1, keepdim=True)[0], flat.max(1, keepdim=True)[0]
    return ((flat - lo) / (hi - lo)).reshape(out.shape)


def _threshold(v, share):
    """The value above which `share` of v lies (from at most 2^20 of its values)."""
    flat = v.reshape(-1)
    return torch.quantile(flat[:: max(1, flat.numel() >> 20)][: 1 << 20].float(), 1.0 - share)


def _density(n, g):
    """(z, y, x) density: 30% of the voxels are not empty."""
    v = _noise((n, n, n), 1, g, octaves=5, cells=5)[0]
    t = _threshold(v, 0.3)
    return (v - t).clamp_min(0) / (1 - t)


def _cloud(domain, g):
    """Leaf origins (L, 3) and values (L, 512): 4% of the 8^3 cells, clustered like a cloud."""
    n = domain // 8
    v = _noise((n, n, n), 1, g, octaves=4, cells=6)[0]
    a = (torch.arange(n, device=DEV) + 0.5) / n * 2 - 1
    r = (a[:, None, None] ** 2 + a[None, :, None] ** 2 + a[None, None, :] ** 2).sqrt()
    v = v * (1 - r).clamp_min(0)
    origins = (v > _threshold(v, 0.04)).nonzero().flip(1) * 8
    corner = torch.rand((origins.shape[0], 1, 3, 3, 3), generator=g, device=DEV)
    values = nnf.interpolate(corner, size=(8, 8, 8), mode="trilinear", align_corners=True)
    return origins.to(torch.int32).contiguous(), (0.05 + 0.95 * values).reshape(-1, 512).contiguous()


def _rays(extent, case, g):
    """Samples of a pinhole camera's rays through a cube, ray-major, jittered steps."""
    w, h, steps = case["width"], case["height"], case["steps"]
    opt = dict(dtype=torch.float64, device=DEV)
    d = nnf.normalize(torch.randn(3, generator=g, **opt), dim=0)
    up = torch.tensor([0.0, 0.0, 1.0] if abs(float(d[2])) < 0.99 else [0.0, 1.0, 0.0], **opt)
    right = nnf.normalize(torch.linalg.cross(d, up), dim=0)
    t = math.tan(math.radians(20.0))
    sx = ((torch.arange(w, **opt) + 0.5) / w * 2 - 1) * t * w / h
    sy = (1 - (torch.arange(h, **opt) + 0.5) / h * 2) * t
    ray = d + sx[None, :, None] * right + sy[:, None, None] * torch.linalg.cross(right, d)
    ray = nnf.normalize(ray, dim=2).reshape(-1, 1, 3)
    radius, span = 1.5 * extent, 0.867 * extent
    s = torch.arange(steps, **opt) + torch.rand((w * h, steps), generator=g, **opt)
    s = radius - span + s * (2 * span / steps)
    return (extent / 2 - radius * d + s[..., None] * ray).reshape(-1, 3).float()


PITCH, EYE_HEIGHT, FAR = math.radians(12.0), 0.04, 1.0


def _view_rows(height):
    """The pixel rows of a view that see the ground plane nearer than FAR."""
    t = math.tan(math.radians(30.0)) * math.cos(PITCH)
    return [y for y in range(height)
            if math.sin(PITCH) - (1 - 2 * (y + 0.5) / height) * t >= EYE_HEIGHT / FAR]


def _plane_view(case, g):
    """(u, v) and its screen derivatives for the pixels of a camera above a ground plane that
    the texture tiles."""
    w, h = case["width"], case["height"]
    opt = dict(dtype=torch.float64, device=DEV)
    eye = torch.rand(2, generator=g, **opt)
    yaw = float(torch.rand(1, generator=g, **opt)) * 2 * math.pi
    fwd = torch.tensor([math.sin(yaw) * math.cos(PITCH), math.cos(yaw) * math.cos(PITCH)], **opt)
    right = torch.tensor([math.cos(yaw), -math.sin(yaw)], **opt)
    up = torch.tensor([math.sin(yaw) * math.sin(PITCH), math.cos(yaw) * math.sin(PITCH)], **opt)
    t = math.tan(math.radians(30.0))

    def hit(x, y):
        sx, sy = (2 * (x + 0.5) / w - 1) * t * w / h, (1 - 2 * (y + 0.5) / h) * t
        reach = EYE_HEIGHT / (math.sin(PITCH) - sy * math.cos(PITCH))
        return eye + reach[:, None] * (fwd + sx[:, None] * right + sy[:, None] * up)

    rows = torch.tensor(_view_rows(h), **opt)
    y, x = rows.repeat_interleave(w), torch.arange(w, **opt).repeat(rows.numel())
    p = hit(x, y)
    grad = torch.cat([hit(x + 1, y) - p, hit(x, y + 1) - p], 1)
    return (p - p.floor()).float().contiguous(), grad.float().contiguous()


NEURAL_LEVELS = 4


def _neural_weights(size, g):
    n = sum((size >> k) ** 2 for k in range(NEURAL_LEVELS))
    latents = 0.5 * torch.randn((n, 8), generator=g, device=DEV)
    parts = []
    for fan_in, fan_out in ((8, 64), (64, 64), (64, 7)):
        parts.append(torch.randn(fan_in * fan_out, generator=g, device=DEV) * math.sqrt(2.0 / fan_in))
        parts.append(0.1 * torch.randn(fan_out, generator=g, device=DEV))
    fallback = torch.rand((sum(max(1, size >> k) ** 2 for k in range(NEURAL_LEVELS, _neural_levels(size))), 7),
                          generator=g, device=DEV)
    return latents, torch.cat(parts), fallback


def _neural_levels(size):
    return size.bit_length()


def _inputs(case, seed):
    """The case's tensors: texels and queries."""
    kind = case["kind"]
    gt, gq = _generator(seed, 1), _generator(seed, 2)
    s = {}
    if kind == "dense":
        s["values"] = _density(case["grid"], gt)
        s["coords"] = _rays(case["grid"], case, gq)
    elif kind == "sparse":
        s["origins"], s["values"] = _cloud(case["domain"], gt)
        s["coords"] = _rays(case["domain"], case, gq)
    elif kind in ("neural", "gradients"):
        s["latents"], s["params"], s["fallback"] = _neural_weights(case["size"], gt)
        if kind == "neural":
            s["coords"] = torch.rand((case["queries"], 2), generator=gq, device=DEV)
            s["lod"] = 4 * torch.rand(case["queries"], generator=gq, device=DEV)
        else:
            s["texels"] = torch.randint(s["latents"].shape[0], (case["batch"],), generator=gq, device=DEV)
            s["targets"] = torch.rand((case["batch"], 7), generator=gq, device=DEV)
    else:
        w, h = case["tex_w"], case["tex_h"]
        s["values"] = _noise((h, w), case["channels"], gt).permute(1, 2, 0).contiguous()
        if kind == "image":
            s["coords"] = torch.rand((case["queries"], 2), generator=gq, device=DEV)
            if case["levels"] > 1:
                s["lod"] = (case["levels"] - 1) * torch.rand(case["queries"], generator=gq, device=DEV)
        else:
            s["coords"], s["grad"] = _plane_view(case, gq)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    if kind == "dense":
        s["texture"] = stf.Texture(stf.KIND_DENSE3D, s["values"], dims=(case["grid"],) * 3,
                                   fmt=stf.FMT_F16 if case["fmt"] == "f16" else stf.FMT_F32)
    elif kind == "sparse":
        s["texture"] = stf.Texture(stf.KIND_SPARSE3D, s["values"], leaf_origins=s["origins"],
                                   fmt=stf.FMT_F32 if case["fmt"] == "f32" else stf.FMT_E4M3_SCALED)
    elif kind in ("neural", "gradients"):
        s["texture"] = stf.NeuralTexture(case["size"], case["size"], NEURAL_LEVELS,
                                         _neural_levels(case["size"]), s["latents"], s["params"], s["fallback"])
    else:
        fmt = {"f32": stf.FMT_F32, "f16": stf.FMT_F16, "dct": stf.FMT_DCT6}[case["fmt"]]
        s["texture"] = stf.Texture(stf.KIND_TEX2D, s["values"], dims=(case["tex_w"], case["tex_h"], 1),
                                   channels=case["channels"], fmt=fmt, mip_levels=case["levels"],
                                   generate_mips=case["levels"] > 1)
    for k in ("values", "origins", "latents", "params", "fallback"):
        s.pop(k, None)
    s["case"], s["seed"] = dict(case), int(seed)
    return s


def run(state):
    case, tex, seed = state["case"], state["texture"], state["seed"]
    kind, stochastic = case["kind"], case.get("form") == "stochastic"
    if kind == "gradients":
        params, latents, loss = tex.gradients(state["texels"], state["targets"])
        return {"params": params, "latents": latents, "loss": loss}
    if kind == "ewa":
        if stochastic:
            return tex.lookup_ewa(state["coords"], state["grad"], MAX_ANISOTROPY, seed=seed)
        return tex.lookup_ewa_deterministic(state["coords"], state["grad"], MAX_ANISOTROPY)
    lod, extra = state.get("lod"), {}
    if kind == "view":
        lod = tex.anisotropic_lod(state["grad"], MAX_ANISOTROPY)
    elif kind == "neural":
        extra["level_mode"] = stf.LEVEL_NEAREST
    if stochastic:
        out = tex.lookup(state["coords"], lod, filter=case["filter"], seed=seed, **extra)
    else:
        out = tex.lookup_deterministic(state["coords"], lod, filter=case["filter"], **extra)
    return {"lod": lod, "texels": out} if kind == "view" else out


# ---------------------------------------------------------------- work

MLP_FLOPS = 2 * (8 * 64 + 64 * 64 + 64 * 7)


def _queries(case):
    if "steps" in case:
        return case["width"] * case["height"] * case["steps"]
    if "queries" in case:
        return case["queries"]
    return case["width"] * len(_view_rows(case["height"]))


def work(case):
    kind = case["kind"]
    if kind == "gradients":
        b = case["batch"]
        return {"bytes": b * (8 + 16 + 28 + 32) + 2 * 4 * 5191, "flops": 3 * b * MLP_FLOPS}
    n = _queries(case)
    taps = 1
    if case["form"] == "deterministic" and "filter" in case:
        taps = (2 if case["filter"] == "linear" else 4) ** (3 if "steps" in case else 2)
    if kind in ("dense", "sparse"):
        # the samples that meet texels: 30% in a dense grid, 6% in the cloud
        size = {"f16": 2, "f32": 4, "e4m3": 1}[case["fmt"]]
        met = n * taps * 0.3 if kind == "dense" else n * taps * 0.06
        held = case["grid"] ** 3 if kind == "dense" else 0.04 * case["domain"] ** 3
        return {"bytes": int(n * 16 + min(met, held) * size), "flops": int(2 * met)}
    if kind == "neural":
        return {"bytes": n * (8 + 4 + 28) + min(n * taps, 4 * case["size"] ** 2 // 3) * 16,
                "flops": n * taps * MLP_FLOPS}
    w, h = case["tex_w"], case["tex_h"]
    c = case["channels"]
    size = {"f32": 4 * c, "f16": 2 * c, "dct": c / 16}[case["fmt"]]
    parts = 2 if taps > 1 and case["levels"] > 1 else 1
    held = w * h * (4 / 3 if case["levels"] > 1 else 1)
    query = 8 + (4 if kind == "image" and case["levels"] > 1 else 0) + (16 if kind in ("view", "ewa") else 0)
    out = 4 * c + (4 if kind == "view" else 0)
    return {"bytes": int(n * (query + out) + min(n * taps * parts, held) * size), "flops": 2 * n * taps * parts * c}


# ---------------------------------------------------------------- the same in 64 bits


def _variates(n0, n1, seed, sample=0):
    """Philox4x32-10 (Salmon et al., SC'11) of the queries n0 .. n1 - 1: four 24-bit uniforms."""
    mask = 0xFFFFFFFF
    q = torch.arange(n0, n1, device=DEV, dtype=torch.int64)
    c = [q & mask, q >> 32, torch.full_like(q, sample), torch.zeros_like(q)]
    k0, k1 = seed & mask, (seed >> 32) & mask
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & mask) ^ c[1] ^ k0, p1 & mask, ((p0 >> 32) & mask) ^ c[3] ^ k1, p0 & mask]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return [(w >> 8).double() * 2.0 ** -24 for w in c]


def _taps(x, filt):
    """First tap and weights (n, T) of each coordinate."""
    b = x.floor()
    f = x - b
    g = 1 - f
    if filt == "linear":
        return b.long(), torch.stack([g, f], -1)
    if filt == "bspline3":
        w = [g ** 3 / 6, f * f * (f / 2 - 1) + 2 / 3, g * g * (g / 2 - 1) + 2 / 3, f ** 3 / 6]
    else:
        w = [-f * g * g / 2, g * (1 + f * (1 - 1.5 * f)), f * (1 + g * (1 - 1.5 * g)), -g * f * f / 2]
    return b.long() - 1, torch.stack(w, -1)


def _pick(x, u, filt):
    """The tap drawn by u with probability |w| / sum|w|, and its sign times the sum."""
    first, w = _taps(x, filt)
    c = w.abs().cumsum(-1)
    total = c[..., -1]
    k = ((u * total)[..., None] >= c[..., :-1]).sum(-1)
    sign = torch.where(w.gather(-1, k[..., None])[..., 0] < 0, -1.0, 1.0)
    return first + k, sign * total if filt == "catmull_rom" else torch.ones_like(total)


def _exact_grid(case, s, seed, fetch):
    """Lookups of a 3D grid; fetch(x, y, z) gives voxels in 64 bits."""
    out = []
    for n0 in range(0, s["coords"].shape[0], 1 << 21):
        x = s["coords"][n0:n0 + (1 << 21)].double()
        if case["form"] == "stochastic":
            u = _variates(n0, n0 + x.shape[0], seed)
            picks = [_pick(x[:, a], u[a], case["filter"]) for a in range(3)]
            v = fetch(*(p[0] for p in picks)) * picks[0][1] * picks[1][1] * picks[2][1]
        else:
            (bx, wx), (by, wy), (bz, wz) = (_taps(x[:, a], case["filter"]) for a in range(3))
            v = torch.zeros(x.shape[0], dtype=torch.float64, device=DEV)
            t = wx.shape[1]
            for k in range(t ** 3):
                i, j, m = k % t, k // t % t, k // t // t
                v += wx[:, i] * wy[:, j] * wz[:, m] * fetch(bx + i, by + j, bz + m)
        out.append(v)
    return torch.cat(out)[:, None]


def _dense_fetch(case, s):
    n = case["grid"]
    v = s["values"].half().double() if case["fmt"] == "f16" else s["values"].double()
    flat = v.reshape(-1)

    def fetch(x, y, z):
        inside = (x >= 0) & (x < n) & (y >= 0) & (y < n) & (z >= 0) & (z < n)
        return torch.where(inside, flat[torch.where(inside, (z * n + y) * n + x, 0)], 0.0)
    return fetch


def _sparse_fetch(case, s):
    n = case["domain"] // 8
    o = s["origins"].long() // 8
    cells = torch.full((n ** 3,), -1, dtype=torch.int64, device=DEV)
    cells[(o[:, 0] * n + o[:, 1]) * n + o[:, 2]] = torch.arange(o.shape[0], device=DEV)
    flat = s["values"].reshape(-1)
    scale = None
    if case["fmt"] == "e4m3":
        scale = s["values"].abs().amax(1) / 448
        flat = (s["values"] / scale[:, None]).to(torch.float8_e4m3fn).float().reshape(-1)

    def fetch(x, y, z):
        inside = (x >= 0) & (x < 8 * n) & (y >= 0) & (y < 8 * n) & (z >= 0) & (z < 8 * n)
        leaf = cells[torch.where(inside, (x // 8 * n + y // 8) * n + z // 8, 0)]
        inside = inside & (leaf >= 0)
        leaf = torch.where(inside, leaf, 0)
        v = flat[leaf * 512 + (x & 7) * 64 + (y & 7) * 8 + (z & 7)].double()
        return torch.where(inside, v if scale is None else v * scale[leaf].double(), 0.0)
    return fetch


def _pyramid(case, values):
    out = [values.double()]
    for _ in range(1, case["levels"]):
        v = out[-1]
        if v.shape[0] > 1:
            v = (v[0::2] + v[1::2]) / 2
        if v.shape[1] > 1:
            v = (v[:, 0::2] + v[:, 1::2]) / 2
        out.append(v)
    return out


def _image_fetch(case, s):
    """fetch(L, x, y): texels of an image pyramid in 64 bits, clamped to the edge; and the sizes."""
    levels = _pyramid(case, s["values"])
    sizes = torch.tensor([[v.shape[1], v.shape[0]] for v in levels], device=DEV)
    c = case["channels"]
    if case["fmt"] != "dct":
        if case["fmt"] == "f16":
            levels = [v.half().double() for v in levels]
        start = torch.tensor([0] + [v.shape[0] * v.shape[1] for v in levels], device=DEV).cumsum(0)
        flat = torch.cat([v.reshape(-1, c) for v in levels])

        def fetch(L, x, y):
            w, h = sizes[L, 0], sizes[L, 1]
            return flat[start[L] + y.clamp_min(0).minimum(h - 1) * w + x.clamp_min(0).minimum(w - 1)]
        return fetch, sizes
    # six DCT coefficients per 8x8 block and channel: DC in 7 bits, the others in 5
    i = torch.arange(8, dtype=torch.float64, device=DEV)
    basis = torch.stack([torch.full_like(i, math.sqrt(0.125))] +
                        [0.5 * torch.cos((2 * i + 1) * u * math.pi / 16) for u in (1, 2)])
    kept = [(0, 0), (1, 0), (0, 1), (2, 0), (1, 1), (0, 2)]
    coef, blocks_w = [], []
    for v in levels:
        h, w = v.shape[:2]
        v = v[torch.arange((h + 7) // 8 * 8, device=DEV).clamp_max(h - 1)]
        v = v[:, torch.arange((w + 7) // 8 * 8, device=DEV).clamp_max(w - 1)]
        t = torch.einsum("byaxc,ux->byauc", v.reshape(v.shape[0] // 8, 8, v.shape[1] // 8, 8, c), basis)
        t = torch.einsum("byauc,vy->baucv", t, basis)
        coef.append(torch.stack([t[:, :, u, :, w2] for u, w2 in kept], -1).reshape(-1, c, 6))
        blocks_w.append((w + 7) // 8)
    start = torch.tensor([0] + [v.shape[0] for v in coef], device=DEV).cumsum(0)
    coef = torch.cat(coef)
    r = coef[..., 1:].abs().amax((0, 2))[:, None]
    away = lambda v: torch.sign(v) * (v.abs() + 0.5).floor()
    dc = away(coef[..., :1] * 127 / 8).clamp(0, 127) * 8 / 127
    ac = away(coef[..., 1:] * 15 / r).clamp(-15, 15) * r / 15
    coef = torch.cat([dc, ac], -1)
    blocks_w = torch.tensor(blocks_w, device=DEV)

    def fetch_dct(L, x, y):
        x = x.clamp_min(0).minimum(sizes[L, 0] - 1)
        y = y.clamp_min(0).minimum(sizes[L, 1] - 1)
        block = start[L] + (y >> 3) * blocks_w[L] + (x >> 3)
        bx, by = basis[:, x & 7], basis[:, y & 7]
        b = torch.stack([bx[u] * by[v] for u, v in kept], -1)
        return (coef[block] * b[:, None, :]).sum(-1)
    return fetch_dct, sizes


def _exact_filter2(case, coords, lod, seed, fetch, sizes, nearest):
    """2D lookups; fetch(L, x, y) gives (n, channels)."""
    out = []
    top = sizes.shape[0] - 1
    for n0 in range(0, coords.shape[0], 1 << 20):
        uv = coords[n0:n0 + (1 << 20)].double()
        n = uv.shape[0]
        lc = torch.zeros(n, dtype=torch.float64, device=DEV) if lod is None else lod[n0:n0 + n].double().clamp(0, top)
        u = _variates(n0, n0 + n, seed) if case["form"] == "stochastic" else None
        raster = lambda L: uv * sizes[L].double() - 0.5
        if u is not None:
            level_u = 0.5 if nearest else u[3]
            L = (lc + level_u).floor().long().clamp_max(top) if lod is not None else lc.long()
            x = raster(L)
            (ix, sx), (iy, sy) = (_pick(x[:, a], u[a], case["filter"]) for a in range(2))
            out.append(fetch(L, ix, iy) * (sx * sy)[:, None])
            continue
        L0 = (lc + 0.5).floor().long().clamp_max(top) if nearest else lc.floor().long()
        frac = torch.zeros_like(lc) if nearest else lc - L0
        v = 0.0
        for L, scale in ((L0, 1 - frac), ((L0 + 1).clamp_max(top), frac)):
            if L is not L0 and not bool((frac > 0).any()):
                continue
            x = raster(L)
            (bx, wx), (by, wy) = (_taps(x[:, a], case["filter"]) for a in range(2))
            for k in range(wx.shape[1] ** 2):
                i, j = k % wx.shape[1], k // wx.shape[1]
                v = v + (wx[:, i] * wy[:, j] * scale)[:, None] * fetch(L, bx + i, by + j)
        out.append(v)
    return torch.cat(out)


def _footprint(grad, sizes):
    """Major and minor axes in uv (the minor lengthened to major / MAX_ANISOTROPY) and log2 of
    the minor's length in level-0 texels."""
    g = grad.double()
    a, b = g[:, :2], g[:, 2:]
    la, lb = ((v * sizes[0].double()).norm(dim=1) for v in (a, b))
    swap = (la < lb)[:, None]
    major, minor = torch.where(swap, b, a), torch.where(swap, a, b)
    lmax, lmin = torch.maximum(la, lb), torch.minimum(la, lb)
    k = torch.where(lmin * MAX_ANISOTROPY < lmax, lmax / (lmin * MAX_ANISOTROPY), 1.0)
    return major, minor * k[:, None], torch.log2(lmin * k).clamp(0, sizes.shape[0] - 1)


def _ellipse(major, minor, uv, size):
    """A, B, C of Q(s, t), the centre and the bounding box [s0, s1] x [t0, t1]."""
    d0, d1 = major * size, minor * size
    k = (2 / d1.norm(dim=1)).clamp_max(1.0)[:, None]
    d0, d1 = d0 * k, d1 * k
    A = d0[:, 1] ** 2 + d1[:, 1] ** 2 + 1
    B = -2 * (d0[:, 0] * d0[:, 1] + d1[:, 0] * d1[:, 1])
    C = d0[:, 0] ** 2 + d1[:, 0] ** 2 + 1
    inv = 1 / (A * C - B * B / 4)
    A, B, C = A * inv, B * inv, C * inv
    det = 4 * A * C - B * B
    hs, ht = 2 / det * (det * C).sqrt(), 2 / det * (A * det).sqrt()
    c = uv * size - 0.5
    box = [(c[:, 0] - hs).ceil(), (c[:, 0] + hs).floor(), (c[:, 1] - ht).ceil(), (c[:, 1] + ht).floor()]
    return A, B, C, c, [b.long() for b in box]


def _exact_ewa(case, s, seed):
    fetch, sizes = _image_fetch(case, s)
    lut = torch.exp(-2 * torch.arange(128, dtype=torch.float64, device=DEV) / 127) - math.exp(-2)
    lut = torch.cat([lut, torch.zeros(1, dtype=torch.float64, device=DEV)])   # outside the ellipse
    stochastic = case["form"] == "stochastic"
    result = torch.zeros((s["coords"].shape[0], case["channels"]), dtype=torch.float64, device=DEV)
    u = _variates(0, s["coords"].shape[0], seed) if stochastic else None
    major, minor, lc = _footprint(s["grad"], sizes)
    top = sizes.shape[0] - 1
    if stochastic:
        parts = [((lc + u[3]).floor().long().clamp_max(top), torch.ones_like(lc))]
    else:
        L0 = lc.floor().long()
        parts = [(L0, 1 - (lc - L0)), ((L0 + 1).clamp_max(top), lc - L0)]
    for L, scale in parts:
        A, B, C, centre, (s0, s1, t0, t1) = _ellipse(major, minor, s["coords"].double(), sizes[L].double())
        # queries in order of their box's size, so that each batch loops over boxes alike
        for q in ((s1 - s0) * 4096 + (t1 - t0)).argsort().split(1 << 18):
            a, b, c, cs, ct = A[q], B[q], C[q], centre[q, 0], centre[q, 1]
            x0, x1, y0, y1, l = s0[q], s1[q], t0[q], t1[q], L[q]

            def texels():
                for dt in range(int((y1 - y0).max()) + 1):
                    for ds in range(int((x1 - x0).max()) + 1):
                        x, y = x0 + ds, y0 + dt
                        ss, tt = x - cs, y - ct
                        r2 = (a * ss + b * tt) * ss + c * tt * tt
                        r2 = torch.where((x <= x1) & (y <= y1), r2, 1.0)
                        yield x, y, lut[(r2 * 128).clamp(0, 128).long()]
            total = torch.zeros_like(a)
            if not stochastic:
                acc = torch.zeros((q.numel(), case["channels"]), dtype=torch.float64, device=DEV)
                for x, y, w in texels():
                    total += w
                    acc += w[:, None] * fetch(l, x, y)
                result[q] += acc * (scale[q] / total)[:, None]
                continue
            for x, y, w in texels():
                total += w
            us, run_sum = u[0][q] * total, torch.zeros_like(a)
            px, py, found = x0.clone(), y0.clone(), torch.zeros_like(x0, dtype=torch.bool)
            for x, y, w in texels():
                run_sum += w
                here = (us < run_sum) & ~found
                px, py, found = torch.where(here, x, px), torch.where(here, y, py), found | here
            result[q] = fetch(l, px, py)
    return result


def _exact_weights(s):
    """Latents and decoder in 64 bits, as the binary16 storage holds them."""
    parts, at = [], 0
    for rows, cols in ((8, 64), (1, 64), (64, 64), (1, 64), (64, 7), (1, 7)):
        p = s["params"][at:at + rows * cols].reshape(rows, cols)
        parts.append(p.half().double() if rows > 1 else p.double()[0])
        at += rows * cols
    return s["latents"].half().double(), parts


def _mlp(z, p):
    return torch.relu(torch.relu(z @ p[0] + p[1]) @ p[2] + p[3]) @ p[4] + p[5]


def _exact_neural(case, s, seed):
    latents, p = _exact_weights(s)
    fallback = s["fallback"].half().double()
    side = [max(1, case["size"] >> k) for k in range(_neural_levels(case["size"]))]
    sizes = torch.tensor([[w, w] for w in side], device=DEV)
    area = sizes[:, 0] * sizes[:, 0]
    start = area.cumsum(0) - area

    def fetch(L, x, y):
        w = sizes[L, 0]
        at = start[L] + y.clamp_min(0).minimum(w - 1) * w + x.clamp_min(0).minimum(w - 1)
        stored = L >= NEURAL_LEVELS
        v = torch.empty((at.numel(), 7), dtype=torch.float64, device=DEV)
        v[~stored] = _mlp(latents[at[~stored]], p)
        v[stored] = fallback[at[stored] - int(start[NEURAL_LEVELS])]
        return v
    return _exact_filter2(case, s["coords"], s["lod"], seed, fetch, sizes, True)


def _exact_gradients(case, s):
    latents, p = _exact_weights(s)
    z = latents[s["texels"]].requires_grad_()
    for v in p:
        v.requires_grad_()
    loss = (_mlp(z, p) - s["targets"].double()).square().sum() / case["batch"]
    loss.backward()
    return {"params": torch.cat([v.grad.reshape(-1) for v in p]), "latents": z.grad, "loss": loss.detach().reshape(1)}


def exact(case, seed):
    s, kind = _inputs(case, seed), case["kind"]
    if kind == "dense":
        return _exact_grid(case, s, seed, _dense_fetch(case, s))
    if kind == "sparse":
        return _exact_grid(case, s, seed, _sparse_fetch(case, s))
    if kind == "gradients":
        return _exact_gradients(case, s)
    if kind == "neural":
        return _exact_neural(case, s, seed)
    if kind == "ewa":
        return _exact_ewa(case, s, seed)
    fetch, sizes = _image_fetch(case, s)
    if kind == "image":
        return _exact_filter2(case, s["coords"], s.get("lod"), seed, fetch, sizes, False)
    lod = _footprint(s["grad"], sizes)[2]
    return {"lod": lod, "texels": _exact_filter2(case, s["coords"], lod, seed, fetch, sizes, False)}
