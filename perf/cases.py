"""Performance cases: the calls that a user of the framework makes for every
frame, over the range of frame sizes, component counts, storage precisions
and options that they are made with.

Kinds of case (the entry point that ``run`` goes through):

- ``apply``: one camera behind a handle, ``GMM.apply`` on frames in device
  memory, with or without the per-stream masks. The handle keeps the state, so
  the masks are the outputs.
- ``noalloc``: one camera whose state the caller owns,
  ``gmm_apply_open3_noalloc`` (tick and 3x3 opening): returns the mask and the
  whole updated state.
- ``pool``: many cameras of mixed sizes, ``Pool.submit_many`` and ``Pool.tick``.
- ``host``: one camera fed from page-locked host memory, ``GMM.apply_host``
  (upload, tick, mask download and wait).

A case holds a short clip of frames that its passes go through in turn, and a
model that has already seen enough of the scene to have settled: a static
camera before a textured background with sensor noise, a flickering region,
moving objects that stand nearer than the background, and 2% of the depth
readings missing.
"""
import ctypes
import math

import numpy as np
import torch

import paper_2110_14934_gb300 as G

CLIP = 16  # frames of a clip (the pool of 64 cameras: 6)
WARM = 320  # ticks that a handle or a pool has taken before the first pass: the background holds most of the weight by then
PRM = dict(alpha=0.01, match_k=2.5, bg_T=0.7, init_var=225.0, init_w=0.05)
TILE = 256  # pixels of a state tile
POOL_SIZES = ((240, 320), (480, 640), (720, 1280), (1080, 1920))
ODD_SIZES = ((237, 321), (479, 633), (720, 1278), (540, 960), (600, 799), (1079, 1917))


def listed():
    def one(name, kind, H, W, M, prec="f32", **more):
        return dict(name=name, kind=kind, H=H, W=W, M=M, prec=prec, **more)

    return [
        # The smallest frame the many-camera workloads use: a call is mostly launch and latency.
        one("apply_320x240_m3", "apply", 240, 320, 3),
        # The Kinect's own frame, with the opening, as the paper's sensor delivers it.
        one("noalloc_640x480_m3", "noalloc", 480, 640, 3),
        # A cropped frame: rows that end inside a mask word, a last tile that is not full.
        one("noalloc_1021x767_m4", "noalloc", 767, 1021, 4),
        # One full-HD camera with the most components: the single-camera headline.
        one("apply_1920x1080_m5", "apply", 1080, 1920, 5),
        # The same with 16-bit state, and the colour and depth answers asked for beside the fused one.
        one("apply_1920x1080_m5_f16", "apply", 1080, 1920, 5, "f16", masks=True),
        # 16-bit state that the caller owns.
        one("noalloc_1280x720_m4_f16", "noalloc", 720, 1280, 4, "f16"),
        # The density-weighted learning rate and the per-channel variance.
        one("noalloc_1280x720_m3_options", "noalloc", 720, 1280, 3, flags=G.FLAG_RHO_ETA | G.FLAG_VAR_PER_CHANNEL),
        # The augmentation alternative: one four-channel mixture per pixel.
        one("noalloc_960x540_m5_augmented", "noalloc", 540, 960, 5, mode=G.MODE_AUGMENTED),
        # The largest frame of the caller-owned path.
        one("noalloc_3840x2160_m3", "noalloc", 2160, 3840, 3),
        # A site with 64 cameras of four sizes on one GPU, launch shape tuned once at start-up: the batched headline.
        dict(name="pool_64_cameras", kind="pool", cams=64, odd=False, prec="f32", tuned=True),
        # A smaller site, frames cropped to odd sizes, 16-bit state, default launch shape.
        dict(name="pool_24_odd_cameras_f16", kind="pool", cams=24, odd=True, prec="f16", tuned=False),
        # Frames that arrive in host memory, one at a time, the mask wanted before the next.
        one("host_1280x720_m5_f16", "host", 720, 1280, 5, "f16"),
    ]


def draw(rng):
    kind = rng.choice(("apply", "apply", "noalloc", "noalloc", "noalloc", "pool", "host"))
    prec = rng.choice(("f32", "f32", "f16"))
    if kind == "pool":
        return dict(kind=kind, cams=int(round(math.exp(rng.uniform(math.log(3), math.log(40))))), odd=rng.random() < 0.5, prec=prec, tuned=False)
    lo, hi = math.log(320 * 240), math.log(3800 * 2150 if kind != "host" else 1920 * 1080)
    pixels = math.exp(rng.uniform(lo, hi))
    W = int(round(math.sqrt(pixels * rng.choice((4 / 3, 16 / 9, 1.0)))))
    if rng.random() < 0.5:
        W = max(32, W // 32 * 32)
    case = dict(kind=kind, H=max(1, int(pixels / W)), W=W, M=rng.choice((3, 4, 5)), prec=prec)
    kinds = rng.random()
    if kinds < 0.12:
        case["flags"] = rng.choice((G.FLAG_RHO_ETA, G.FLAG_VAR_PER_CHANNEL, G.FLAG_RHO_ETA | G.FLAG_VAR_PER_CHANNEL))
    elif kinds < 0.24:
        case["mode"] = G.MODE_AUGMENTED
    if kind == "apply":
        case["masks"] = rng.random() < 0.3
    return case


# ---------------------------------------------------------------- frames
def _clip(H, W, frames, gen, dev):
    """uint8 [frames, H, W, 3] and uint16 millimetres (in int16) [frames, H, W]."""
    def uniform(lo, hi, *shape):
        return lo + (hi - lo) * torch.rand(shape, generator=gen, device=dev)

    yy = torch.linspace(0, 1, H, device=dev).view(H, 1, 1)
    xx = torch.linspace(0, 1, W, device=dev).view(1, W, 1)
    colour = uniform(50, 130, 3) + uniform(-40, 40, 3) * xx + uniform(-40, 40, 3) * yy
    back = (1500 + 2500 * (0.3 * xx + 0.7 * yy)).squeeze(2)
    # a tenth of the picture flickers (leaves, a screen): phase by place
    top, left = uniform(0, 0.68, 2).tolist()
    flicker = ((yy >= top) & (yy < top + 0.32) & (xx >= left) & (xx < left + 0.32)).float()
    phase = 40.0 * (xx + yy)
    rgb = torch.empty((frames, H, W, 3), dtype=torch.uint8, device=dev)
    depth = torch.empty((frames, H, W), dtype=torch.int16, device=dev)
    tint, near = uniform(0, 255, 6, 3), uniform(700, 1400, 6)
    for t in range(frames):
        c = colour + 25.0 * flicker * torch.sin(2 * math.pi * t / 17.3 + phase)
        z = back
        place = uniform(0.05, 0.95, 6, 2).tolist()
        for k, (cy, cx) in enumerate(place):  # a walking rectangle, five smaller ellipses
            if k == 0:
                inside = ((yy - cy).abs() < 0.08) & ((xx - cx).abs() < 0.06)
            else:
                inside = ((yy - cy) / 0.04) ** 2 + ((xx - cx) / 0.03) ** 2 < 1
            c = torch.where(inside, tint[k], c)
            z = torch.where(inside.squeeze(2), near[k], z)
        c = c + 3.0 * torch.randn((H, W, 3), generator=gen, device=dev)
        z = z + 5.0 * torch.randn((H, W), generator=gen, device=dev)
        z = torch.where(torch.rand((H, W), generator=gen, device=dev) < 0.02, torch.zeros_like(z), z)
        rgb[t] = c.round().clamp(0, 255).to(torch.uint8)
        depth[t] = z.round().clamp(0, 32767).to(torch.int16)
    return rgb, depth


# ---------------------------------------------------------------- the method in plain torch
class _Plain:
    """The per-pixel method on flat tensors, in any floating type: makes the
    settled states that callers own, and the 64-bit values of one tick."""

    def __init__(self, case, dtype):
        self.M, self.dtype = case["M"], dtype
        self.augmented = case.get("mode", 0) == G.MODE_AUGMENTED
        self.flags = case.get("flags", 0)
        f32 = lambda v: float(np.float32(v))  # noqa: E731 (the library takes float32 parameters)
        self.alpha, self.T, self.init_w = f32(PRM["alpha"]), f32(PRM["bg_T"]), f32(PRM["init_w"])
        self.k2, self.init_var, self.scale = f32(PRM["match_k"]) ** 2, f32(PRM["init_var"]), f32(255.0 / 4095.0)
        self.mix = None

    def samples(self, rgb, depth):
        x = rgb.reshape(-1, 3).t().to(self.dtype).contiguous()
        return x, depth.reshape(1, -1).to(self.dtype)

    def fresh(self, x):
        D, N = x.shape
        return [x.new_full((self.M, N), 1.0 / self.M), x[None].repeat(self.M, 1, 1), x.new_full((self.M, N), self.init_var)]

    def start(self, rgb, depth):
        x, z = self.samples(rgb, depth)
        self.mix = [self.fresh(torch.cat([x, self.scale * z]) if self.augmented else x)]
        self.byte = torch.zeros(z.shape[1], dtype=torch.int32, device=x.device)
        self.started = None
        if not self.augmented:
            self.mix.append(self.fresh(z))
            self.started = torch.zeros(z.shape[1], dtype=torch.bool, device=x.device)

    def step(self, mix, x, alpha):
        """One tick of one mixture; returns it and the foreground bits."""
        w, mu, v = mix
        M, D = mu.shape[:2]
        d2 = ((x - mu) ** 2).sum(1)
        hit = d2 < self.k2 * v
        free, sel = torch.ones_like(hit[0]), []
        for i in range(M):
            sel.append(hit[i] & free)
            free = free & ~hit[i]
        sel = torch.stack(sel)
        gain = sel.clone()
        sel[M - 1] |= free
        w = w * (1 - alpha) + alpha * gain
        w[M - 1] = torch.where(free, torch.full_like(w[0], self.init_w), w[M - 1])
        w = w / w.sum(0)
        rho = torch.full_like(w[0], alpha)
        vj = torch.where(sel, v, torch.zeros_like(v)).sum(0)
        if self.flags & G.FLAG_RHO_ETA:
            d2j = torch.where(sel, d2, torch.zeros_like(d2)).sum(0)
            s2 = vj if self.flags & G.FLAG_VAR_PER_CHANNEL else vj / D
            rho = (alpha * (2 * math.pi * s2) ** (-0.5 * D) * torch.exp(-d2j / (2 * s2))).clamp(max=1.0)
        muj = torch.where(sel[:, None], mu, torch.zeros_like(mu)).sum(0)
        moved = (1 - rho) * muj + rho * x
        d2n = ((x - moved) ** 2).sum(0)
        if self.flags & G.FLAG_VAR_PER_CHANNEL:
            d2n = d2n / D
        vn = ((1 - rho) * vj + rho * d2n).clamp(min=1.0)
        moved = torch.where(free, x, moved)
        vn = torch.where(free, torch.full_like(vn, self.init_var), vn)
        mu = torch.where(sel[:, None], moved, mu)
        v = torch.where(sel, vn, v)
        key = w / v.sqrt()
        rows = [[w[i], v[i], key[i], sel[i]] + [mu[i, c] for c in range(D)] for i in range(M)]
        for last in range(M - 1, 0, -1):  # a stable exchange sort, best first
            for i in range(last):
                swap = rows[i + 1][2] > rows[i][2]
                for k in range(4 + D):
                    a, b = rows[i][k], rows[i + 1][k]
                    rows[i][k], rows[i + 1][k] = torch.where(swap, b, a), torch.where(swap, a, b)
        before = torch.zeros_like(w[0])
        total = torch.zeros_like(w[0])
        for r in rows:
            before = torch.where(r[3], total, before)
            total = total + r[0]
        mix = [torch.stack([r[0] for r in rows]), torch.stack([torch.stack(r[4:]) for r in rows]), torch.stack([r[1] for r in rows])]
        return mix, free | (before > self.T)

    def tick(self, rgb, depth, alpha=None):
        alpha = self.alpha if alpha is None else alpha
        x, z = self.samples(rgb, depth)
        seen = z[0] > 0
        if self.augmented:
            z = torch.where(seen, self.scale * z[0], self.mix[0][1][0, 3])[None]
            self.mix[0], fg = self.step(self.mix[0], torch.cat([x, z]), alpha)
            self.byte = fg.int()
            return
        self.mix[0], fc = self.step(self.mix[0], x, alpha)
        new, fd = self.step(self.mix[1], z, alpha)
        begin, go = seen & ~self.started, seen & self.started
        first = self.fresh(z)
        for k in range(3):
            self.mix[1][k] = torch.where(go, new[k], torch.where(begin, first[k], self.mix[1][k]))
        fd = torch.where(go, fd, torch.where(seen, torch.zeros_like(fd), fc))
        self.started = self.started | seen
        F, count = (self.byte & 1).bool(), (self.byte >> 1 & 7) - 3
        same, up, down = fc == fd, count == 3, count == -3
        moved = torch.where(F == fc, count + 1, count - 1)
        count = torch.where(same | up | down, torch.zeros_like(count), moved)
        F = torch.where(same, fd, torch.where(up, fc, torch.where(down, fd, F)))
        self.byte = F.int() | (count + 3 << 1) | (self.started.int() << 4)

    def planes(self):
        """[M, 8, N]: w_c, mu_r, mu_g, mu_b, v_c, w_d, mu_d, v_d."""
        w, mu, v = self.mix[0]
        zero = torch.zeros_like(w)
        if self.augmented:
            return torch.stack([w, mu[:, 0], mu[:, 1], mu[:, 2], v, zero, mu[:, 3], zero], 1)
        wd, mud, vd = self.mix[1]
        on = self.started
        return torch.stack([w, mu[:, 0], mu[:, 1], mu[:, 2], v, wd * on, mud[:, 0] * on, vd * on], 1)

    def load(self, planes, byte):
        p = planes.to(self.dtype)
        self.byte = byte.int()
        if self.augmented:
            self.mix = [[p[:, 0].clone(), torch.stack([p[:, 1], p[:, 2], p[:, 3], p[:, 6]], 1), p[:, 4].clone()]]
            return
        self.started = (byte >> 4 & 1).bool()
        wd, vd = p[:, 5].clone(), p[:, 7].clone()
        wd[:, ~self.started], vd[:, ~self.started] = 1.0 / self.M, self.init_var
        self.mix = [[p[:, 0].clone(), p[:, 1:4].contiguous(), p[:, 4].clone()], [wd, p[:, 6:7].contiguous(), vd]]


def _settled(case, rgb, depth):
    """Planes [M, 8, N] (float32, exact in the storage type) and List-1 bytes of a model that has settled on the clip."""
    m = _Plain(case, torch.float32)
    m.start(rgb[0], depth[0])
    for t in range(1, 2 * len(rgb)):  # quickly at first, at the model's own rate at last
        m.tick(rgb[t % len(rgb)], depth[t % len(rgb)], 0.06 if t < 26 else None)
    planes = m.planes()
    if case["prec"] == "f16":
        weights = torch.zeros(8, dtype=torch.bool, device=planes.device)
        weights[[0, 5]] = True
        planes = torch.where(weights[None, :, None], planes.bfloat16().float(), planes.half().float())
    return planes, m.byte


def _tiled(values, H, W):
    """[..., H*W] -> [..., tiles, TILE]: rows padded to 32 pixels, tiles of TILE consecutive padded pixels, zeros in the padding."""
    lead = values.shape[:-1]
    v = torch.nn.functional.pad(values.reshape(*lead, H, W), (0, -W % 32)).flatten(-2)
    return torch.nn.functional.pad(v, (0, -v.shape[-1] % TILE)).reshape(*lead, -1, TILE)


def _state_parts(planes, H, W, prec):
    """The planes in the order of the caller-owned state: FP32 one array
    [tiles, M, 8, TILE]; FP16/BF16 the weights, the red and green means, and
    the rest, each [tiles, M, TILE, ...]."""
    t = _tiled(planes, H, W).permute(2, 0, 1, 3)  # [tiles, M, 8, TILE]
    if prec == "f32":
        return [t.contiguous()]
    pick = lambda *f: t[:, :, list(f)].permute(0, 1, 3, 2).contiguous()  # noqa: E731
    return [pick(0, 5), pick(1, 2), pick(3, 4, 6, 7)]


def _views(state, tiles, M, prec):
    """The parts of _state_parts as views of the state's own bytes."""
    if prec == "f32":
        return [state[: tiles * M * 8 * TILE * 4].view(torch.float32).view(tiles, M, 8, TILE)]
    body = state[: tiles * M * 8 * TILE * 2]
    h = body.view(torch.float16).view(tiles, M, 2, TILE, 4)
    return [body.view(torch.bfloat16).view(tiles, M, 2, TILE, 4)[:, :, 0, :, :2], h[:, :, 0, :, 2:], h[:, :, 1]]


# ---------------------------------------------------------------- preparation
def _prec(case):
    return G.PREC_F16 if case["prec"] == "f16" else G.PREC_F32


def _model_args(case):
    return dict(PRM, precision=_prec(case), mode=case.get("mode", G.MODE_FUSION), flags=case.get("flags", 0))


def _generator(seed):
    dev = torch.device("cuda")
    return torch.Generator(device=dev).manual_seed(int(seed)), dev


def _prepare_noalloc(case, seed):
    gen, dev = _generator(seed)
    H, W, M = case["H"], case["W"], case["M"]
    rgb, depth = _clip(H, W, CLIP, gen, dev)
    planes, byte = _settled(case, rgb, depth)
    state = torch.zeros(G.state_bytes(H, W, M, _prec(case)), dtype=torch.uint8, device=dev)
    bytes_ = _tiled(byte, H, W).to(torch.uint8)
    parts = _views(state, bytes_.shape[0], M, case["prec"])
    for view, values in zip(parts, _state_parts(planes, H, W, case["prec"])):
        view.copy_(values)
    fusion = state[-bytes_.numel():]
    fusion.copy_(bytes_.flatten())
    mask = torch.zeros((H, G.mask_words_per_row(W)), dtype=torch.int32, device=dev)
    cfg = G.make_config(H, W, M, **_model_args(case))
    return dict(case=case, lib=G.load_library(), cfg=cfg, rgb=rgb, depth=depth, t=0, state=state, mask=mask,
                out=dict(planes=parts, fusion=fusion, mask=mask))


def _prepare_apply(case, seed):
    gen, dev = _generator(seed)
    H, W = case["H"], case["W"]
    rgb, depth = _clip(H, W, CLIP, gen, dev)
    g = G.GMM(H, W, case["M"], **_model_args(case))
    masks = [g.new_mask() for _ in range(3 if case.get("masks") else 1)]
    frames = [(rgb[t], depth[t]) for t in range(CLIP)]
    for t in range(WARM):
        g.apply(*frames[t % CLIP], *masks)
    return dict(case=case, g=g, frames=frames, masks=masks, t=0)


def _prepare_host(case, seed):
    gen, dev = _generator(seed)
    H, W = case["H"], case["W"]
    rgb, depth = _clip(H, W, CLIP, gen, dev)
    g = G.GMM(H, W, case["M"], **_model_args(case))
    for t in range(WARM):
        g.apply(rgb[t % CLIP], depth[t % CLIP])
    rgb_h, depth_h = rgb.cpu().pin_memory(), depth.cpu().pin_memory()
    mask = torch.zeros((H, G.mask_words_per_row(W)), dtype=torch.int32).pin_memory()
    frames = [(rgb_h[t].numpy(), depth_h[t].numpy()) for t in range(CLIP)]
    return dict(case=case, g=g, frames=frames, keep=(rgb_h, depth_h, mask), mask=mask.numpy().view(np.uint32), t=0)


def _pool_cameras(case):
    sizes = ODD_SIZES if case["odd"] else POOL_SIZES
    return [(*sizes[k % len(sizes)], (3, 5, 4, 5, 3)[k % 5] if case["odd"] else (5, 3, 5)[k // 4 % 3]) for k in range(case["cams"])]


def _prepare_pool(case, seed):
    gen, dev = _generator(seed)
    clip = CLIP if case["cams"] < 32 else 6
    pool = G.Pool(precision=_prec(case), max_cams=case["cams"])
    cams, clips, masks = [], [], []
    for H, W, M in _pool_cameras(case):
        clips.append(_clip(H, W, clip, gen, dev))
        masks.append(torch.zeros((H, G.mask_words_per_row(W)), dtype=torch.int32, device=dev))
        cams.append(pool.admit(H, W, M, **PRM))
    mask_ptrs = [m.data_ptr() for m in masks]
    frames = [([c[0][t].data_ptr() for c in clips], [c[1][t].data_ptr() for c in clips], mask_ptrs) for t in range(clip)]
    for t in range(WARM):
        pool.submit_many(cams, *frames[t % clip])
        pool.tick()
    if case["tuned"]:
        pool.submit_many(cams, *frames[0])
        pool.autotune(2)
        pool.tick()
    pool.use_graph(True)
    return dict(case=case, pool=pool, cams=cams, clips=clips, frames=frames, masks=masks, t=0)


def prepare(case, seed):
    return {"noalloc": _prepare_noalloc, "apply": _prepare_apply, "host": _prepare_host, "pool": _prepare_pool}[case["kind"]](case, seed)


# ---------------------------------------------------------------- one pass
def run(s):
    kind, t = s["case"]["kind"], s["t"]
    s["t"] = t + 1
    if kind == "noalloc":
        k = t % CLIP
        rc = s["lib"].gmm_apply_open3_noalloc(ctypes.byref(s["cfg"]), s["state"].data_ptr(), 0, s["rgb"][k].data_ptr(), s["depth"][k].data_ptr(),
                                              s["mask"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        if rc != 0:
            raise RuntimeError("gmm_apply_open3_noalloc: %d" % rc)
        return s["out"]
    if kind == "pool":
        s["pool"].submit_many(s["cams"], *s["frames"][t % len(s["frames"])])
        s["pool"].tick()
        return s["masks"]
    if kind == "host":
        return s["g"].apply_host(*s["frames"][t % CLIP], s["mask"])
    s["g"].apply(*s["frames"][t % CLIP], *s["masks"])
    return s["masks"]


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    """Bytes per pixel in the state's own layout: every weight read and
    written, every variance read (the ranking needs them all), the mean of one
    component per mixture read, its mean and variance written; the frame, the
    List-1 byte both ways and the mask bits once. The unmatched components'
    means and variances do not change in a tick."""
    total_b = total_f = 0.0
    if case["kind"] == "pool":
        views = [(H, W, M, False) for H, W, M in _pool_cameras(case)]
    else:
        views = [(case["H"], case["W"], case["M"], case.get("mode", 0) == G.MODE_AUGMENTED)]
    size = 2 if case["prec"] == "f16" else 4
    for H, W, M, augmented in views:
        streams, means = (1, 4) if augmented else (2, 4)
        values = streams * M * 3 + 2 * means + streams
        masks = 3 if case.get("masks") else 1
        total_b += H * W * (values * size + 5 + 2 + masks / 8)
        total_f += H * W * (10 * streams * M + 60)
    return {"bytes": total_b, "flops": total_f}


def exact(case, seed):
    """One tick in 64 bits from the same state and frame: the state's values
    (masks and bytes are whole numbers). A handle or a pool gives masks alone."""
    if case["kind"] != "noalloc":
        return None
    gen, dev = _generator(seed)
    rgb, depth = _clip(case["H"], case["W"], CLIP, gen, dev)
    planes, byte = _settled(case, rgb, depth)
    m = _Plain(case, torch.float64)
    m.load(planes, byte)
    m.tick(rgb[0], depth[0])
    return dict(planes=_state_parts(m.planes(), case["H"], case["W"], case["prec"]), fusion=None, mask=None)
