"""The workloads this library is timed on, through its public Python entry points.

A case is one call a user makes: the decode of a texture grid or of a list of
texture coordinates in one of the precision forms, a training step (continuous
latents, QAT latents, or the autograd function's forward and backward), the
batched decode of many materials, or a rendered frame.  Shapes follow the
repository's own workloads: 4 BC1 latents at 1/4 .. 1/32 of the output side with
half-texel shifts on the 2nd and 4th, He-initialised ReLU MLPs 12-D-..-D-9,
uniform random BC1 blocks (both modes), 2048^2 sinusoid targets, Voronoi frames.

`exact` restates every case in 64-bit torch arithmetic.  Two things are taken
as they are defined rather than in 64 bits, because they choose which texels are
read: a texture coordinate is an FP32 value (a grid's texel centre (i + 1/2) / W
rounded once), and the texel coordinate u W - 1/2 + shift is rounded once to FP32.
"""
import math

import torch

import paper_2506_06040_gb300 as nb
from paper_2506_06040_gb300.train import ContinuousModel, NbtcDecodeFn, QatModel, padded

SHIFTS = (0.0, 0.5, 0.0, 0.5)
FORMS = {"fp32": nb.FP32, "fp32_tc": nb.FP32_TC, "fp16": nb.FP16, "fp16_split": nb.FP16_SPLIT,
         "e4m3": nb.FP8_E4M3, "e4m3_split": nb.FP8_E4M3_SPLIT}
OUT_BYTES = {"fp32": 4, "fp32_tc": 4, "fp16": 2, "fp16_split": 2, "e4m3": 2, "e4m3_split": 2}
C = 9  # output channels: albedo RGB, normal XY, roughness, metalness, AO, displacement


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # one small texture (or one streamed 256^2 tile) decoded in full precision: the call's latency counts
        dict(name="grid_fp32_256", kind="grid", form="fp32", w=256, h=256, hid=32, depth=2, wrap=False),
        # a whole 4096^2 texture set in plain FP32: the offline or reference-quality decode
        dict(name="grid_fp32_4096", kind="grid", form="fp32", w=4096, h=4096, hid=64, depth=2, wrap=False),
        # the same set at FP32 accuracy on the tensor cores
        dict(name="grid_fp32tc_4096", kind="grid", form="fp32_tc", w=4096, h=4096, hid=64, depth=2, wrap=False),
        # a texture set decoded in FP16 at load time: the throughput form
        dict(name="grid_fp16_4096", kind="grid", form="fp16", w=4096, h=4096, hid=64, depth=3, wrap=False),
        # a texture of no particular size, at the FP16 error bound (rows that no tile divides)
        dict(name="grid_fp16split_ragged", kind="grid", form="fp16_split", w=1500, h=1000, hid=64, depth=3, wrap=False),
        # scattered lookups (ray hits, feedback samples): a list of tiled texture coordinates, an odd count
        dict(name="uv_e4m3split_1m", kind="uv", form="e4m3_split", n=1_000_003, side=4096, hid=64, depth=3, wrap=True),
        # one optimisation step of the compressor at full size
        dict(name="train_1m", kind="train", batch=1 << 20, side=4096, target=2048, stride=4, loss="mse"),
        # the decoder inside somebody's own torch program: differentiable forward, then backward, a small odd batch
        dict(name="autograd_50k", kind="autograd", batch=50_001, side=1024, stride=3),
        # fine-tuning of the BC1 latents themselves, a quarter batch on a half-size texture
        dict(name="qat_256k", kind="qat", batch=1 << 18, side=2048, target=1024, stride=4, loss="l1"),
        # a level's materials decoded together when it is loaded
        dict(name="batch_24", kind="batch", materials=24, smax=2048),
        # a rendered frame's G-buffer: per-pixel materials, trilinear latents
        dict(name="frame_2160p", kind="frame", materials=64, w=3840, h=2160, smax=2048, aniso=False),
        # a rendered frame with anisotropic latents (2 to 16 probes a pixel)
        dict(name="frame_1080p_aniso", kind="frame", materials=16, w=1920, h=1080, smax=2048, aniso=True),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["grid", "grid", "grid", "uv", "train", "autograd", "qat", "batch", "frame"])
    if kind in ("grid", "uv"):
        form = rng.choice(sorted(FORMS))
        c = dict(kind=kind, form=form, hid=rng.choice([16, 32, 64, 64]), depth=rng.choice([1, 2, 3]),
                 wrap=rng.random() < 0.5)
        if kind == "grid":
            # plain FP32 costs about ten times the other forms a texel, and more on ragged rows
            top = 4096 if form != "fp32" else 3000 if c["depth"] < 3 else 2048
            c["w"], c["h"] = _logint(rng, 160, top), _logint(rng, 160, top)
            if rng.random() < 0.5:  # texture sides are mostly multiples of 128
                c["w"] = max(128, c["w"] // 128 * 128)
        else:
            c["n"], c["side"] = _logint(rng, 5_000, 2_000_000), 1 << rng.randint(8, 12)
        return c
    if kind in ("train", "qat"):
        return dict(kind=kind, batch=_logint(rng, 4_000, 1 << 20), side=1 << rng.randint(9, 12),
                    target=rng.choice([256, 500, 1024, 2048]), stride=rng.choice([3, 4, 4]),
                    loss=rng.choice(["mse", "l1"]))
    if kind == "autograd":
        return dict(kind=kind, batch=_logint(rng, 4_000, 400_000), side=1 << rng.randint(8, 12),
                    stride=rng.choice([3, 4]))
    if kind == "batch":
        return dict(kind=kind, materials=rng.randint(2, 40), smax=rng.choice([512, 1024, 2048]))
    w, h = rng.choice([(1280, 720), (1920, 1080), (2560, 1440), (3840, 2160)])
    aniso = rng.random() < 0.4 and w < 1920
    return dict(kind=kind, materials=rng.randint(3, 64), w=w, h=h, smax=rng.choice([512, 1024, 2048]), aniso=aniso)


# ------------------------------------------------------------------ inputs

_ctx = None


def _context():
    """The process's library context, as a program keeps it."""
    global _ctx
    if _ctx is None:
        _ctx = nb.Context(0)
    return _ctx


def _gen(seed, stream=0):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 1009 + stream)


def _normal(g, shape, std):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float32) * std


def _uniform(g, shape, lo=0.0, hi=1.0):
    return torch.rand(shape, generator=g, device="cuda", dtype=torch.float32) * (hi - lo) + lo


def _mlp(g, dims):
    """He-initialised weights [out, in] and small biases."""
    ws = [_normal(g, (o, i), math.sqrt(2.0 / i)) for i, o in zip(dims, dims[1:])]
    return ws, [_normal(g, (o,), 0.01) for o in dims[1:]]


def _dims(case):
    return [12] + [case["hid"]] * case["depth"] + [C]


def _level_sides(w, h):
    """Latents at 1/4 .. 1/32 of the output, in whole 4x4 blocks."""
    return [(max(4, (w >> (k + 2)) // 4 * 4), max(4, (h >> (k + 2)) // 4 * 4)) for k in range(4)]


def _mips(side):
    m = 1
    while (side >> m) >= 4 and (side >> m) % 4 == 0 and (side >> (m - 1)) % 2 == 0:
        m += 1
    return m


def _raw_levels(g, sides, mips):
    """Per level (blocks int64 with all mips back to back, w, h, mips, shift): uniform random bits."""
    out = []
    for k, (w, h) in enumerate(sides):
        m = _mips(w) if mips else 1
        n = sum((max(4, w >> i) // 4) * (max(4, h >> i) // 4) for i in range(m))
        blocks = torch.randint(-2 ** 63, 2 ** 63 - 1, (n,), generator=g, device="cuda", dtype=torch.int64)
        out.append((blocks, w, h, m, SHIFTS[k]))
    return out


def _raw_material(g, sides, dims, mips=False):
    return _raw_levels(g, sides, mips), *_mlp(g, dims)


def _material(raw, wrap):
    levels, ws, bs = raw
    return nb.Material([(b.cpu().numpy().view("uint64"), w, h, m, s) for b, w, h, m, s in levels],
                       [w.cpu().numpy() for w in ws], [b.cpu().numpy() for b in bs], nb.WRAP if wrap else nb.CLAMP)


def _decode_raw(case, seed):
    sides = _level_sides(case["w"], case["h"]) if case["kind"] == "grid" else _level_sides(case["side"], case["side"])
    return _raw_material(_gen(seed), sides, _dims(case))


def _decode_uv(case, seed):
    # tiled coordinates where the material repeats, [0, 1) where it is clamped
    return _uniform(_gen(seed, 1), (case["n"], 2), 0.0, 4.0 if case["wrap"] else 1.0)


def _train_raw(case, seed):
    """Latents [h, w, 3], MLP, uv, and the target (a sum of 16 sinusoids and noise per channel) where there is one."""
    g = _gen(seed)
    sides = _level_sides(case["side"], case["side"])
    lat = [_normal(g, (h, w, 3), 0.1) for w, h in sides]
    ws, bs = _mlp(g, [12, 64, 64, C])
    uv = _uniform(g, (case["batch"], 2))
    target = None
    if case.get("target"):
        n = case["target"]
        x = (torch.arange(n, device="cuda", dtype=torch.float32) + 0.5) / n
        f, th, ph = _uniform(g, (C, 16), 1.0, 64.0), _uniform(g, (C, 16), 0.0, 2 * math.pi), _uniform(g, (C, 16), 0.0, 2 * math.pi)
        ax = 2 * math.pi * (f * th.cos())[..., None] * x
        by = 2 * math.pi * (f * th.sin())[..., None] * x + ph[..., None]
        waves = torch.einsum("cjy,cjx->yxc", by.cos(), ax.sin()) + torch.einsum("cjy,cjx->yxc", by.sin(), ax.cos())
        target = (0.5 + (0.5 / 16) * waves + _normal(g, (n, n, C), 0.02)).contiguous()
    dy = _normal(g, (case["batch"], C), 1.0) if case["kind"] == "autograd" else None
    return lat, ws, bs, uv, target, dy


def _qat_raw(case, seed):
    g = _gen(seed, 2)
    sides = _level_sides(case["side"], case["side"])
    return ([_normal(g, (h // 4, w // 4, 3), 1.0) for w, h in sides],
            [_normal(g, (h // 4, w // 4, 3), 1.0) for w, h in sides], [_normal(g, (h, w), 1.0) for w, h in sides])


def _batch_sizes(case):
    """Output sides of the materials: multiples of 128, spread log-uniformly over 256 .. smax, in no order of size."""
    n, lo, hi = case["materials"], math.log(256), math.log(case["smax"])
    at = [((7 * i + 3) % n + 0.5) / n if n % 7 else (i + 0.5) / n for i in range(n)]
    return [min(case["smax"], max(256, int(round(math.exp(lo + (hi - lo) * x) / 128.0)) * 128)) for x in at]


def _batch_raw(case, seed, mips):
    return [_raw_material(_gen(seed, 10 + i), _level_sides(s, s), [12, 64, 64, C], mips)
            for i, s in enumerate(_batch_sizes(case))]


def _frame_raw(case, seed):
    """Voronoi material ids (one region in sixteen without a material), tiled uv, lod, and derivatives stretched
    1x (top row) to 16x (bottom row) along a direction per material."""
    w, h, m = case["w"], case["h"], case["materials"]
    g = _gen(seed, 4)
    regions = m + max(1, m // 15)
    sx, sy = _uniform(g, (regions,), 0.0, w), _uniform(g, (regions,), 0.0, h)
    scale, phi = _uniform(g, (regions,), 1.0, 8.0), _uniform(g, (regions,), 0.0, math.pi)
    px = torch.arange(w, device="cuda", dtype=torch.float32) + 0.5
    py = torch.arange(h, device="cuda", dtype=torch.float32) + 0.5
    best = torch.full((h, w), math.inf, device="cuda")
    ids = torch.zeros((h, w), device="cuda", dtype=torch.int64)
    for k in range(regions):
        d = (py[:, None] - sy[k]) ** 2 + (px[None, :] - sx[k]) ** 2
        ids = torch.where(d < best, k, ids)
        best = torch.minimum(best, d)
    s = scale[ids]
    uv = torch.stack([s * px[None, :] / h, s * py[:, None] / h], dim=-1).contiguous()
    bias = _uniform(g, (h, w), 0.0, 3.0)
    mat_id = torch.where(ids < m, ids, -1).to(torch.int32).contiguous()
    if not case["aniso"]:
        return mat_id, uv, (bias + torch.log2(s / h)).contiguous(), None
    f, r = s / h, 1.0 + 15.0 * py[:, None] / h
    co, si = phi[ids].cos(), phi[ids].sin()
    duv = torch.stack([f * r * co, f * r * si, -f * si, f * co], dim=-1).contiguous()
    return mat_id, uv, torch.zeros_like(bias), duv


def prepare(case, seed):
    ctx, kind = _context(), case["kind"]
    if kind in ("grid", "uv"):
        mat, form = _material(_decode_raw(case, seed), case["wrap"]), FORMS[case["form"]]
        gw, gh = (case["w"], case["h"]) if kind == "grid" else (case["side"], case["side"])
        absmax = nb.fp8_calibrate(ctx, mat, gw, gh) if case["form"].startswith("e4m3") else None
        packed = None if form == nb.FP32 else nb.pack_mlp(ctx, mat, form, absmax)
        n = gw * gh if kind == "grid" else case["n"]
        out = torch.empty((n, C), device="cuda", dtype=torch.float32 if OUT_BYTES[case["form"]] == 4 else torch.float16)
        where = dict(grid=(gw, gh)) if kind == "grid" else dict(uv=_decode_uv(case, seed))
        return dict(kind=kind, ctx=ctx, mat=mat, form=form, packed=packed, where=where, out=out)
    if kind in ("train", "qat", "autograd"):
        lat, ws, bs, uv, target, dy = _train_raw(case, seed)
        wn, bn = [w.cpu().numpy() for w in ws], [b.cpu().numpy() for b in bs]
        if kind == "qat":
            e0, e1, alpha = ([t.cpu().numpy() for t in ts] for ts in _qat_raw(case, seed))
            model = QatModel(e0, e1, alpha, SHIFTS, wn, bn, latent_stride=case["stride"])
        else:
            model = ContinuousModel([l.cpu().numpy() for l in lat], SHIFTS, wn, bn, latent_stride=case["stride"])
        state = dict(kind=kind, ctx=ctx, model=model, uv=uv, dy=dy)
        if kind == "autograd":
            state["leaves"] = [t.detach().requires_grad_(True) for t in (*model.latents, model.weights, model.biases)]
        else:
            # the 4-float layout goes with a padded target, the 3-float one with the plain target
            state["target"] = padded(target) if case["stride"] == 4 else target
            state["loss"] = nb.LOSS_L1 if case["loss"] == "l1" else nb.LOSS_MSE
        return state
    frame = outs = None
    raws = _batch_raw(case, seed, mips=kind == "frame")
    mats = [_material(r, True) for r in raws]
    if kind == "batch":
        outs = [(torch.zeros((s * s, C), device="cuda", dtype=torch.float16), s, s) for s in _batch_sizes(case)]
    else:
        mat_id, uv, lod, duv = _frame_raw(case, seed)
        frame = dict(mat_id=mat_id, uv=uv, lod=lod,
                     out=torch.zeros((case["h"], case["w"], C), device="cuda", dtype=torch.float16))
        if duv is not None:
            frame.update(duv=duv, max_aniso=16)
    return dict(kind=kind, ctx=ctx, plan=nb.Batch(ctx, mats, outs, frame), outs=outs, frame=frame)


def run(state):
    kind, ctx = state["kind"], state["ctx"]
    if kind in ("grid", "uv"):
        return nb.decode(ctx, state["mat"], state["form"], state["packed"], out=state["out"], **state["where"])
    if kind == "autograd":
        leaves = state["leaves"]
        for t in leaves:
            t.grad = None
        y = NbtcDecodeFn.apply(ctx, state["model"], state["uv"], *leaves)
        y.backward(state["dy"])
        return dict(y=y.detach(), grads=[t.grad for t in leaves])
    if kind in ("train", "qat"):
        m = state["model"]
        loss = m.train_step(ctx, state["uv"], state["target"], loss=state["loss"])
        got = dict(loss=loss, grad_w=m.grad_w, grad_b=m.grad_b, latent_grads=m.latent_grads, weights=m.weights,
                   biases=m.biases)
        if kind == "train":
            got["latents"] = m.latents
        else:
            got.update(e0=m.e0, e1=m.e1, alpha=m.alpha, g_e0=m.g_e0, g_e1=m.g_e1, g_alpha=m.g_alpha)
        return got
    if kind == "batch":
        state["plan"].decode()
        return [t for t, _, _ in state["outs"]]
    state["plan"].render()
    return state["frame"]["out"]


# ------------------------------------------------------------------ work

def _mlp_flops(dims):
    return 2 * sum(i * o for i, o in zip(dims, dims[1:]))


def _mlp_bytes(dims):
    return 4 * sum(i * o + o for i, o in zip(dims, dims[1:]))


def _level_bytes(sides, mips=False):
    """Blocks of the levels, 8 bytes each; the mips add about a third."""
    return sum(w * h // 2 for w, h in sides) * (4 / 3 if mips else 1.0)


def work(case):
    kind = case["kind"]
    if kind in ("grid", "uv"):
        dims = _dims(case)
        n = case["w"] * case["h"] if kind == "grid" else case["n"]
        sides = _level_sides(case["w"], case["h"]) if kind == "grid" else _level_sides(case["side"], case["side"])
        # a short list of coordinates touches at most 4 blocks a level and sample
        blocks = _level_bytes(sides) if kind == "grid" else min(_level_bytes(sides), n * 4 * 4 * 8)
        return dict(bytes=blocks + _mlp_bytes(dims) + n * (C * OUT_BYTES[case["form"]] + (8 if kind == "uv" else 0)),
                    flops=n * _mlp_flops(dims))
    dims = [12, 64, 64, C]
    if kind in ("train", "qat", "autograd"):
        b, texels = case["batch"], sum(w * h for w, h in _level_sides(case["side"], case["side"]))
        # backward: the weights' and the inputs' products; the autograd function recomputes nothing it must
        flops = 3 * b * _mlp_flops(dims)
        if kind == "autograd":  # uv and dy in, y out, latents in, their gradients out
            return dict(bytes=b * (8 + 8 * C) + 24 * texels, flops=flops)
        target = min(case["target"] ** 2, 4 * b) * C * 4
        if kind == "train":  # latents and both moments read and written, the gradient written
            return dict(bytes=b * 8 + target + 12 * texels * 7, flops=flops)
        # per texel alpha and its moments read and written, its gradient and dL/dT written; per block 6 endpoints likewise
        return dict(bytes=b * 8 + target + texels * (28 + 12) + texels / 16 * 6 * 28, flops=flops)
    if kind == "batch":
        n = sum(s * s for s in _batch_sizes(case))
        return dict(bytes=n * 2 * C + n * (1 / 16 + 1 / 64 + 1 / 256 + 1 / 1024) / 2, flops=n * _mlp_flops(dims))
    n = case["w"] * case["h"] * (1 - 1 / 16)
    per = 4 + 8 + 4 + 2 * C + (16 if case["aniso"] else 0)
    return dict(bytes=n * per, flops=n * _mlp_flops(dims))


# ------------------------------------------------------------------ 64-bit values

def _bc1_texels(blocks, w, h):
    """One mip's RGB in [0, 1], [h, w, 3] FP64: endpoints widened by bit replication, thirds (or halves) rounded to
    nearest, index 3 of a three-colour block black."""
    b = blocks.view(h // 4, w // 4)
    c0, c1, bits = b & 0xFFFF, (b >> 16) & 0xFFFF, (b >> 32) & 0xFFFFFFFF

    def widen(c):
        r, g, bl = (c >> 11) & 31, (c >> 5) & 63, c & 31
        return torch.stack([(r << 3) | (r >> 2), (g << 2) | (g >> 4), (bl << 3) | (bl >> 2)], dim=-1)

    e0, e1, four = widen(c0), widen(c1), (c0 > c1)[..., None]
    third = torch.where(four, (2 * e0 + e1 + 1) // 3, (e0 + e1 + 1) // 2)
    fourth = torch.where(four, (e0 + 2 * e1 + 1) // 3, torch.zeros_like(e0))
    palette = torch.stack([e0, e1, third, fourth], dim=-2)                     # [hb, wb, 4, 3]
    at = torch.arange(16, device=b.device)
    idx = (bits[..., None] >> (2 * at)) & 3                                    # [hb, wb, 16]
    rgb = torch.gather(palette, 2, idx[..., None].expand(*idx.shape, 3))       # [hb, wb, 16, 3]
    rgb = rgb.view(h // 4, w // 4, 4, 4, 3).permute(0, 2, 1, 3, 4).reshape(h, w, 3)
    return rgb.to(torch.float64) / 255.0


def _level_mips(level):
    blocks, w, h, mips, _ = level
    out, at = [], 0
    for m in range(mips):
        wm, hm = max(4, w >> m), max(4, h >> m)
        n = (wm // 4) * (hm // 4)
        out.append(_bc1_texels(blocks[at:at + n], wm, hm))
        at += n
    return out


def _axis(u, n, shift, wrap):
    """Neighbours and weight along one axis of FP32 coordinates u."""
    if wrap:
        u = u - u.floor()
    t = (u.double() * n + (shift - 0.5)).float()
    if not wrap:
        t = t.clamp(-1.0, float(n))
    fl = t.floor()
    a = fl.long()
    if wrap:
        return a % n, (a + 1) % n, (t - fl).double()
    return a.clamp(0, n - 1), (a + 1).clamp(0, n - 1), (t - fl).double()


def _bilinear_at(img, u, v, shift, wrap):
    """(flat indices, weights) of the four taps of img [h, w, c] at FP32 (u, v)."""
    h, w = img.shape[:2]
    xa, xb, fx = _axis(u, w, shift, wrap)
    ya, yb, fy = _axis(v, h, shift, wrap)
    return ((ya * w + xa, (1 - fx) * (1 - fy)), (ya * w + xb, fx * (1 - fy)),
            (yb * w + xa, (1 - fx) * fy), (yb * w + xb, fx * fy))


def _bilinear(img, u, v, shift, wrap):
    flat = img.reshape(-1, img.shape[-1])
    return sum(wt[:, None] * flat[i] for i, wt in _bilinear_at(img, u, v, shift, wrap))


def _forward(x, ws, bs):
    for l, (w, b) in enumerate(zip(ws, bs)):
        x = x @ w.double().T + b.double()
        if l + 1 < len(ws):
            x = x.relu()
    return x


def _chunks(n, size=1 << 20):
    for i in range(0, n, size):
        yield i, min(n, i + size)


def _grid_coords(i, n):
    return ((i.double() + 0.5) / n).float()


def _exact_decode(case, seed):
    levels, ws, bs = _decode_raw(case, seed)
    imgs, wrap = [_level_mips(lv)[0] for lv in levels], case["wrap"]
    uv = _decode_uv(case, seed) if case["kind"] == "uv" else None
    n = case["n"] if uv is not None else case["w"] * case["h"]
    out = torch.empty((n, C), device="cuda", dtype=torch.float64)
    for a, b in _chunks(n):
        if uv is not None:
            u, v = uv[a:b, 0], uv[a:b, 1]
        else:
            t = torch.arange(a, b, device="cuda")
            u, v = _grid_coords(t % case["w"], case["w"]), _grid_coords(t // case["w"], case["h"])
        x = torch.cat([_bilinear(img, u, v, lv[4], wrap) for img, lv in zip(imgs, levels)], dim=-1)
        out[a:b] = _forward(x, ws, bs)
    return out


def _exact_batch(case, seed):
    outs = []
    for s, (levels, ws, bs) in zip(_batch_sizes(case), _batch_raw(case, seed, False)):
        imgs = [_level_mips(lv)[0] for lv in levels]
        out = torch.empty((s * s, C), device="cuda", dtype=torch.float64)
        for a, b in _chunks(s * s):
            t = torch.arange(a, b, device="cuda")
            u, v = _grid_coords(t % s, s), _grid_coords(t // s, s)
            x = torch.cat([_bilinear(img, u, v, lv[4], True) for img, lv in zip(imgs, levels)], dim=-1)
            out[a:b] = _forward(x, ws, bs)
        outs.append(out)
    return outs


def _trilinear(mips, w0, u, v, lod, shift):
    lam = (lod + math.log2(w0)).clamp(0.0, float(len(mips) - 1))
    m0 = lam.floor().long()
    m1, t = (m0 + 1).clamp(max=len(mips) - 1), lam - m0
    out = torch.zeros((len(u), 3), device=u.device, dtype=torch.float64)
    for m, img in enumerate(mips):
        wt = torch.where(m0 == m, 1 - t, 0.0) + torch.where(m1 == m, t, 0.0)
        sel = wt.nonzero()[:, 0]
        if len(sel):
            out[sel] += wt[sel, None] * _bilinear(img, u[sel], v[sel], shift, True)
    return out


def _exact_frame(case, seed):
    mat_id, uv, lod, duv = _frame_raw(case, seed)
    ids, uv, lod = mat_id.reshape(-1), uv.reshape(-1, 2), lod.reshape(-1)
    out = torch.zeros((len(ids), C), device="cuda", dtype=torch.float64)
    for m, (levels, ws, bs) in enumerate(_batch_raw(case, seed, True)):
        px = (ids == m).nonzero()[:, 0]
        if not len(px):
            continue
        mips = [_level_mips(lv) for lv in levels]
        for a, b in _chunks(len(px)):
            p = px[a:b]
            u, v, base = uv[p, 0], uv[p, 1], lod[p].double()
            if duv is None:
                x = torch.cat([_trilinear(mp, lv[1], u, v, base, lv[4]) for mp, lv in zip(mips, levels)], dim=-1)
            else:
                # the number of probes is decided in FP32: products, sums, roots and the quotient rounded one by one
                d = duv.reshape(-1, 4)[p]
                dx, dy = (d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]).sqrt(), (d[:, 2] * d[:, 2] + d[:, 3] * d[:, 3]).sqrt()
                along = dx >= dy
                big, small = torch.where(along, dx, dy), torch.where(along, dy, dx)
                n = (big / small).ceil().clamp(max=16.0)
                au, av = torch.where(along, d[:, 0], d[:, 2]).double(), torch.where(along, d[:, 1], d[:, 3]).double()
                base = base + (big.double() / n.double()).log2()
                x = torch.zeros((len(p), 12), device="cuda", dtype=torch.float64)
                for i in range(1, int(n.max()) + 1):
                    s = (n >= i).nonzero()[:, 0]
                    off = (float(i) / (n[s] + 1) - 0.5).double()
                    uu, vv = (u[s].double() + off * au[s]).float(), (v[s].double() + off * av[s]).float()
                    x[s] += torch.cat([_trilinear(mp, lv[1], uu, vv, base[s], lv[4]) for mp, lv in zip(mips, levels)], dim=-1)
                x /= n.double()[:, None]
            out[p] = _forward(x, ws, bs)
    return out.reshape(case["h"], case["w"], C)


def _adam(p, g, lr, eps=1e-8):
    """The first Adam step: the bias-corrected moments are g and g^2."""
    return p.double() - lr * g / (g.abs() + eps)


def _exact_train(case, seed):
    kind = case["kind"]
    lat, ws, bs, uv, target, dy = _train_raw(case, seed)
    if kind == "qat":
        e0, e1, alpha = _qat_raw(case, seed)

        def levels(p, n):  # the nearest of n + 1 levels of sigmoid(p), decided by FP32 thresholds
            t = torch.tensor([math.log(((j + 0.5) / n) / (1 - (j + 0.5) / n)) for j in range(n)], device="cuda").float()
            return torch.bucketize(p, t, right=True).double() / n

        def spread(e):  # [h/4, w/4, 3] -> [h, w, 3]
            return e.repeat_interleave(4, 0).repeat_interleave(4, 1)

        def ends(e):
            return torch.stack([levels(e[..., 0].contiguous(), 31), levels(e[..., 1].contiguous(), 63),
                                levels(e[..., 2].contiguous(), 31)], dim=-1)

        blend = [levels(a, 3)[..., None] for a in alpha]
        q0, q1 = [spread(ends(e)) for e in e0], [spread(ends(e)) for e in e1]
        lat = [(1 - a) * x + a * y for a, x, y in zip(blend, q0, q1)]
    lat = [l.double().requires_grad_(True) for l in lat]
    ws, bs = [w.double().requires_grad_(True) for w in ws], [b.double().requires_grad_(True) for b in bs]
    n = case["batch"]
    loss, ys = 0.0, []
    for a, b in _chunks(n, 1 << 18):
        u, v = uv[a:b, 0], uv[a:b, 1]
        x = torch.cat([_bilinear(l, u, v, s, False) for l, s in zip(lat, SHIFTS)], dim=-1)
        y = _forward(x, ws, bs)
        if kind == "autograd":
            ys.append(y.detach())
            y.backward(dy[a:b].double())
            continue
        d = y - _bilinear(target.double(), u, v, 0.0, False)
        part = (d.abs() if case["loss"] == "l1" else d.square()).sum() / (n * C)
        part.backward()
        loss += float(part.detach())
    cat = lambda ts: torch.cat([t.detach().reshape(-1) for t in ts])  # noqa: E731
    gw, gb, gl = cat([w.grad for w in ws]), cat([b.grad for b in bs]), [l.grad for l in lat]
    if kind == "autograd":
        return dict(y=torch.cat(ys), grads=[*gl, gw, gb])
    got = dict(loss=torch.tensor([loss], dtype=torch.float64), grad_w=gw, grad_b=gb, latent_grads=gl,
               weights=_adam(cat(ws), gw, 1e-3), biases=_adam(cat(bs), gb, 1e-3))
    if kind == "train":
        got["latents"] = [_adam(l.detach(), g, 1e-2) for l, g in zip(lat, gl)]
        return got

    def slope(p):
        s = p.double().sigmoid()
        return s * (1 - s)

    def per_block(t):  # [h, w, 3] summed over 4x4 blocks
        h, w = t.shape[:2]
        return t.reshape(h // 4, 4, w // 4, 4, 3).sum(dim=(1, 3))

    g0 = [per_block(g * (1 - a)) * slope(e) for g, a, e in zip(gl, blend, e0)]
    g1 = [per_block(g * a) * slope(e) for g, a, e in zip(gl, blend, e1)]
    ga = [(g * (y - x)).sum(-1) * slope(p) for g, x, y, p in zip(gl, q0, q1, alpha)]
    got.update(g_e0=g0, g_e1=g1, g_alpha=ga, e0=[_adam(p, g, 1e-2) for p, g in zip(e0, g0)],
               e1=[_adam(p, g, 1e-2) for p, g in zip(e1, g1)], alpha=[_adam(p, g, 1e-2) for p, g in zip(alpha, ga)])
    return got


def exact(case, seed):
    kind = case["kind"]
    if kind in ("grid", "uv"):
        return _exact_decode(case, seed)
    if kind in ("train", "qat", "autograd"):
        return _exact_train(case, seed)
    return _exact_batch(case, seed) if kind == "batch" else _exact_frame(case, seed)
