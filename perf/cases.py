"""Cases of the framework's performance: what its users have it do.

Every case goes through a public entry point of ``paper_2312_00229_gb300.api``
(arXiv 2312.00229: the 2x zoom and its adjoint, the batched form, the cascade,
tensor-WENO resampling and the zoom to any size).  Frames that live in host
memory (``api.HostPipeline``) run the same kernel as the frames here; the host
copies around it bound them, so they are timed end to end by ``bench.py``.

``listed`` gives the cases, ``draw`` one more of the same ranges, ``prepare``
the inputs on the GPU, ``run`` one pass, ``work`` the bytes and operations it
cannot do without, ``exact`` the floating outputs in 64 bits.
"""
from __future__ import annotations

import math
import random

import torch
import torch.nn.functional as F

from paper_2312_00229_gb300 import api

_DTYPES = {"u8": torch.uint8, "f16": torch.float16, "bf16": torch.bfloat16, "f32": torch.float32}
_BYTES = {"u8": 1, "f16": 2, "bf16": 2, "f32": 4}

# FP32 operations the method needs (beta = 2; differences shared between
# neighbouring stencils): per input sample and channel of a 2x zoom, and per
# output sample of the separable tensor interpolation (28 per 1-D interpolant).
_ZOOM_OPS = 162
_SPLINE_OPS = 28


def listed():
    return [
        # a sprite or an icon: the smallest calls, where launch latency counts
        dict(name="sprite_u8", kind="zoom", dtype="u8", layout="chw", planes=3, h=48, w=64,
             beta=2.0, out_mode=0, art=True),
        # one decoded full-HD picture, pixels interleaved as decoders give them
        dict(name="hd_interleaved_u8", kind="zoom", dtype="u8", layout="hwc", planes=3, h=1080,
             w=1920, beta=2.0, out_mode=0, art=False),
        # one UHD video frame, planar: the benchmark's frame
        dict(name="uhd_u8", kind="zoom", dtype="u8", layout="chw", planes=3, h=2160, w=3840,
             beta=2.0, out_mode=0, art=False),
        # a photograph of odd sides in a model's storage type
        dict(name="photo_bf16", kind="zoom", dtype="bf16", layout="chw", planes=3, h=1367, w=2049,
             beta=2.0, out_mode=0, art=False),
        # a sampled field on the 2n-1 grid with beta = 1, the other exponent
        # the method's authors use
        dict(name="field_f32", kind="zoom", dtype="f32", layout="chw", planes=1, h=1025, w=1025,
             beta=1.0, out_mode=1, art=False),
        # the zoom as a layer of a training step: forward and adjoint on a batch
        dict(name="train_f32", kind="train", dtype="f32", batch=32, planes=3, h=512, w=512),
        # one step of an inverse problem on one image
        dict(name="inverse_f32", kind="train", dtype="f32", batch=1, planes=3, h=256, w=256),
        # a folder of pictures of different sizes in one launch
        dict(name="folder_f16", kind="batch", dtype="f16", planes=3, count=64, lo=64, hi=1024,
             sides=1),
        # pixel art enlarged eight times
        dict(name="art_8x_u8", kind="cascade", dtype="u8", planes=3, h=512, w=512, levels=3),
        # a full-HD picture to three times its size: doublings, then resampling
        dict(name="hd_to_3x_u8", kind="zoom_to", dtype="u8", planes=3, h=1080, w=1920, oh=3240,
             ow=5760),
        # the tensor interpolation alone: the same enlargement
        dict(name="resample_3x_u8", kind="resample", dtype="u8", planes=3, h=1080, w=1920, oh=3240,
             ow=5760),
        # and a preview of a quarter of the sides
        dict(name="preview_u8", kind="resample", dtype="u8", planes=3, h=1080, w=1920, oh=270,
             ow=480),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["zoom", "zoom", "zoom", "train", "batch", "cascade", "zoom_to", "resample"])
    dtype = rng.choice(["u8", "u8", "f16", "bf16", "f32"])
    planes = rng.choice([1, 3, 3])
    if kind == "zoom":
        layout = rng.choice(["chw", "chw", "hwc"]) if planes == 3 else "chw"
        return dict(kind=kind, dtype=dtype, layout=layout, planes=planes, h=_log(rng, 32, 2160),
                    w=_log(rng, 32, 3840), beta=rng.choice([2.0, 2.0, 1.0]),
                    out_mode=rng.choice([0, 0, 1]), art=rng.random() < 0.3)
    if kind == "train":
        return dict(kind=kind, dtype="f32", batch=_log(rng, 1, 32), planes=planes,
                    h=_log(rng, 64, 512), w=_log(rng, 64, 512))
    if kind == "batch":
        lo = _log(rng, 48, 256)
        return dict(kind=kind, dtype=dtype, planes=planes, count=_log(rng, 4, 64), lo=lo,
                    hi=min(1024, lo * rng.randint(2, 8)), sides=rng.randint(1, 1 << 20))
    if kind == "cascade":
        return dict(kind=kind, dtype=dtype, planes=planes, h=_log(rng, 48, 512),
                    w=_log(rng, 48, 512), levels=rng.choice([2, 3]))
    h, w = _log(rng, 96, 1080), _log(rng, 96, 1920)
    f = rng.uniform(1.2, 3.0) if kind == "zoom_to" else math.exp(rng.uniform(math.log(0.2),
                                                                            math.log(3.0)))
    return dict(kind=kind, dtype=dtype, planes=planes, h=h, w=w, oh=max(2, round(h * f)),
                ow=max(2, round(w * f)))


# ---- inputs ---------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _uniform(g, shape, lo=0.0, hi=1.0):
    return torch.rand(shape, generator=g, device="cuda") * (hi - lo) + lo


def _scene(g, planes, h, w):
    """Smooth shading, hard-edged half planes and sensor noise, in [0, 1]."""
    y = torch.arange(h, device="cuda", dtype=torch.float32).view(1, h, 1)
    x = torch.arange(w, device="cuda", dtype=torch.float32).view(1, 1, w)
    img = torch.full((planes, h, w), 0.5, device="cuda")
    for k in range(6):
        f = _uniform(g, (planes, 1, 1, 3), -0.04, 0.04)
        img += 0.07 * torch.sin(f[..., 0] * x + f[..., 1] * y + 80.0 * f[..., 2])
    for k in range(6):
        a = float(_uniform(g, (1,), 0.0, 2 * math.pi))
        d = float(_uniform(g, (1,), 0.2, 0.8))
        c = _uniform(g, (planes, 1, 1), -0.15, 0.15)
        side = math.cos(a) * (x - d * w) + math.sin(a) * (y - d * h)
        img += c * (side > 0)
    img += (2.0 / 255.0) * torch.randn((planes, h, w), generator=g, device="cuda")
    return img.clamp_(0.0, 1.0)


def _art(g, planes, h, w):
    """Blocks of a palette of 16 colours and one-pixel diagonals."""
    palette = _uniform(g, (16, planes))
    blocks = torch.randint(0, 16, ((h + 7) // 8, (w + 7) // 8), generator=g, device="cuda")
    idx = blocks.repeat_interleave(8, 0).repeat_interleave(8, 1)[:h, :w].clone()
    y = torch.arange(h, device="cuda").view(h, 1)
    x = torch.arange(w, device="cuda").view(1, w)
    idx[((x + y) % 37) == 0] = 3
    idx[((2 * x - y) % 53) == 0] = 11
    return palette[idx].permute(2, 0, 1).contiguous()


def _store(img, dtype):
    if dtype == "u8":
        return (img * 255.0).round().to(torch.uint8)
    return img.to(_DTYPES[dtype])


def _sides(case):
    """Sides of a folder's pictures, uniform in [lo, hi]: part of the case."""
    rng = random.Random(case["sides"])
    return [(rng.randint(case["lo"], case["hi"]), rng.randint(case["lo"], case["hi"]))
            for _ in range(case["count"])]


def _images(case, seed):
    """The stored input images of a case."""
    g = _gen(seed)
    kind, p = case["kind"], case["planes"]
    if kind == "train":
        n = case["batch"] * p
        x = _scene(g, n, case["h"], case["w"]).view(case["batch"], p, case["h"], case["w"])
        go = torch.randn((case["batch"], p, 2 * case["h"], 2 * case["w"]), generator=g,
                         device="cuda")
        return [x, go]
    if kind == "batch":
        return [_store((_art if i % 2 else _scene)(g, p, h, w), case["dtype"])
                for i, (h, w) in enumerate(_sides(case))]
    art = case.get("art", kind == "cascade")
    img = _store((_art if art else _scene)(g, p, case["h"], case["w"]), case["dtype"])
    if case.get("layout") == "hwc":
        img = img.permute(1, 2, 0).contiguous()
    return [img]


def prepare(case, seed):
    imgs = _images(case, seed)
    state = {"case": case, "x": imgs[0]}
    kind = case["kind"]
    if kind == "zoom":
        state["params"] = api.Params(beta=case["beta"], out_mode=case["out_mode"])
    elif kind == "train":
        state["x"].requires_grad_(True)
        state["grad_out"] = imgs[1]
    elif kind == "batch":
        # the folder's plan: descriptors, outputs and workspace on the device
        state["plan"] = api.BatchedPlan(imgs)
    return state


def run(state):
    case, x = state["case"], state["x"]
    kind = case["kind"]
    if kind == "zoom":
        return api.zoom2x(x, state["params"], layout=case["layout"])
    if kind == "train":
        y = api.zoom2x(x)
        (gx,) = torch.autograd.grad(y, x, state["grad_out"])
        return [y.detach(), gx]
    if kind == "batch":
        return state["plan"].run()
    if kind == "cascade":
        return api.cascade_zoom(x, case["levels"])
    if kind == "zoom_to":
        return api.zoom_to(x, case["oh"], case["ow"])
    return api.resample(x, case["oh"], case["ow"])


def work(case):
    kind, p, e = case["kind"], case["planes"], _BYTES[case["dtype"]]
    if kind == "batch":
        n_in = float(p * sum(h * w for h, w in _sides(case)))
        return {"bytes": 5.0 * e * n_in, "flops": float(_ZOOM_OPS * n_in)}
    n_in = float(p * case["h"] * case["w"])
    if kind == "zoom":
        return {"bytes": 5.0 * e * n_in, "flops": _ZOOM_OPS * n_in}
    if kind == "train":
        n_in *= case["batch"]
        # input and output of the forward; input, output gradient and input
        # gradient of the adjoint, which does the forward's work and about
        # twice that again
        return {"bytes": 5.0 * e * n_in + 6.0 * e * n_in, "flops": 4.0 * _ZOOM_OPS * n_in}
    if kind == "cascade":
        lv = case["levels"]
        return {"bytes": e * n_in * (1 + 4.0 ** lv),
                "flops": _ZOOM_OPS * n_in * sum(4.0 ** k for k in range(lv))}
    n_out = float(p * case["oh"] * case["ow"])
    # a reduction reads 4 x 4 samples an output at most
    n_read = min(n_in, 16.0 * n_out)
    # columns first: one interpolant per output row and input column it reads
    cols = min(case["w"], 4 * case["ow"])
    spline = _SPLINE_OPS * (n_out + p * case["oh"] * float(cols))
    if kind == "resample":
        return {"bytes": e * (n_read + n_out), "flops": spline}
    n, m, ops = case["h"], case["w"], 0.0
    while n < case["oh"] or m < case["ow"]:
        ops += _ZOOM_OPS * p * n * m
        n, m = 2 * n - 1, 2 * m - 1
    return {"bytes": e * (n_in + n_out), "flops": ops + _SPLINE_OPS * (n_out + p * case["oh"] * m)}


# ---- 64-bit values ----------------------------------------------------------------
def _value64(img):
    """Stored samples as the method reads them (8-bit codes are u / 255)."""
    return img.double() / 255.0 if img.dtype == torch.uint8 else img.double()


_KAPPA2 = 13.0 / 12.0


def _zoom64(a, beta=2.0, out_mode=0, h=1.0, k_eps=1e-8, nbr_c=0.125):
    """The 2x zoom of planes [N, n, m] in 64 bits, differentiable."""
    n, m = a.shape[-2:]
    pad = 6  # an output reads 4 samples before and 5 after it
    e = F.pad(a.unsqueeze(0), (pad, pad, pad, pad), mode="replicate").squeeze(0)
    eps, w = k_eps * h * h, nbr_c * h * h

    def at(t, dr, dc):
        return t.roll((-dr, -dc), (-2, -1))

    def directions(stencils):
        si, ip = [], []
        for n0, n1, n2 in stencils:
            g, s = n1 - n0, n0 - 2.0 * n1 + n2
            si.append(g * g + _KAPPA2 * s * s)
            ip.append(0.375 * n0 + 0.75 * n1 - 0.125 * n2)
        return si, ip

    def blend(si, nbrs, ip):
        num = den = 0.0
        for k in range(4):
            d = si[k] + w * sum(at(src[k], dr, dc) for src, dr, dc in nbrs)
            al = (eps + d) ** (-beta)
            num, den = num + al * ip[k], den + al
        return num / den

    si, ip = directions([
        (e, at(e, 1, 1), at(e, 2, 2)), (at(e, 1, 1), e, at(e, -1, -1)),
        (at(e, 0, 1), at(e, 1, 0), at(e, 2, -1)), (at(e, 1, 0), at(e, 0, 1), at(e, -1, 2))])
    x = blend(si, [(si, -1, 0), (si, 1, 0), (si, 0, -1), (si, 0, 1)], ip)
    si_e, ip_e = directions([
        (e, at(e, 0, 1), at(e, 0, 2)), (at(e, 0, 1), e, at(e, 0, -1)),
        (at(x, -1, 0), x, at(x, 1, 0)), (x, at(x, -1, 0), at(x, -2, 0))])
    si_s, ip_s = directions([
        (at(x, 0, -1), x, at(x, 0, 1)), (x, at(x, 0, -1), at(x, 0, -2)),
        (e, at(e, 1, 0), at(e, 2, 0)), (at(e, 1, 0), e, at(e, -1, 0))])
    ve = blend(si_e, [(si_s, -1, 0), (si_s, 0, 0), (si_s, -1, 1), (si_s, 0, 1)], ip_e)
    vs = blend(si_s, [(si_e, 0, -1), (si_e, 0, 0), (si_e, 1, -1), (si_e, 1, 0)], ip_s)

    def crop(t):
        return t[..., pad:pad + n, pad:pad + m]

    top = torch.stack([crop(e), crop(ve)], -1)
    bottom = torch.stack([crop(vs), crop(x)], -1)
    u = torch.stack([top, bottom], -3).reshape(a.shape[0], 2 * n, 2 * m)
    return u[..., :2 * n - 1, :2 * m - 1] if out_mode else u


def _spline64(a, n_out, eps):
    """1-D WENO interpolation along the last axis to n_out aligned samples."""
    n = a.shape[-1]
    if n == 1:
        return a.expand(*a.shape[:-1], n_out)
    j = torch.arange(n_out, device=a.device, dtype=torch.int64)
    den = max(n_out - 1, 1)
    i = torch.clamp(j * (n - 1) // den, max=n - 2)
    t = (j * (n - 1) - i * den).double() / den
    v = [a[..., (i + d).clamp(0, n - 1)] for d in (-1, 0, 1, 2)]
    g, sl, sr = v[2] - v[1], v[0] - 2 * v[1] + v[2], v[1] - 2 * v[2] + v[3]
    al = (2 - t) / 3 / (eps + g * g + _KAPPA2 * sl * sl) ** 2
    ar = (1 + t) / 3 / (eps + g * g + _KAPPA2 * sr * sr) ** 2
    return v[1] + g * t + (t * t - t) / 2 * (al * sl + ar * sr) / (al + ar)


def _resample64(a, oh, ow, h=1.0):
    eps = 1e-8 * h * h
    z = _spline64(a.transpose(-1, -2), oh, eps).transpose(-1, -2)
    return _spline64(z, ow, eps)


def exact(case, seed):
    if case["dtype"] == "u8":  # codes: rounded, no 64-bit values
        return None
    kind = case["kind"]
    imgs = _images(case, seed)
    if kind == "train":
        x, go = imgs
        n, m = case["h"], case["w"]
        xs, gs = x.view(-1, n, m), go.view(-1, 2 * n, 2 * m)
        y, gx = [], []
        step = max(1, (1 << 21) // (n * m))  # planes at a time
        for k in range(0, xs.shape[0], step):
            a = xs[k:k + step].double().requires_grad_(True)
            u = _zoom64(a)
            gx += torch.autograd.grad(u, a, gs[k:k + step].double())
            y.append(u.detach())
        return [torch.cat(y).view(go.shape), torch.cat(gx).view(x.shape)]
    if kind == "batch":
        return [_zoom64(_value64(im)) for im in imgs]
    a = imgs[0]
    if case.get("layout") == "hwc":
        u = _zoom64(_value64(a.permute(2, 0, 1)), case["beta"], case["out_mode"])
        return u.permute(1, 2, 0)
    a = _value64(a)
    if kind == "zoom":
        return _zoom64(a, case["beta"], case["out_mode"])
    if kind == "cascade":
        for k in range(case["levels"]):
            a = _zoom64(a, h=0.5 ** k)
        return a
    k = 0
    if kind == "zoom_to":
        while a.shape[-2] < case["oh"] or a.shape[-1] < case["ow"]:
            a, k = _zoom64(a, out_mode=1, h=0.5 ** k), k + 1
    return _resample64(a, case["oh"], case["ow"], h=0.5 ** k)
