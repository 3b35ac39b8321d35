"""The work that users of the framework have it do, as cases to be timed and compared.

Three groups, over the range of sizes that the bench and the tests of this
repository use (256x256 / 2,000 Gaussians up to 2040x1356 / 200,000):

* ``fit``: one training step of a `Fit` context (formation, binning, render
  and loss, backward, optimiser), in the forms the library offers;
* ``render`` / ``decode_render`` / ``vq``: the forward-only pass of a viewer
  or a decoder (`Renderer`, `codec_decode`, `vq_decode`);
* ``autograd``: `rasterize` inside a PyTorch program, forward and backward.

Images, Gaussians, codebooks and upstream gradients are drawn on the GPU from
the seed with the distributions of the repository's synthetic workloads.
"""
from __future__ import annotations

import math
import random

import torch

import paper_2403_08551_gb300 as gi

LR = (1e-3, 1e-2, 1e-2)        # the workload's Adam rates: positions, covariance, colour
LR_PAPER = (1e-3, 1e-3, 1e-3)  # the paper's recipe (Adan)
ADAN = (0.98, 0.92, 0.99)      # its decay factors, the library's defaults
BATCH_SHAPES = ((256, 256), (512, 384), (768, 512), (1024, 768))


def listed():
    return [
        # a small image: a step is a handful of short launches
        dict(name="fit_256x256_2k", kind="fit", W=256, H=256, n=2000, T=16, mode="plain"),
        # the headline workload: a Kodak-shaped image and 70,000 Gaussians
        dict(name="fit_768x512_70k", kind="fit", W=768, H=512, n=70000, T=16, mode="plain"),
        # a full-size DIV2K-shaped image, 30 % of the Gaussians in 10 % of the area
        dict(name="fit_2040x1356_200k", kind="fit", W=2040, H=1356, n=200000, T=16, mode="plain", skew=True),
        # images of uneven sizes fitted together, Gaussians in proportion to their pixels
        dict(name="fit_batch16", kind="fit", images=16, shapes=3000, T=16, mode="plain"),
        # the paper's own parameters and optimiser (tanh positions, Adan)
        dict(name="fit_paper_768x512_70k", kind="fit", W=768, H=512, n=70000, T=16, mode="paper"),
        # quantisation-aware fine-tuning of the codec, the paper's 6 bits and 2 x 8 entries
        dict(name="fit_codec_768x512_70k", kind="fit", W=768, H=512, n=70000, T=16, mode="codec", size=8),
        # the alpha-blending form of the ablation at its 30,000 Gaussians
        dict(name="fit_blend_768x512_30k", kind="fit", W=768, H=512, n=30000, T=16, mode="blend"),
        # a differentiable render in a PyTorch program, an odd image and count
        dict(name="autograd_517x389_20011", kind="autograd", W=517, H=389, n=20011, T=16),
        # a viewer's frame
        dict(name="render_768x512_70k", kind="render", W=768, H=512, n=70000, T=16),
        dict(name="render_2040x1356_100k", kind="render", W=2040, H=1356, n=100000, T=16, skew=True),
        # decoding a stored image: codec stream to pixels
        dict(name="decode_render_768x512_50k", kind="decode_render", W=768, H=512, n=50000, T=16, size=8),
        # the attribute decode of a whole batch of images
        dict(name="vq_decode_3m2", kind="vq", n=3200000, size=256, stages=2),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(("fit", "fit", "fit", "autograd", "render", "decode_render", "vq"))
    if kind == "vq":
        n = int(_log(rng, 20000, 3200000))
        return dict(kind=kind, n=n - n % 4 if rng.random() < 0.5 else n, size=rng.choice((8, 64, 256)),
                    stages=rng.choice((1, 2, 3)))
    pixels = _log(rng, 256 * 256, 2040 * 1356)
    aspect = rng.uniform(0.7, 1.6)
    W, H = int(math.sqrt(pixels * aspect)), int(math.sqrt(pixels / aspect))
    n = int(max(500, min(200000, W * H * _log(rng, 0.03, 0.2))))
    if kind == "fit" and rng.random() < 0.2:
        return dict(kind=kind, images=rng.randint(2, 12), shapes=rng.randint(1, 1 << 20), T=16, mode="plain")
    case = dict(kind=kind, W=W, H=H, n=n, T=16)
    if kind == "fit":
        mode = rng.choice(("plain", "plain", "plain", "paper", "rs", "paper_rs", "codec", "separate", "blend"))
        case["mode"] = mode
        if mode == "plain":
            case["T"] = rng.choice((8, 16, 16, 32))
        if mode == "codec":
            case["size"] = rng.choice((8, 16, 256))
        if mode == "codec" or mode == "blend":  # kept to the sizes of the bench
            case["W"], case["H"], case["n"] = min(W, 1024), min(H, 768), min(n, 70000)
    elif kind == "decode_render":
        case["size"] = rng.choice((8, 64, 256))
    if kind != "decode_render" and case.get("mode", "plain") == "plain" and rng.random() < 0.3:
        case["skew"] = True
    return case


# --------------------------------------------------------------------------- inputs

def _image(W, H, g):
    """A smooth image with sharper detail on top, values in [0, 1]."""
    up = torch.nn.functional.interpolate
    coarse = torch.rand((1, 3, H // 64 + 2, W // 64 + 2), generator=g, device="cuda")
    fine = torch.rand((1, 3, H // 8 + 2, W // 8 + 2), generator=g, device="cuda") - 0.5
    x = up(coarse, size=(H, W), mode="bicubic", align_corners=False)
    x = 0.15 + 0.7 * x + 0.3 * up(fine, size=(H, W), mode="bilinear", align_corners=False)
    return x[0].permute(1, 2, 0).clamp(0, 1).contiguous()


def _uni(shape, lo, hi, g):
    return torch.rand(shape, generator=g, device="cuda") * (hi - lo) + lo


def _gaussians(W, H, n, g, skew=False):
    """Pixel-space parameters [n, 8]: position, Cholesky vector, colour."""
    x, y = _uni((n,), 0, W, g), _uni((n,), 0, H, g)
    if skew:
        k = int(0.3 * n)
        rw, rh = math.sqrt(0.1) * W, math.sqrt(0.1) * H
        at = torch.randperm(n, generator=g, device="cuda")[:k]
        o = torch.rand(2, generator=g, device="cuda")
        x[at] = o[0] * (W - rw) + _uni((k,), 0, rw, g)
        y[at] = o[1] * (H - rh) + _uni((k,), 0, rh, g)
    l1, l3 = torch.exp(_uni((n,), 0, math.log(8.0), g)), torch.exp(_uni((n,), 0, math.log(8.0), g))
    l2 = _uni((n,), -2, 2, g)
    c = _uni((n, 3), 0, 0.2, g)
    return torch.cat([x[:, None], y[:, None], l1[:, None], l2[:, None], l3[:, None], c], 1).contiguous()


def _raw(p, W, H, mode, g):
    """The parameters as the mode stores them."""
    p = p.clone()
    if mode in ("rs", "paper_rs"):
        n = p.shape[0]
        p[:, 2] = _uni((n,), -math.pi, math.pi, g)
    if mode in ("paper", "paper_rs"):
        size = torch.tensor([W, H], device="cuda", dtype=torch.float32)
        if mode == "paper_rs":  # the scales are columns 3 and 4
            p[:, 3] = torch.exp(_uni((n,), 0, math.log(8.0), g))
        p[:, 0:2] = torch.atanh((p[:, 0:2] / size * 2 - 1).clamp(-0.999, 0.999))
        p[:, 3 if mode == "paper_rs" else 2] -= 0.5
        p[:, 4] -= 0.5
    elif mode == "rs":
        p[:, 3] = torch.exp(_uni((n,), 0, math.log(8.0), g))
    return p


def _shapes(case):
    """[(W, H, n)] of the case's images."""
    if "images" not in case:
        return [(case["W"], case["H"], case["n"])]
    r = random.Random(case["shapes"])
    sizes = [r.choice(BATCH_SHAPES) for _ in range(case["images"])]
    return [(W, H, max(5000, round(70000 * W * H / 786432))) for W, H in sizes]


def _inputs(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    kind = case["kind"]
    if kind == "vq":
        n, M, B = case["n"], case["stages"], case["size"]
        lo = torch.tensor([[1.0, -2.0, 1.0], [0.0, 0.0, 0.0]], device="cuda")
        hi = torch.tensor([[8.0, 2.0, 8.0], [0.2, 0.2, 0.2]], device="cuda")
        u = torch.rand((2, M, B, 3), generator=g, device="cuda")
        cb = lo[:, None, None] + u * (hi - lo)[:, None, None]
        cb[:, 1:] = 0.1 * (2 * u[:, 1:] - 1) * (hi - lo)[:, None, None]
        return dict(means16=_uni((n, 2), 0, 768, g).half(), codebooks=cb.contiguous(),
                    idx=torch.randint(0, B, (2, M, n), generator=g, device="cuda", dtype=torch.uint8))
    if kind == "decode_render":
        W, H, n, B = case["W"], case["H"], case["n"], case["size"]
        p = _gaussians(W, H, n, g)
        lo, gamma = p[:, 2:5].amin(0), (p[:, 2:5].amax(0) - p[:, 2:5].amin(0)) / 63
        codes = torch.zeros((n, 4), dtype=torch.uint8, device="cuda")
        codes[:, :3] = torch.round((p[:, 2:5] - lo) / gamma).clamp(0, 63).to(torch.uint8)
        cb = torch.stack([_uni((B, 3), 0, 0.2, g), _uni((B, 3), -0.02, 0.02, g)])
        return dict(means16=p[:, 0:2].half(), codes=codes, gamma_beta=gamma.tolist() + lo.tolist(), codebooks=cb,
                    idx=torch.randint(0, B, (2, n), generator=g, device="cuda", dtype=torch.uint8))
    mode = case.get("mode", "plain")
    images, params = [], []
    for W, H, n in _shapes(case):
        images.append(_image(W, H, g))
        params.append(_raw(_gaussians(W, H, n, g, case.get("skew", False)), W, H, mode, g))
    d = dict(images=images, params=params)
    if mode in ("separate", "blend"):
        d["logits"] = [_uni((p.shape[0],), -1, 2, g) for p in params]
    if mode == "codec":  # ranges of the quantiser and codebooks drawn from the colours
        p = params[0]
        lo, hi = p[:, 2:5].amin(0), p[:, 2:5].amax(0)
        at = torch.randint(0, p.shape[0], (2, case["size"]), generator=g, device="cuda")
        cb = torch.stack([p[at[0], 5:8], 0.2 * (p[at[1], 5:8] - 0.1)]).contiguous()
        d["codec"] = dict(bits=6, codebooks=cb, gamma=((hi - lo) / 63).tolist(), beta=lo.tolist())
    if kind == "autograd":
        W, H, _ = _shapes(case)[0]
        d["upstream"] = torch.randn((H, W, 3), generator=g, device="cuda") * 1e-3
    return d


def _capacity(rect_n):
    return max(4096, 8 * rect_n)


def _views(f, mode):
    """What a training loop reads of a step: views of the context's own
    buffers, each of which keeps the context (and so the buffers) alive."""
    out = dict(image=f.out, grads=f.grads, params=f.params, m=f.adam_m, v=f.adam_v)
    if mode in ("paper", "paper_rs"):
        out.update(n=f.adan_n)
    if mode == "codec":
        out.update(codebooks=f.codebooks, gamma_beta=f.codec_gb[0])
    if mode in ("separate", "blend"):
        out.update(logits=f.opacity_logit, logit_grads=f.opacity_grad)
    out = {k: t.view(t.shape) for k, t in out.items()}
    for t in out.values():
        t.owner = f
    return out


def prepare(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    if kind == "fit":
        mode = case["mode"]
        kw = dict(tile=case["T"], lr=LR, capacity_factor=4.0)  # room for the Gaussians to grow, as in a long fit
        if mode in ("paper", "paper_rs"):
            kw.update(lr=LR_PAPER, param_mode="paper", optimizer="adan", lr_halve_every=20000)
        if mode in ("rs", "paper_rs"):
            kw.update(cov="rs")
        if mode == "codec":
            kw.update(codec=d["codec"], lr=(2.5e-4, 2.5e-4, 2.5e-4))
        if mode in ("separate", "blend"):
            kw.update(opacity=mode, opacity_logits=d["logits"])
        f = gi.Fit(d["images"], d["params"], **kw)
        return dict(kind=kind, fit=f, out=_views(f, mode))
    if kind == "autograd":
        p = d["params"][0]
        leaf = [p[:, a:b].contiguous().requires_grad_() for a, b in ((0, 2), (2, 5), (5, 8))]
        return dict(kind=kind, leaf=leaf, up=d["upstream"], W=case["W"], H=case["H"], T=case["T"])
    if kind == "render":
        p = d["params"][0]
        r = gi.Renderer(case["W"], case["H"], case["n"], case["T"], capacity=_capacity(case["n"]))
        return dict(kind=kind, renderer=r, args=[p[:, a:b].contiguous() for a, b in ((0, 2), (2, 5), (5, 8))])
    if kind == "decode_render":
        r = gi.Renderer(case["W"], case["H"], case["n"], case["T"], capacity=_capacity(case["n"]))
        return dict(kind=kind, renderer=r, stream=d)
    n = case["n"]
    return dict(kind=kind, out=tuple(torch.empty((n, k), device="cuda") for k in (2, 3, 3)), **d)


def run(s):
    kind = s["kind"]
    if kind == "fit":
        s["fit"].step(1)
        return s["out"]
    if kind == "autograd":
        image = gi.rasterize(*s["leaf"], s["W"], s["H"], s["T"])
        gm, gl, gc = torch.autograd.grad(image, s["leaf"], s["up"])
        return dict(image=image.detach(), means=gm, chol=gl, color=gc)
    if kind == "render":
        return s["renderer"](*s["args"])
    if kind == "decode_render":
        return s["renderer"](*gi.codec_decode(s["stream"]))
    return gi.vq_decode(s["means16"], s["idx"], s["codebooks"], out=s["out"])


# --------------------------------------------------------------------------- required work

def _pairs(W, H, n, T):
    """Expected (tile, Gaussian) pairs of n Gaussians drawn as _gaussians draws them."""
    r = random.Random(1)
    total, samples = 0.0, 2000
    tw, th = -(-W // T), -(-H // T)
    for _ in range(samples):
        l1, l3, l2 = math.exp(r.uniform(0, math.log(8))), math.exp(r.uniform(0, math.log(8))), r.uniform(-2, 2)
        x, y, rx, ry = r.uniform(0, W), r.uniform(0, H), 3 * l1, 3 * math.hypot(l2, l3)
        a = min(tw, int((x + rx) // T) + 1) - max(0, int((x - rx) // T))
        b = min(th, int((y + ry) // T) + 1) - max(0, int((y - ry) // T))
        total += a * b
    return n * total / samples


def work(case):
    kind = case["kind"]
    if kind == "vq":  # FP16 positions and indices in, 8 floats out
        n, M = case["n"], case["stages"]
        return {"bytes": n * (4 + 2 * M + 32), "flops": n * 6 * M}
    shapes = _shapes(case)
    n = sum(s[2] for s in shapes)
    pix = sum(s[0] * s[1] for s in shapes)
    evals = sum(_pairs(*s, case["T"]) for s in shapes) * case["T"] ** 2
    if kind in ("render", "decode_render"):
        return {"bytes": n * (32 if kind == "render" else 10) + pix * 12, "flops": evals * 13}
    if kind == "autograd":
        return {"bytes": n * (32 + 32) + pix * 24, "flops": evals * (13 + 24)}
    state = {"paper": 5, "paper_rs": 5}.get(case["mode"], 3)  # parameters and optimiser averages, read and written
    return {"bytes": n * 32 * (2 * state + 1) + pix * 24, "flops": evals * (13 + 24)}


# --------------------------------------------------------------------------- 64-bit values

F64 = torch.float64


def _form(p, W, H, mode, codec, logit):
    """Rendered position, Cholesky vector, colour and opacity of raw parameters, in 64 bits."""
    x, y, a, b, e, c = p[:, 0], p[:, 1], p[:, 2], p[:, 3], p[:, 4], p[:, 5:8]
    if mode in ("paper", "paper_rs"):
        x, y = (torch.tanh(x) + 1) / 2 * W, (torch.tanh(y) + 1) / 2 * H
    half = 0.5 if mode in ("paper", "paper_rs") else 0.0
    if mode in ("rs", "paper_rs"):
        s1, s2, co, si = b + half, e + half, torch.cos(a), torch.sin(a)
        l1 = torch.sqrt((co * s1) ** 2 + (si * s2) ** 2)
        l2 = co * si * (s1 * s1 - s2 * s2) / l1
        l3 = (s1 * s2).abs() / l1
    else:
        l1, l2, l3 = a + half, b, e + half
    o = None
    if logit is not None:
        o = torch.sigmoid(logit)
        if mode == "separate":
            c = c * o[:, None]
    if codec is not None:  # 16-bit positions, 6-bit Cholesky vector, greedy two-stage colour (straight through)
        x, y = (v + (v.detach().float().half().to(F64) - v.detach()) for v in (x, y))
        gamma, beta = codec["gb"]
        l = torch.stack([l1, l2, l3], 1)
        with torch.no_grad():
            t = (l.float() - beta.float()) / gamma.float()
            code = torch.round(t.clamp(0, 63)).to(F64)
            inside = (t >= 0) & (t <= 63)
        lin = torch.where(inside, l + (code - t.to(F64)).detach() * gamma, code.detach() * gamma + beta)
        exact = (code.float() * gamma.detach().float() + beta.detach().float()).to(F64)
        l = lin + (exact - lin).detach()
        l1, l2, l3 = l[:, 0], l[:, 1], l[:, 2]
        r, q = c.detach().float(), torch.zeros_like(c)
        for m, book in enumerate(codec["books"]):
            pick = torch.cat([((book[None] - part[:, None]) ** 2).sum(-1).argmin(1) for part in r.split(8192)])
            codec["pick"].append(pick)
            codec["resid"].append(r)
            q = q + book[pick].to(F64)
            r = r - book[pick]
        c = c + (q - c).detach()
    return x, y, l1, l2, l3, c, o


def _pair_list(f, W, H, T):
    """(Gaussian, tile) of every pair, from the 3-sigma rectangles in 32 bits, by tile and then by Gaussian."""
    x, y, l1, l2, l3 = (v.detach().float() for v in f[:5])
    tw, th = -(-W // T), -(-H // T)
    rx, ry = 3.0 * l1.abs(), 3.0 * torch.sqrt(l2 * l2 + l3 * l3)

    def span(m, r, n):
        return (torch.floor((m - r) / T).clamp(0, n).long(), (torch.floor((m + r) / T) + 1).clamp(0, n).long())

    (x0, x1), (y0, y1) = span(x, rx, tw), span(y, ry, th)
    w, h = (x1 - x0).clamp(min=0), (y1 - y0).clamp(min=0)
    cnt = w * h
    gid = torch.repeat_interleave(torch.arange(cnt.numel(), device="cuda"), cnt)
    j = torch.arange(gid.numel(), device="cuda") - torch.repeat_interleave(torch.cumsum(cnt, 0) - cnt, cnt)
    tid = (y0[gid] + j // w[gid]) * tw + x0[gid] + j % w[gid]
    order = torch.argsort(tid, stable=True)
    return gid[order], tid[order], tw, th


def _eval(f, g, t, tw, T):
    x, y, l1, l2, l3 = (v.detach()[g] for v in f[:5])
    at = torch.arange(T, device="cuda", dtype=F64) + 0.5
    dx = (t % tw * T)[:, None] + at - x[:, None]
    dy = (t // tw * T)[:, None] + at - y[:, None]
    z1 = (dx / l1[:, None])[:, None, :]
    z2 = (dy[:, :, None] - l2[:, None, None] * z1) / l3[:, None, None]
    return z1, z2, torch.exp(-0.5 * (z1 * z1 + z2 * z2))


def _to_tiles(img, tw, th, T):
    H, W, _ = img.shape
    pad = torch.zeros((th * T, tw * T, 3), device="cuda", dtype=F64)
    pad[:H, :W] = img
    return pad.view(th, T, tw, T, 3).permute(0, 2, 1, 3, 4).reshape(th * tw, T, T, 3)


def _to_image(tiles, tw, th, T, W, H):
    return tiles.view(th, tw, T, T, 3).permute(0, 2, 1, 3, 4).reshape(th * T, tw * T, 3)[:H, :W].contiguous()


CHUNK = 1 << 24  # pixel evaluations at once


def _render64(f, pairs, W, H, T):
    g, t, tw, th = pairs
    tiles = torch.zeros((tw * th, T, T, 3), device="cuda", dtype=F64)
    for i in range(0, g.numel(), CHUNK // (T * T)):
        gi_, ti = g[i:i + CHUNK // (T * T)], t[i:i + CHUNK // (T * T)]
        w = _eval(f, gi_, ti, tw, T)[2]
        tiles.index_add_(0, ti, w[..., None] * f[5].detach()[gi_][:, None, None, :])
    return _to_image(tiles, tw, th, T, W, H)


def _chain(f, g, parts, grads):
    """Adds a chunk's sums of dL/dz1, dL/dz2 terms to the gradients of position and Cholesky vector."""
    l1, l2, l3 = (v.detach()[g] for v in f[2:5])
    p2, p2z1, p2z2, ez1, ez1z1 = parts  # sums of dL/dz2, dL/dz2 z1, dL/dz2 z2, dL/dz1 (direct), dL/dz1 z1
    p1, p1z1 = ez1 - l2 / l3 * p2, ez1z1 - l2 / l3 * p2z1
    for k, v in enumerate((-p1 / l1, -p2 / l3, -p1z1 / l1, -p2z1 / l3, -p2z2 / l3)):
        grads[k].index_add_(0, g, v)


def _backward64(f, pairs, dl, W, H, T):
    g, t, tw, th = pairs
    n = f[0].numel()
    dt = _to_tiles(dl, tw, th, T)
    grads = [torch.zeros(n, device="cuda", dtype=F64) for _ in range(5)]
    gc = torch.zeros((n, 3), device="cuda", dtype=F64)
    for i in range(0, g.numel(), CHUNK // (T * T)):
        gi_, ti = g[i:i + CHUNK // (T * T)], t[i:i + CHUNK // (T * T)]
        z1, z2, w = _eval(f, gi_, ti, tw, T)
        G = dt[ti]
        gc.index_add_(0, gi_, (G * w[..., None]).sum((1, 2)))
        e = -(G * f[5].detach()[gi_][:, None, None, :]).sum(-1) * w  # dL/dsigma
        s = lambda v: v.sum((1, 2))  # noqa: E731
        _chain(f, gi_, (s(e * z2), s(e * z2 * z1), s(e * z2 * z2), s(e * z1), s(e * z1 * z1)), grads)
    return grads, gc


def _blend64(f, pairs, target, W, H, T):
    """Image, gradients of position / Cholesky vector, colour and opacity of the sorted alpha-blending."""
    g, t, tw, th = pairs
    nt, n = tw * th, f[0].numel()
    count = torch.bincount(t, minlength=nt)
    first = torch.cumsum(count, 0) - count
    longest = int(count.max())
    col, op = f[5].detach(), f[6].detach()
    inside = _to_tiles(torch.ones((H, W, 3), device="cuda", dtype=F64), tw, th, T)[..., 0] > 0
    C = torch.zeros((nt, T, T, 3), device="cuda", dtype=F64)
    dl = dt = None
    grads = [torch.zeros(n, device="cuda", dtype=F64) for _ in range(5)]
    gc, go = torch.zeros((n, 3), device="cuda", dtype=F64), torch.zeros(n, device="cuda", dtype=F64)
    for back in (False, True):
        Tr, P, live = torch.ones((nt, T, T), device="cuda", dtype=F64), torch.zeros_like(C), inside.clone()
        for j in range(longest):
            ti = torch.nonzero(count > j)[:, 0]
            gj = g[first[ti] + j]
            z1, z2, w = _eval(f, gj, ti, tw, T)
            raw = op[gj][:, None, None] * w
            a = raw.clamp(max=0.99)
            seen = live[ti] & (raw >= 1 / 255)
            stop = seen & (Tr[ti] * (1 - a) < 1e-4)
            live[ti] &= ~stop
            seen &= ~stop
            a = torch.where(seen, a, torch.zeros_like(a))
            at, c = a * Tr[ti], col[gj][:, None, None, :]
            P[ti] += c * at[..., None]
            if back:
                G = dt[ti]
                gc.index_add_(0, gj, (G * at[..., None]).sum((1, 2)))
                da = (G * (c * Tr[ti][..., None] - (C[ti] - P[ti]) / (1 - a)[..., None])).sum(-1)
                da = torch.where(seen & (raw <= 0.99), da, torch.zeros_like(da))
                go.index_add_(0, gj, (da * w).sum((1, 2)))
                e = -da * a
                s = lambda v: v.sum((1, 2))  # noqa: E731
                _chain(f, gj, (s(e * z2), s(e * z2 * z1), s(e * z2 * z2), s(e * z1), s(e * z1 * z1)), grads)
            Tr[ti] *= 1 - a
        C = P
        if not back:
            img = _to_image(C, tw, th, T, W, H)
            dl = 2 * (img - target) / (3 * W * H)
            dt = _to_tiles(dl, tw, th, T)
    return img, grads, gc, go


def _optimise(p, g, lr, adan):
    """First step of the optimiser: parameters and averages."""
    if adan:
        b1, _, b3 = ADAN
        m, n = (1 - b1) * g, (1 - b3) * g * g
        return p - lr * g / (g.abs() + 1e-8), m, torch.zeros_like(m), n
    m, v = (1 - 0.9) * g, (1 - 0.999) * g * g
    return p - lr * g / (g.abs() + 1e-8), m, v, None


def _fit64(case, d):
    mode, T = case["mode"], case["T"]
    lr = {"paper": LR_PAPER, "paper_rs": LR_PAPER, "codec": (2.5e-4,) * 3}.get(mode, LR)
    image, grads, logit_grads, codec = [], [], None, None
    for (W, H, n), target, p in zip(_shapes(case), d["images"], d["params"]):
        raw = p.to(F64).requires_grad_()
        logit = d["logits"][0].to(F64).requires_grad_() if "logits" in d else None
        if mode == "codec":
            q = d["codec"]
            gb = [torch.tensor(q[k], device="cuda", dtype=torch.float32).to(F64).requires_grad_() for k in ("gamma", "beta")]
            codec = dict(gb=gb, books=q["codebooks"], pick=[], resid=[])
        f = _form(raw, W, H, mode, codec, logit)
        pairs = _pair_list(f, W, H, T)
        if mode == "blend":
            img, ga, gc, go = _blend64(f, pairs, target.to(F64), W, H, T)
        else:
            img = _render64(f, pairs, W, H, T)
            ga, gc = _backward64(f, pairs, 2 * (img - target) / (3 * W * H), W, H, T)
            go = None
        outs, seeds = list(f[:6]), ga + [gc]
        if go is not None:
            outs, seeds = outs + [f[6]], seeds + [go]
        leaves = [raw] + ([logit] if logit is not None else []) + (codec["gb"] if codec else [])
        got = torch.autograd.grad(outs, leaves, seeds, allow_unused=True)
        image.append(img.reshape(-1))
        grads.append(got[0])
        if logit is not None:
            logit_grads = got[1]
    image, grads = torch.cat(image), torch.cat(grads)
    rate = torch.tensor([lr[0]] * 2 + [lr[1]] * 3 + [lr[2]] * 3, device="cuda", dtype=F64)
    params, m, v, nn = _optimise(torch.cat(d["params"]).to(F64), grads, rate, mode in ("paper", "paper_rs"))
    out = dict(image=image, grads=grads, params=params, m=m, v=v)
    if nn is not None:
        out.update(n=nn)
    if mode == "codec":
        size, books = case["size"], []
        for book, pick, resid in zip(codec["books"].to(F64), codec["pick"], codec["resid"]):
            hits = 0.99 + 0.01 * torch.bincount(pick, minlength=size).to(F64)
            total = 0.99 * book + 0.01 * torch.zeros_like(book).index_add_(0, pick, resid.to(F64))
            books.append(total / ((hits + 1e-5) / (hits.sum() + size * 1e-5) * hits.sum())[:, None])
        gb, ggb = torch.cat([x.detach() for x in codec["gb"]]), torch.cat(got[-2:])
        out.update(codebooks=torch.stack(books), gamma_beta=_optimise(gb, ggb, lr[1], False)[0])
    if logit_grads is not None:
        out.update(logits=_optimise(d["logits"][0].to(F64), logit_grads, lr[2], False)[0], logit_grads=logit_grads)
    return out


def exact(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    if kind == "vq":
        n, rows = case["n"], []
        for a in range(2):
            s = torch.zeros((n, 3), device="cuda", dtype=F64)
            for m in range(case["stages"]):
                s += d["codebooks"][a, m].to(F64)[d["idx"][a, m].long()]
            rows.append(s)
        return (d["means16"].to(F64), *rows)
    if kind == "fit":
        return _fit64(case, d)
    W, H, T = case["W"], case["H"], case["T"]
    if kind == "decode_render":
        gb = torch.tensor(d["gamma_beta"], device="cuda", dtype=F64)
        l = d["codes"][:, :3].to(F64) * gb[:3] + gb[3:]
        c = sum(d["codebooks"][m].to(F64)[d["idx"][m].long()] for m in range(2))
        p = torch.cat([d["means16"].to(F64), l, c], 1)
    else:
        p = d["params"][0].to(F64)
    f = _form(p, W, H, "plain", None, None)
    pairs = _pair_list(f, W, H, T)
    image = _render64(f, pairs, W, H, T)
    if kind != "autograd":
        return image
    ga, gc = _backward64(f, pairs, d["upstream"].to(F64), W, H, T)
    return dict(image=image, means=torch.stack(ga[:2], 1), chol=torch.stack(ga[2:], 1), color=gc)
