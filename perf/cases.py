"""The renderer's work as its users run it, case by case: inputs, one pass, the
64-bit answer, the work a pass cannot do without, and how exact it has to be.

A case is one kind of call over one range of sizes:
  call     plan      a prepared Plan: forward, and the adjoint when `bwd` is set
           oneshot   render_batched() with nothing prepared (inference code)
           autograd  GSRenderBatched inside a training step: images and the
                     gradients of the five parameter tensors
  images   1, or a batch; `sizes` > 0 draws every image's LR size and scale
           from that seed within [lr_lo, lr_h] x [lr_lo, lr_w] and
           [scale_lo, scale]
  m        Gaussians per LR pixel on the reference grid; 0: `n` Gaussians at
           absolute centres
  window   "sigma" (k-sigma box) or "ratio" (Algorithm 1, ratio r); k holds k or r
  head     "" physical parameters, "toy" / "paper": raw head outputs whose
           activations run inside the render
  adjoint  0 the default, 2 the bitwise reproducible one
"""
import math
import statistics

import numpy as np
import torch

import paper_2501_06838_gb300 as gs
from paper_2501_06838_gb300.render import WINDOW_RATIO, WINDOW_SIGMA

DEVICE = "cuda"
DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
BASE = {"call": "plan", "bwd": False, "images": 1, "sizes": 0, "lr_lo": 0, "scale_lo": 0.0, "n": 0,
        "m": 1, "dtype": "f32", "window": "sigma", "k": 3.0, "norm": 0, "align": 0, "head": "",
        "adjoint": 0, "sig_lo": 0.3, "sig_hi": 2.0}


class Head:
    """Constants of a fused Gaussian head (sigma = lo + span sigmoid, rho = scale tanh)."""

    def __init__(self, sigma_lo, sigma_span, rho_scale, offset_scale, offset_tanh):
        self.sigma_lo, self.sigma_span, self.rho_scale = sigma_lo, sigma_span, rho_scale
        self.offset_scale, self.offset_tanh = offset_scale, offset_tanh


# the training step's head (sigma up to 3 LR px) and the inference pipeline's
HEADS = {"toy": Head(0.2, 2.8, 0.9, 1.0, 1), "paper": Head(0.0, 1.0, 0.99, 1.0, 0)}


def _case(**kw):
    c = dict(BASE)
    c.update(kw)
    return c


def listed():
    return [
        # a thumbnail preview: the smallest call, launches and latency only
        _case(name="thumb_x4", lr_h=48, lr_w=48, scale=4.0),
        # fitting one 1024 x 1024 image: forward and adjoint, the benchmark's default step
        _case(name="fit_x4", bwd=True, lr_h=256, lr_w=256, scale=4.0),
        # a large print from BF16 parameters, forward and adjoint: the largest image
        _case(name="print_x12_bf16", bwd=True, lr_h=270, lr_w=480, scale=12.0, m=4, dtype="bf16",
              sig_lo=0.2, sig_hi=3.0),
        # odd sizes, FP16 storage, pixel centres aligned across scales, peak colours
        _case(name="odd_x3.7_f16", bwd=True, lr_h=203, lr_w=271, scale=3.7, m=4, dtype="f16",
              norm=1, align=1, sig_lo=0.2, sig_hi=1.5),
        # a served batch of 16 images of uneven sizes and scales, forward
        _case(name="serve16_uneven", images=16, sizes=1, lr_lo=64, lr_h=360, lr_w=480,
              scale_lo=1.5, scale=12.0),
        # inference of the paper's shape: 720 x 720 out, 16 raw BF16 Gaussians per LR
        # pixel straight from the network, Algorithm 1's window, nothing prepared
        _case(name="paper_x4_infer", call="oneshot", lr_h=180, lr_w=180, scale=4.0, m=16,
              dtype="bf16", window="ratio", k=0.1, head="paper"),
        # a training step's render: 16 crops at scales in [1, 4], raw BF16 head outputs
        _case(name="train16_crops", call="autograd", bwd=True, images=16, sizes=2, lr_lo=48,
              lr_h=48, lr_w=48, scale_lo=1.0, scale=4.0, dtype="bf16", head="toy"),
        # the paper's training shape: 16 Gaussians per LR pixel, Algorithm 1's window
        _case(name="train4_ratio", call="autograd", bwd=True, images=4, sizes=3, lr_lo=48,
              lr_h=48, lr_w=48, scale_lo=1.0, scale=4.0, m=16, window="ratio", k=0.1,
              head="paper"),
        # bitwise reproducible gradients, odd output width
        _case(name="reproducible_x5", bwd=True, lr_h=150, lr_w=203, scale=5.0, adjoint=2),
        # Gaussians at absolute centres (no reference grid): the sorted pair list
        _case(name="scatter_x3", bwd=True, lr_h=240, lr_w=320, scale=3.0, m=0, n=100_000),
        # one image, nothing prepared, a common upscale
        _case(name="oneshot_x6", call="oneshot", lr_h=96, lr_w=128, scale=6.0),
        # a deep zoom far past the training scales, forward and adjoint
        _case(name="zoom_x24", bwd=True, lr_h=48, lr_w=64, scale=24.0, m=4, norm=1),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _one_draw(rng):
    kind = rng.choice(("plan", "plan", "train", "train", "serve", "paper", "crops", "ratio",
                       "reproducible", "scatter", "oneshot"))
    h, w = int(_log(rng, 24, 400)), int(_log(rng, 24, 480))
    s = round(_log(rng, 1.3, 16.0), 2)
    dtype = rng.choice(("f32", "f32", "bf16", "f16"))
    m = rng.choice((1, 1, 4, 9, 16))
    hi = rng.choice((1.5, 2.0, 3.0))
    if kind in ("plan", "train"):
        return _case(bwd=kind == "train", lr_h=h, lr_w=w, scale=s, m=m, dtype=dtype, sig_hi=hi,
                     norm=rng.choice((0, 0, 1)), align=rng.choice((0, 0, 1)))
    if kind == "serve":
        return _case(images=rng.randint(2, 16), sizes=rng.randint(10, 10_000),
                     lr_lo=rng.choice((24, 48, 64)), lr_h=rng.randint(80, 360),
                     lr_w=rng.randint(80, 480), scale_lo=1.5, scale=max(2.0, s), dtype=dtype)
    if kind == "paper":
        lr = int(_log(rng, 40, 200))
        return _case(call="oneshot", lr_h=lr, lr_w=lr + rng.randint(-8, 8),
                     scale=round(rng.uniform(2.0, 8.0), 2), m=16, dtype="bf16", window="ratio",
                     k=0.1, head="paper")
    if kind == "crops":
        lr = rng.choice((32, 48, 49, 64))
        return _case(call="autograd", bwd=True, images=rng.randint(2, 24),
                     sizes=rng.randint(10, 10_000), lr_lo=lr, lr_h=lr, lr_w=lr, scale_lo=1.0,
                     scale=4.0, dtype=rng.choice(("bf16", "f32")), head="toy")
    if kind == "ratio":
        lr = rng.choice((32, 48, 51))
        return _case(call="autograd", bwd=True, images=rng.randint(1, 4),
                     sizes=rng.randint(10, 10_000), lr_lo=lr, lr_h=lr, lr_w=lr, scale_lo=1.0,
                     scale=4.0, m=rng.choice((4, 9, 16)), window="ratio", k=0.1, head="paper")
    if kind == "reproducible":
        return _case(bwd=True, lr_h=h, lr_w=w, scale=min(s, 8.0), m=rng.choice((1, 4)), adjoint=2)
    if kind == "scatter":
        return _case(bwd=True, lr_h=h, lr_w=w, scale=min(s, 6.0), m=0,
                     n=int(_log(rng, 2_000, 400_000)))
    return _case(call="oneshot", lr_h=h, lr_w=w, scale=s, m=rng.choice((1, 4)), dtype=dtype)


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        c = _one_draw(rng)
        if _cost(c) <= most and all(max(oh, ow) <= 8192 for _, _, _, oh, ow in _sizes(c)):
            return c


# ---------------------------------------------------------------------------
# Sizes, work, tolerance.
# ---------------------------------------------------------------------------
def _f32(x):
    return float(np.float32(x))


def _sizes(case):
    """(lr_h, lr_w, scale, out_h, out_w) of every image."""
    got = []
    rng = np.random.Generator(np.random.PCG64(case["sizes"]))
    for _ in range(case["images"]):
        h, w, s = case["lr_h"], case["lr_w"], case["scale"]
        if case["sizes"]:
            h = int(rng.integers(min(case["lr_lo"], h), h + 1))
            w = int(rng.integers(min(case["lr_lo"], w), w + 1))
            s = rng.uniform(min(case["scale_lo"], s), s)
        s = _f32(s)
        got.append((h, w, s, int(math.floor(s * h)), int(math.floor(s * w))))
    return got


def _count(case, h, w):
    return case["n"] if case["m"] == 0 else case["m"] * h * w


def _pairs(case):
    """Expected (Gaussian, pixel) pairs: windows clipped at the image's edges."""
    def cover(win, size):   # mean overlap of a window centred anywhere in the image
        return win - win * win / (4.0 * size) if win < 2.0 * size else float(size)

    qs = [(i + 0.5) / 48 for i in range(48)]
    if case["head"]:
        hd, nd = HEADS[case["head"]], statistics.NormalDist()
        sig = [hd.sigma_lo + hd.sigma_span / (1.0 + math.exp(-1.5 * nd.inv_cdf(q))) for q in qs]
    else:
        sig = [case["sig_lo"] * (case["sig_hi"] / case["sig_lo"]) ** q for q in qs]
    total = 0.0
    for h, w, s, oh, ow in _sizes(case):
        if case["window"] == "ratio":
            ex, ey = cover(2 * s * case["k"] * w, ow), cover(2 * s * case["k"] * h, oh)
        else:
            ex = sum(cover(2 * s * case["k"] * v, ow) for v in sig) / len(sig)
            ey = sum(cover(2 * s * case["k"] * v, oh) for v in sig) / len(sig)
        total += _count(case, h, w) * ex * ey
    return total


def _cost(case):
    return _pairs(case) * (31.0 if case["bwd"] else 10.0) + 12.0 * sum(a * b for _, _, _, a, b in _sizes(case))


def work(case):
    """Per pair: exponent 3 and colours 6 flops and one exp2 forward; exponent,
    g . c, colour and moment sums 20 flops and one exp2 in the adjoint."""
    item = 4 if case["dtype"] == "f32" else 2
    n = sum(_count(case, h, w) for h, w, _, _, _ in _sizes(case))
    px = sum(a * b for _, _, _, a, b in _sizes(case))
    b = n * 9 * item + 12 * px
    if case["bwd"]:
        b += 12 * px + n * 9 * (item if case["call"] == "autograd" else 4)
    return {"bytes": b, "flops": _pairs(case) * (31 if case["bwd"] else 10)}


def tolerance(case):
    """About four times the relative error against exact() that was measured:
    1.3e-7 to 2.8e-7 for float32 sums; 4e-7 to 1.4e-6 forward and up to 2.2e-5
    in the gradients under the paper's head (sigma down to 0 and |rho| up to
    0.99); gradients returned in 16 bits flip a rounding now and then."""
    if case["call"] == "autograd" and case["dtype"] != "f32":
        return {"rel": 3e-4, "max": 0.02}
    if case["head"] == "paper":
        return {"rel": 9e-5 if case["bwd"] else 6e-6}
    return {"rel": 1.5e-6 if case["bwd"] else 1e-6}


# ---------------------------------------------------------------------------
# Inputs and one pass.
# ---------------------------------------------------------------------------
def _draw_params(case, h, w, gen, device):
    """The five parameter tensors of one image in their storage type."""
    n = _count(case, h, w)
    f = dict(device=device, dtype=torch.float32, generator=gen)
    if case["head"]:
        z = torch.randn((n, 9), **f)
        off = z[:, 0:2] * (0.25 / math.sqrt(max(1, case["m"])))
        rest = z[:, 2:9] * 1.5
        ts = (off, rest[:, 0:2], rest[:, 2], rest[:, 3:6], rest[:, 6])
    else:
        u = torch.rand((n, 9), **f)
        if case["m"] == 0:
            off = u[:, 0:2] * torch.tensor([w, h], device=device) - 0.5
        else:
            off = (u[:, 0:2] - 0.5) / math.sqrt(case["m"])
        lo, hi = math.log(case["sig_lo"]), math.log(case["sig_hi"])
        ts = (off, torch.exp(lo + u[:, 2:4] * (hi - lo)), 1.8 * u[:, 4] - 0.9, u[:, 5:8], u[:, 8])
    return [t.to(DTYPES[case["dtype"]]).contiguous() for t in ts]


def _inputs(case, seed):
    """Per image: parameters, view, upstream gradient (None when there is no adjoint)."""
    gen = torch.Generator(device=DEVICE).manual_seed(int(seed) % (1 << 62))
    params, views, gouts = [], [], []
    for h, w, s, oh, ow in _sizes(case):
        params.append(_draw_params(case, h, w, gen, DEVICE))
        v = gs.View(h, w, oh, ow, s, trunc_k=case["k"], norm=case["norm"], align=case["align"],
                    window=WINDOW_RATIO if case["window"] == "ratio" else WINDOW_SIGMA)
        if case["adjoint"]:
            v.adjoint = case["adjoint"]
        views.append(v)
        gouts.append(torch.randn((3, oh, ow), device=DEVICE, generator=gen) if case["bwd"] else None)
    return params, views, gouts


def prepare(case, seed):
    params, views, gouts = _inputs(case, seed)
    head = HEADS.get(case["head"])
    st = {"case": case, "views": views, "gouts": gouts, "head": head}
    if case["call"] == "autograd":
        st["sizes"] = [int(p[2].shape[0]) for p in params]
        st["leaves"] = [torch.cat([p[k] for p in params]).requires_grad_() for k in range(5)]
        return st
    st["gs"] = [gs.Gaussians(*p, ref_grid_m=case["m"], head=head) for p in params]
    if case["call"] == "plan":
        st["plan"] = gs.Plan(st["gs"], views, with_grads=case["bwd"],
                             grad_outs=gouts if case["bwd"] else None)
    return st


def run(state):
    case = state["case"]
    if case["call"] == "plan":
        plan = state["plan"]
        outs = plan.fwd()
        return {"images": outs, "grads": plan.bwd()} if case["bwd"] else {"images": outs}
    if case["call"] == "oneshot":
        outs, _ = gs.render_batched(state["gs"], state["views"])
        return {"images": outs}
    outs = gs.GSRenderBatched.apply(state["views"], case["m"], state["sizes"], state["head"],
                                    *state["leaves"])
    grads = torch.autograd.grad(outs, state["leaves"], state["gouts"])
    return {"images": [o.detach() for o in outs], "grads": list(grads)}


# ---------------------------------------------------------------------------
# The same in 64 bits, pair by pair. Only the windows' integer edges follow
# the float32 sequence that defines them.
# ---------------------------------------------------------------------------
def _exp_seq(x):
    x = x.clamp(-87.0, 88.0)
    n = torch.round(x * 1.44269502162933349609375)
    r = (x - n * 0.693359375) - n * -2.12194441701285541057586669921875e-4
    p = torch.full_like(x, 1.9841270113829523324966431e-4)
    for c in (1.3888889225199818611145020e-3, 8.3333337679505348205566406e-3,
              4.1666667908430099487304688e-2, 0.16666667163372039794921875, 0.5, 1.0, 1.0):
        p = p * r
        p = p + c
    return torch.ldexp(p, n.to(torch.int32))


def _tanh_seq(x):
    e = _exp_seq(-2.0 * x.abs())
    t = (1.0 - e) / (1.0 + e)
    return torch.where(x < 0, -t, t)


def _grid(case, h, w, device):
    """Reference positions of the Gaussians, float32 values."""
    m = case["m"]
    if m == 0:
        return 0.0, 0.0
    r = math.isqrt(m)
    d = np.array([np.float32(2 * a + 1 - r) / np.float32(2 * r) for a in range(r)], np.float32)
    px = np.arange(w, dtype=np.float32)[:, None] + d[None, :]      # [w, a]
    py = np.arange(h, dtype=np.float32)[:, None] + d[None, :]      # [h, b]
    px = np.broadcast_to(px[None, :, None, :], (h, w, r, r)).reshape(-1)
    py = np.broadcast_to(py[:, None, :, None], (h, w, r, r)).reshape(-1)
    return (torch.from_numpy(np.ascontiguousarray(a)).to(device) for a in (px, py))


def _windows(case, h, w, s, oh, ow, px, py, par):
    """Integer windows (x0, x1, y0, y1) by the float32 sequence; empty ones x0 > x1."""
    off, sig = par[0].float(), par[1].float()
    hd = HEADS.get(case["head"])
    if hd:
        off = float(hd.offset_scale) * (_tanh_seq(off) if hd.offset_tanh else off)
        sg = 1.0 / (1.0 + _exp_seq(-sig))
        sig = sg * _f32(hd.sigma_span)
        sig = sig + _f32(hd.sigma_lo)
    edges = []
    for ax, p, lr, last in ((0, px, w, ow - 1), (1, py, h, oh - 1)):
        c = (off[:, ax] + p) * s
        if case["align"]:
            c = c + _f32(_f32(0.5 * s) - 0.5)
        sk = _f32(np.float32(s) * np.float32(case["k"]))
        if case["window"] == "ratio":
            r = _f32(np.float32(sk) * np.float32(lr))
            lo, hi = torch.floor(c - r) + 1.0, torch.ceil(c + r) - 1.0
        else:
            r = sig[:, ax] * sk
            lo, hi = torch.ceil(c - r), torch.floor(c + r)
        lo, hi = lo.clamp(min=0.0), hi.clamp(max=float(last))
        bad = (lo > last) | (hi < 0) | (lo > hi)
        edges += [torch.where(bad, 1.0, lo).long(), torch.where(bad, 0.0, hi).long()]
    return edges


def _exact_image(case, size, par, gout):
    h, w, s, oh, ow = size
    dev = par[0].device
    px, py = _grid(case, h, w, dev)
    x0, x1, y0, y1 = _windows(case, h, w, s, oh, ow, px, py, par)
    raw = [t.double().requires_grad_(gout is not None) for t in par]
    hd = HEADS.get(case["head"])
    if hd:
        off = hd.offset_scale * (torch.tanh(raw[0]) if hd.offset_tanh else raw[0])
        sig = _f32(hd.sigma_lo) + _f32(hd.sigma_span) * torch.sigmoid(raw[1])
        rho = _f32(hd.rho_scale) * torch.tanh(raw[2])
        rgb, alpha = torch.sigmoid(raw[3]), torch.sigmoid(raw[4])
    else:
        off, sig, rho, rgb, alpha = raw
    mux, muy = off[:, 0] + px, off[:, 1] + py
    sx, sy = sig[:, 0], sig[:, 1]
    D = (1.0 - rho) * (1.0 + rho)
    a, b, c = 1.0 / (sx * sx * D), -2.0 * rho / (sx * sy * D), 1.0 / (sy * sy * D)
    L = torch.zeros_like(rho) if case["norm"] else -torch.log(2.0 * math.pi * sx * sy * torch.sqrt(D))
    col = alpha[:, None] * rgb
    A, B, C, Ld, MX, MY, K = (t.detach() for t in (a, b, c, L, mux, muy, col))
    h0 = 0.5 / s - 0.5 if case["align"] else 0.0
    wd, hg = (x1 - x0 + 1).clamp(min=0), (y1 - y0 + 1).clamp(min=0)
    area = wd * hg
    live = torch.nonzero(area).flatten()
    ends = torch.cumsum(area[live], 0)
    img = torch.zeros((3, oh * ow), dtype=torch.float64, device=dev)
    go = gout.double().reshape(3, -1) if gout is not None else None
    mom = torch.zeros((9, par[2].shape[0]), dtype=torch.float64, device=dev)
    host = ends.cpu().numpy()
    at, total, step = 0, int(host[-1]) if len(host) else 0, 30_000_000
    while at < len(host):
        base = int(host[at - 1]) if at else 0
        to = max(at + 1, int(np.searchsorted(host, base + step, side="right")))
        g = live[at:to]
        cnt = area[g]
        i = torch.repeat_interleave(g, cnt)
        k = torch.arange(int(host[to - 1]) - base, device=dev) - torch.repeat_interleave(ends[at:to] - base - cnt, cnt)
        row = torch.div(k, wd[i], rounding_mode="floor")
        x, y = x0[i] + (k - row * wd[i]), y0[i] + row
        dx, dy = x.double() / s + h0 - MX[i], y.double() / s + h0 - MY[i]
        wt = torch.exp(-0.5 * (A[i] * dx * dx + B[i] * dx * dy + C[i] * dy * dy) + Ld[i])
        pix = y * ow + x
        for ch in range(3):
            img[ch].index_add_(0, pix, K[i, ch] * wt)
        if go is not None:
            gk = [go[ch][pix] for ch in range(3)]
            G = (gk[0] * K[i, 0] + gk[1] * K[i, 1] + gk[2] * K[i, 2]) * wt
            vals = (G, G * dx, G * dy, G * dx * dx, G * dx * dy, G * dy * dy, gk[0] * wt, gk[1] * wt, gk[2] * wt)
            for q, v in enumerate(vals):
                mom[q, g] = torch.segment_reduce(v, "sum", lengths=cnt)
        at = to
    image = img.reshape(3, oh, ow)
    if go is None:
        return image, None
    S0, S10, S01, S20, S11, S02 = mom[:6]
    loss = (-0.5 * (a * S20 + b * S11 + c * S02) + L * S0 + mux * (A * S10 + 0.5 * B * S01)
            + muy * (C * S01 + 0.5 * B * S10)).sum() + (col * mom[6:9].T).sum()
    return image, torch.autograd.grad(loss, raw)


def exact(case, seed):
    params, _, gouts = _inputs(case, seed)
    images, grads = [], []
    for size, par, go in zip(_sizes(case), params, gouts):
        im, gr = _exact_image(case, size, par, go)
        images.append(im)
        if gr is not None:
            grads.append(gr)
    if not case["bwd"]:
        return {"images": images}
    if case["call"] == "autograd":
        return {"images": images, "grads": [torch.cat([g[k] for g in grads]) for k in range(5)]}
    flat = [torch.cat([g[0], g[1], g[2][:, None], g[3], g[4][:, None]], 1) for g in grads]
    return {"images": images, "grads": flat}
