"""Performance cases of the stereo matching and refinement paths, through the public `Context`.

The paths: the coarse matcher (one small pair up to a batch of driving-camera frames, and its SGM
and domain-transform variants), the refinement network in its four forms (BF16, FP8, FP32, the
paper's Table I network), the whole pipeline from device images and from host images, and a
training step.  1242 x 375 with 48 coarse disparities and a 9 x 9 window is the framework's
driving-camera workload, 256 x 128 with 16 disparities its small one.
"""
from __future__ import annotations

import math

import torch
import torch.nn.functional as F

from paper_2305_11566_gb300 import binding, synth

NETS = {"small": synth.NET_SMALL, "wide": synth.NET_WIDE, "table1": "table1"}
# the four frame sizes of the KITTI recordings
KITTI_SIZES = ((1242, 375), (1241, 376), (1226, 370), (1224, 370))
KL_WEIGHT = 1e-3
_streams = []


def _stream():
    """The one side stream of the program (the pipeline replays CUDA graphs off the default stream)."""
    if not _streams:
        _streams.append(torch.cuda.Stream())
    return _streams[0]


def listed():
    return [
        # One small pair, e.g. a robot's low-resolution camera: a single launch, latency is all.
        {"name": "coarse_one_small", "kind": "coarse", "n": 1, "W": 256, "H": 128, "D": 16, "k": 7, "scores": False},
        # Coarse maps of a recorded drive, many frames a call.
        {"name": "coarse_batch", "kind": "coarse", "n": 64, "W": 1242, "H": 375, "D": 48, "k": 9, "scores": False},
        # The paper's own coarse stage (ZNCC + semi-global matching + occlusion check + median)
        # over a recorded drive.
        {"name": "coarse_sgm_batch", "kind": "variant", "n": 64, "W": 1242, "H": 375, "D": 48, "k": 9, "cost": "zncc",
         "agg": "sgm", "iters": 2, "post": True},
        # The robustness study's census + domain-transform setting.
        {"name": "coarse_census_dt", "kind": "variant", "n": 16, "W": 1242, "H": 375, "D": 48, "k": 9, "cost": "census",
         "agg": "dt", "iters": 2, "post": False},
        # One camera frame at a time, matched and refined: the real-time loop.
        {"name": "pipeline_bf16_frame", "kind": "pipeline", "form": "bf16", "net": "wide", "n": 1, "W": 1242, "H": 375,
         "D": 48, "k": 9, "mix": ""},
        # The serving batch: match and refine 64 frames a call.
        {"name": "pipeline_bf16_batch", "kind": "pipeline", "form": "bf16", "net": "wide", "n": 64, "W": 1242, "H": 375,
         "D": 48, "k": 9, "mix": ""},
        # Frames of the four recording sizes (odd widths among them) from pinned host memory,
        # results back to the host: an offline job over a data set.
        {"name": "pipeline_host_mixed", "kind": "host", "form": "bf16", "net": "wide", "n": 32, "W": 1242, "H": 375,
         "D": 48, "k": 9, "mix": "kitti"},
        # Quantised refinement of coarse maps that another matcher made.
        {"name": "refine_fp8_batch", "kind": "refine", "form": "fp8", "net": "wide", "n": 32, "W": 1242, "H": 375,
         "D": 48, "k": 9, "mix": ""},
        # Full-precision refinement: the form that results are checked against.
        {"name": "refine_fp32_batch", "kind": "refine", "form": "fp32", "net": "wide", "n": 8, "W": 1242, "H": 375,
         "D": 48, "k": 9, "mix": ""},
        # The paper's Table I network on a batch of frames.
        {"name": "refine_table1_batch", "kind": "refine", "form": "fp32", "net": "table1", "n": 16, "W": 1242, "H": 375,
         "D": 48, "k": 9, "mix": ""},
        # A training step (forward, loss, backward, Adam) on full frames with the tensor-core forward.
        {"name": "train_bf16_frames", "kind": "train", "form": "bf16", "net": "small", "n": 16, "W": 1242, "H": 375,
         "D": 48, "k": 9},
        # A full-precision training step on a minibatch of crops.
        {"name": "train_fp32_crops", "kind": "train", "form": "fp32", "net": "wide", "n": 8, "W": 256, "H": 128, "D": 16,
         "k": 7},
    ]


def draw(rng):
    """One more case: kind by use, sizes spread over their logarithm, odd ones included."""
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["coarse", "coarse", "variant", "variant", "pipeline", "pipeline", "host", "refine", "refine",
                       "refine", "train", "train"])
    c = {"kind": kind}
    form, net = "bf16", "wide"
    if kind in ("pipeline", "host"):
        form = rng.choice(["bf16", "bf16", "fp8"])
        net = "wide" if form == "fp8" else rng.choice(["wide", "wide", "small"])
    elif kind == "refine":
        form = rng.choice(["bf16", "fp8", "fp32", "table1"])
        net = {"fp8": "wide", "table1": "table1"}.get(form) or rng.choice(["wide", "small"])
        form = "fp32" if form == "table1" else form
    elif kind == "train":
        form, net = rng.choice(["bf16", "fp32"]), rng.choice(["small", "wide"])
    most = {"coarse": 64, "pipeline": 64, "host": 32, "train": 4 if net == "wide" else 16}.get(kind)
    if kind == "variant":
        agg = rng.choice(["sgm", "sgm", "dt", "none"])
        most = 64 if agg == "sgm" else 16
    elif kind == "refine":
        most = 16 if net == "table1" else 8 if form == "fp32" else 32
    area = most * 1242 * 375  # pixels of the kind's listed case
    W = log_int(200, 1400)
    H = min(log_int(100, 460), W)
    n = log_int(1, max(1, min(most, area // (W * H))))
    if kind in ("train",):
        n = min(n, 16)
    k = rng.choice([5, 7, 9, 9, 11])
    D = min(log_int(8, 96 if kind != "variant" else 64), W // 4)
    c.update(n=n, W=W, H=H, D=D, k=k)
    if kind == "coarse":
        c["scores"] = rng.random() < 0.25
        c["n"] = min(n, 21) if c["scores"] else n
    elif kind == "variant":
        c.update(cost=rng.choice(["zncc", "census"]), agg=agg, iters=rng.choice([1, 2, 3]) if agg == "dt" else 2,
                 post=rng.random() < 0.5)
    else:
        c.update(form=form, net=net)
        if kind != "train":
            c["mix"] = "scaled" if n >= 4 and rng.random() < 0.4 else ""
    return c


# ---------------------------------------------------------------- sizes and work
def sizes(case):
    """[(W, H, D)] of the case's pairs."""
    mix = case.get("mix", "")
    out = []
    for i in range(case["n"]):
        W, H, D = case["W"], case["H"], case["D"]
        if mix == "kitti":
            W, H = KITTI_SIZES[i % len(KITTI_SIZES)]
        elif mix == "scaled":
            f = (1.0, 0.77, 0.52, 0.26)[i % 4]
            W, H = max(4 * case["k"], int(W * f)), max(4 * case["k"], int(H * f))
        out.append((W, H, min(D, W // 4)))
    return out


def _levels(H, W):
    out = [(H, W)]
    for _ in range(3):
        H, W = (H + 1) // 2, (W + 1) // 2
        out.append((H, W))
    return out


def _net_flops(net, H, W):
    """Multiply-adds x 2 of one refinement; a nearest-x2 decoder layer needs 4 taps a pixel (the
    taps that fall on one input pixel share its weight sum)."""
    lv = _levels(H, W)
    px = [h * w for h, w in lv]
    if net == "table1":
        f = 0
        for (_, co, ci, ks), (p, t) in zip(synth.TABLE1_LAYERS, [
                (px[1], 25), (px[1], 25), (px[2], 25), (px[2], 25), (px[3], 25), (px[3], 25), (px[3], 1), (px[3], 1),
                (px[3], 25), (px[2], 6.25), (px[2], 25), (px[1], 6.25), (px[0], 6.25)]):
            f += 2 * p * t * co * ci
        return f
    s = NETS[net]
    (c1, c2, c3), z, (d1, d2, d3) = s.enc, s.latent, s.dec
    return 2 * (px[1] * 9 * 2 * c1 + px[2] * 9 * c1 * c2 + px[3] * 9 * c2 * c3 + px[3] * c3 * z + px[2] * 4 * z * d1
                + px[1] * 4 * d1 * d2 + px[0] * 4 * d2 * d3 + px[0] * 9 * d3)


def _weight_floats(net):
    if net == "table1":
        return sum(co * k * k * ci + co for _, co, ci, k in synth.TABLE1_LAYERS)
    return NETS[net].n_params()


def work(case):
    nbytes = flops = 0.0
    kind = case["kind"]
    for W, H, D in sizes(case):
        h, w = H // 4, W // 4
        img, cells = W * H, h * w * D
        if kind in ("coarse", "variant", "pipeline", "host"):
            nbytes += 2 * img
            flops += 2 * img + 12 * cells  # box sums; product sums slid both ways and the score
        if kind == "coarse":
            nbytes += h * w * (10 if case["scores"] else 2)
        elif kind == "variant":
            nbytes += h * w * 2
            flops += cells * {"none": 1, "sgm": 4 * 7, "dt": case["iters"] * 4 * 2}[case["agg"]]
        else:
            nbytes += 4 * img
            f = _net_flops(case["net"], H, W)
            flops += f
            if kind in ("refine", "train"):
                nbytes += img + 2 * h * w
            if kind == "train":  # eps, mu, logvar, ground truth; input and weight gradients
                lat = NETS[case["net"]].latent
                h3, w3 = _levels(H, W)[3]
                nbytes += 2 * h * w + 12 * h3 * w3 * lat + 4 * img
                flops += 2 * f
    if kind not in ("coarse", "variant"):
        nbytes += 4 * _weight_floats(case["net"]) * (6 if kind == "train" else 1)
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------- inputs
def _noise(g, n, H, W):
    """4-octave lattice noise, each image scaled to 0..255 (float32 [n, H, W])."""
    acc = torch.zeros(n, H, W, device="cuda")
    for cell, amp in ((32, 1.0), (16, 0.5), (8, 0.25), (4, 0.125)):
        gh, gw = H // cell + 2, W // cell + 2
        lat = torch.rand(n, 1, gh, gw, device="cuda", generator=g)
        acc += amp * F.interpolate(lat, size=(gh * cell, gw * cell), mode="bilinear")[:, 0, :H, :W]
    lo, hi = acc.amin((1, 2), keepdim=True), acc.amax((1, 2), keepdim=True)
    return (acc - lo) / (hi - lo) * 255.0


def _scene(g, n, W, H, D):
    """n textured pairs with piecewise-planar disparity: left, right (uint8 [n, H, pitch]), disparity."""
    pitch = (W + 15) // 16 * 16
    dmax = 4.0 * max(1, D - 1)
    left = _noise(g, n, H, W).round()
    u = torch.rand(n, 5, 4, 1, 1, device="cuda", generator=g)
    xs = torch.arange(W, device="cuda", dtype=torch.float32)
    ys = torch.arange(H, device="cuda", dtype=torch.float32)[:, None]
    best = torch.full((n, H, W), float("inf"), device="cuda")
    gt = torch.zeros(n, H, W, device="cuda")
    for j in range(4):  # planes on the Voronoi cells of 4 points
        px, py = u[:, 0, j] * W, u[:, 1, j] * H
        d2 = (xs - px) ** 2 + (ys - py) ** 2
        plane = ((0.1 + 0.8 * u[:, 2, j]) + (u[:, 3, j] - 0.5) * 0.6 * (xs - px) / W
                 + (u[:, 4, j] - 0.5) * 0.6 * (ys - py) / H) * dmax
        near = d2 < best
        gt = torch.where(near, plane, gt)
        best = torch.where(near, d2, best)
    gt = gt.clamp(0.0, dmax)
    src = xs.long() + gt.round().long()
    right = torch.where(src < W, left.gather(2, src.clamp(max=W - 1)), _noise(g, n, H, W))
    right = right + 2.0 * torch.randn(n, H, W, device="cuda", generator=g)
    out = torch.zeros(2, n, H, pitch, device="cuda", dtype=torch.uint8)
    out[0, :, :, :W] = left.to(torch.uint8)
    out[1, :, :, :W] = right.round().clamp(0, 255).to(torch.uint8)
    return out[0], out[1], gt


def _weights(net, g):
    """He-normal weights and small biases, flat float32 on the GPU."""
    if net == "table1":
        layers = [(co, ci, k) for _, co, ci, k in synth.TABLE1_LAYERS]
    else:
        layers = [(co, ci, k) for _, co, ci, k in NETS[net].layers()]
    parts = []
    for co, ci, k in layers:
        parts.append(torch.randn(co * k * k * ci, device="cuda", generator=g) * math.sqrt(2.0 / (ci * k * k)))
        parts.append(torch.randn(co, device="cuda", generator=g) * 0.02)
    return torch.cat(parts)


def _inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    s = {"w": _weights(case["net"], g)} if "net" in case else {}
    sz = sizes(case)
    left, right, gt = [None] * len(sz), [None] * len(sz), [None] * len(sz)
    for size in dict.fromkeys(sz):
        at = [i for i, x in enumerate(sz) if x == size]
        L, R, d = _scene(g, len(at), *size)
        for j, i in enumerate(at):
            left[i], right[i], gt[i] = L[j], R[j], d[j]
    s.update(sizes=sz, left=left, right=right)
    if case["kind"] in ("refine", "train"):
        # a matcher's map: the scene's disparity at quarter size with 3 % wrong matches
        s["coarse"] = []
        for (W, H, D), d in zip(sz, gt):
            c = (d[2::4, 2::4][:H // 4, :W // 4] / 4).round()
            wrong = torch.rand(c.shape, device="cuda", generator=g) < 0.03
            c = torch.where(wrong, torch.randint(0, D, c.shape, device="cuda", generator=g).float(), c)
            s["coarse"].append(c.clamp(0, D - 1).to(torch.int16).contiguous())
    if case["kind"] == "train":
        lat = NETS[case["net"]].latent
        s["coarse"] = [c.float() for c in s["coarse"]]
        s["gt"] = [d.contiguous() for d in gt]
        s["eps"] = [torch.randn(*_levels(H, W)[3], lat, device="cuda", generator=g) for W, H, _ in sz]
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    kind, sz = case["kind"], s["sizes"]
    if "net" in case:
        s["ctx"] = binding.Context(NETS[case["net"]], case["k"], case["form"])
        s["ctx"].set_weights(s["w"])
    else:
        s["ctx"] = binding.Context(synth.NET_SMALL, case["k"], "bf16")
    s["pairs"] = [binding.DevicePair(L, R, W, H, D) for L, R, (W, H, D) in zip(s["left"], s["right"], sz)]
    if kind == "coarse":
        s["out"] = [torch.empty(H // 4, W // 4, dtype=torch.int16, device="cuda") for W, H, _ in sz]
    elif kind == "variant":
        s["opts"] = binding.coarse_opts(case["cost"], case["agg"], dt_iters=case["iters"], smp=case["post"],
                                        median=case["post"], P1=0.1 if case["cost"] == "zncc" else 1.0,
                                        P2=0.5 if case["cost"] == "zncc" else 6.0)
    elif kind in ("pipeline", "refine"):
        s["out"] = [torch.empty(H, W, device="cuda") for W, H, _ in sz]
        s["stream"] = _stream()
    elif kind == "host":
        s["stream"] = _stream()
        s["host"] = []
        for imgs in (s["left"], s["right"]):
            s["host"].append([torch.empty(t.shape, dtype=torch.uint8, pin_memory=True).copy_(t) for t in imgs])
        s["out"] = [torch.empty(H, W, pin_memory=True) for W, H, _ in sz]
        s["args"] = ([W for W, _, _ in sz], [H for _, H, _ in sz], [t.stride(0) for t in s["left"]],
                     [D for _, _, D in sz])
    else:
        s["step"] = 0
    return s


def run(s):
    kind, ctx = s["case"]["kind"], s["ctx"]
    if kind == "coarse":
        if s["case"]["scores"]:
            disp, best, second = ctx.coarse_match(s["pairs"], scores=True, out=s["out"])
            return {"disp": disp, "best": best, "second": second}
        return ctx.coarse_match(s["pairs"], out=s["out"])
    if kind == "variant":
        return ctx.coarse_match_ex(s["pairs"], s["opts"])
    if kind == "pipeline":
        return ctx.pipeline(s["pairs"], stream=s["stream"], out=s["out"])
    if kind == "refine":
        return ctx.refine(s["pairs"], s["coarse"], stream=s["stream"], out=s["out"])
    if kind == "host":
        W, H, pitch, D = s["args"]
        return ctx.pipeline_host(s["host"][0], s["host"][1], W, H, pitch, D, s["out"], stream=s["stream"])
    # the weights move with every step, as in a user's loop
    Y, mu, lv = ctx.refine_train(s["pairs"], s["coarse"], s["eps"])
    loss, gY, gmu, glv = ctx.loss(s["pairs"], Y, s["gt"], mu, lv, KL_WEIGHT)
    grad, _ = ctx.refine_backward(gY, gmu, glv, False, s["coarse"])
    s["step"] += 1
    ctx.adam_step(grad, s["step"])
    return {"Y": Y, "mu": mu, "logvar": lv, "loss": loss, "grad": grad}


# ---------------------------------------------------------------- 64-bit values
def _conv(x, w, b, stride=1):
    """[Ci, H, W] with w [Co, k, k, Ci], zero padding k // 2, as k * k matrix products."""
    k = w.shape[1]
    H, W = x.shape[1], x.shape[2]
    Ho, Wo = (H + stride - 1) // stride, (W + stride - 1) // stride
    xp = F.pad(x, (k // 2,) * 4)
    out = b[:, None]
    for ky in range(k):
        for kx in range(k):
            v = xp[:, ky:ky + (Ho - 1) * stride + 1:stride, kx:kx + (Wo - 1) * stride + 1:stride]
            out = out + w[:, ky, kx] @ v.reshape(x.shape[0], -1)
    return out.reshape(-1, Ho, Wo)


def _deconv(x, w, b, hw):
    """Stride-2 transposed convolution, padding k // 2, output 2n cropped to hw."""
    z = torch.zeros(x.shape[0], 2 * x.shape[1], 2 * x.shape[2], dtype=x.dtype, device=x.device)
    z[:, ::2, ::2] = x
    return _conv(z, w.flip(1, 2), b)[:, :hw[0], :hw[1]]


def _bilinear(c, H, W, scale):
    """[h, w] sampled at half-pixel centres on H x W, source clamped."""
    h, w = c.shape
    sx = ((torch.arange(W, device=c.device, dtype=c.dtype) + 0.5) / scale - 0.5).clamp(0, w - 1)
    sy = ((torch.arange(H, device=c.device, dtype=c.dtype) + 0.5) / scale - 0.5).clamp(0, h - 1)
    x0, y0 = sx.long(), sy.long()
    x1, y1 = (x0 + 1).clamp(max=w - 1), (y0 + 1).clamp(max=h - 1)
    fx, fy = sx - x0, (sy - y0)[:, None]
    top = (1 - fx) * c[y0][:, x0] + fx * c[y0][:, x1]
    bot = (1 - fx) * c[y1][:, x0] + fx * c[y1][:, x1]
    return (1 - fy) * top + fy * bot


def _split(layers, flat):
    out, o = {}, 0
    for name, co, ci, k in layers:
        n = co * k * k * ci
        out[name] = (flat[o:o + n].view(co, k, k, ci), flat[o + n:o + n + co])
        o += n + co
    return out


def _refine64(P, left, coarse, eps=None):
    """The small network in 64 bits: (Y, mu, logvar) with latents [H3, W3, C]."""
    H, W = left.shape
    lv = _levels(H, W)
    U = 4 * _bilinear(coarse, H, W, 4)
    x = torch.stack([left / 256, U / 256])
    for n in ("enc1", "enc2", "enc3"):
        x = _conv(x, *P[n], stride=2).relu()
    mu = _conv(x, *P["mu"])
    logvar = None
    z = mu
    if eps is not None:
        logvar = _conv(x, *P["logvar"])
        z = mu + eps.permute(2, 0, 1) * (logvar / 2).exp()
    for n, (h, w) in (("dec1", lv[2]), ("dec2", lv[1]), ("dec3", lv[0])):
        z = z.repeat_interleave(2, 1)[:, :h].repeat_interleave(2, 2)[:, :, :w]
        z = _conv(z, *P[n]).relu()
    Y = U + _conv(z, *P["final"])[0]
    return Y, mu.permute(1, 2, 0), None if logvar is None else logvar.permute(1, 2, 0)


def _table1_64(P, left, coarse):
    H, W = left.shape
    lv = _levels(H, W)
    act = lambda v: F.leaky_relu(v, 0.1)  # noqa: E731
    (h2, w2), (h4, w4), (h8, w8) = lv[1:]
    Lp = F.pad(left[None, None], (0, 2 * w2 - W, 0, 2 * h2 - H), mode="replicate")
    X1 = F.avg_pool2d(Lp, 2)[0] / 256
    X0 = 4 * _bilinear(coarse, h2, w2, 2)[None] / 256
    fe1, fe2 = act(_conv(X0, *P["FE_1"])), act(_conv(X1, *P["FE_2"]))
    en1 = act(_conv(torch.cat([fe1, fe2]), *P["EN_1"], stride=2))
    en1r = act(_conv(en1, *P["EN_1_R"]))
    en2 = act(_conv(torch.cat([en1, en1r]), *P["EN_2"], stride=2))
    en2r = act(_conv(en2, *P["EN_2_R"]))
    mu = _conv(torch.cat([en2, en2r]), *P["heads"])[:1]
    d1 = act(_conv(mu - 1, *P["D_1"]))
    d1r = act(_conv(torch.cat([d1, en2, en2r]), *P["D_1_R"]))
    d2 = act(_deconv(torch.cat([d1, en2, en2r, d1r]), *P["D_2"], (h4, w4)))
    d2r = act(_conv(torch.cat([d2, en1, en1r]), *P["D_2_R"]))
    d = act(_deconv(torch.cat([d2, en1, en1r, d2r]), *P["D"], (h2, w2)))
    return 256 * _deconv(torch.cat([d, X0, fe1, fe2]), *P["Y"], (H, W))[0]


def _zncc64(left, right, k, D):
    """(disparity, best score, best of the others) per quarter-size pixel; sums are whole numbers
    below 2^53, so only the last division rounds."""
    def box(v):
        h, w = v.shape[0] // 4, v.shape[1] // 4
        return v[:4 * h, :4 * w].reshape(h, 4, w, 4).sum((1, 3))

    def window(v):
        v = sum(v[i:v.shape[0] - k + 1 + i] for i in range(k))
        return sum(v[:, i:v.shape[1] - k + 1 + i] for i in range(k))

    r, N = k // 2, k * k
    L, R = (F.pad(box(v)[None, None], (r,) * 4, mode="replicate")[0, 0] for v in (left, right))
    sl, sr = window(L), window(R)
    vl, vr = N * window(L * L) - sl * sl, N * window(R * R) - sr * sr
    h, w = sl.shape
    rho = torch.full((D, h, w), -2.0, dtype=torch.float64, device=left.device)
    for d in range(D):
        e = w - d
        num = N * window(L[:, d:] * R[:, :R.shape[1] - d]) - sl[:, d:] * sr[:, :e]
        den = vl[:, d:].sqrt() * vr[:, :e].sqrt()
        rho[d, :, d:] = torch.where(den > 0, num / den, 0.0)
    best, at = rho.max(0)
    at = (rho == best).to(torch.int8).argmax(0)  # the lowest d of a tie
    second = rho.scatter(0, at[None], -2.0).amax(0)
    return at, best, second


def exact(case, seed):
    kind = case["kind"]
    if kind == "variant" or (kind == "coarse" and not case["scores"]):
        return None  # whole numbers
    s = _inputs(case, seed)
    f64 = [(L[:, :W].double(), R[:, :W].double(), D) for L, R, (W, _, D) in zip(s["left"], s["right"], s["sizes"])]
    if kind == "coarse":
        got = [_zncc64(L, R, case["k"], D) for L, R, D in f64]
        return {"disp": [None] * len(got), "best": [b for _, b, _ in got], "second": [x for _, _, x in got]}
    table1 = case["net"] == "table1"
    layers = synth.TABLE1_LAYERS if table1 else NETS[case["net"]].layers()
    flat = s["w"].double()
    if kind == "train":
        flat.requires_grad_(True)
        P = _split(layers, flat)
        n_px = sum(W * H for W, H, _ in s["sizes"])
        n_lat = sum(e.numel() for e in s["eps"])
        out = {"Y": [], "mu": [], "logvar": []}
        rec = kl = 0.0
        for (L, _, _), c, e, gt in zip(f64, s["coarse"], s["eps"], s["gt"]):
            Y, mu, lv = _refine64(P, L, c.double(), e.double())
            a = F.smooth_l1_loss(Y, gt.double(), reduction="sum") / n_px
            b = 0.5 * (mu * mu + lv.exp() - 1 - lv).sum() / n_lat
            (a + KL_WEIGHT * b).backward()
            rec, kl = rec + a.detach(), kl + b.detach()
            for name, v in (("Y", Y), ("mu", mu), ("logvar", lv)):
                out[name].append(v.detach())
            del Y, mu, lv, a, b
        return {**out, "loss": torch.stack([rec + KL_WEIGHT * kl, rec, kl]), "grad": flat.grad}
    P = _split(layers, flat)
    out = []
    with torch.no_grad():
        for i, (L, R, D) in enumerate(f64):
            c = s["coarse"][i].double() if kind == "refine" else _zncc64(L, R, case["k"], D)[0].double()
            Y = (_table1_64 if table1 else _refine64)(P, L, c)
            out.append(Y if table1 else Y[0])
    return [v.cpu() for v in out] if kind == "host" else out
