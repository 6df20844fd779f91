"""The work that users of this library have it do, as cases that can be timed.

Every case goes through the public Python entry points (``codec.Codec``,
``codec.DecodePlan``, ``codec.LocalModel``, ``codec.LocalModelNLL``,
``nlc.nlc_compress`` into a buffer that the program keeps).  A case
is a dict of plain values:

  kind    decode, plan, encode, roundtrip, sample, bits, nll, adjoint, model
  h, C, R, K, prec     the model (prec: fp32, bf16, sheared)
  n, H, W              n images of H x W; with lo > 0 their sides are drawn
                       from lo .. H and lo .. W instead (an uneven batch)
  big                  side of one more, larger image in front (0: none)
  patch                side of the coding units (0: whole images)
  layout, sched        stream layout and decode schedule, where they apply

The images are natural-image-like (1/f Gaussian field, mixed channels,
constant-colour polygons with hard edges, sensor noise), the models predict
them as a trained one does: random hidden layers under a head that is fitted
to such images, so that code lengths, posteriors and the number of active
mixture components are those of real use.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2201_05213_gb300 import codec as CD
from paper_2201_05213_gb300 import nlc as N
from paper_2201_05213_gb300 import synth

PREC = {"fp32": N.NLC_FP32, "bf16": N.NLC_BF16, "sheared": N.NLC_BF16_SHEARED}
SCHED = {"raster": N.NLC_SCHED_RASTER, "wavefront": N.NLC_SCHED_WAVEFRONT,
         "sequential": N.NLC_SCHED_SEQUENTIAL}
DEV = "cuda"
MAX_PX = 12 * 1024 * 1024  # pixels of the largest listed case


def _case(kind, prec="bf16", h=3, C=64, R=2, K=10, n=1, H=32, W=32, lo=0, big=0, patch=0,
          layout="row", sched="wavefront", **more):
    return dict(kind=kind, prec=prec, h=h, C=C, R=R, K=K, n=n, H=H, W=W, lo=lo, big=big,
                patch=patch, layout=layout, sched=sched, **more)


def listed():
    return [
        # the smallest use: one thumbnail to a file and back with the paper's plain method (one
        # stream, pixel after pixel, FP32)
        dict(_case("roundtrip", "fp32", C=32, layout="unit", sched="sequential"),
             name="roundtrip_thumb_fp32"),
        # opening one picture: nothing but its own wavefront to run in parallel
        dict(_case("decode", H=384, W=509), name="decode_picture_bf16"),
        # a batch of pictures of unlike sizes in one call (a data loader, an album)
        dict(_case("decode", n=48, H=512, W=512, lo=32), name="decode_uneven_bf16"),
        # many small images under the FP32 model, one stream per row
        dict(_case("decode", "fp32", n=64, H=64, W=64), name="decode_small_fp32"),
        # serving large images: patches of all images decoded in parallel, a plan kept for the
        # batch shape
        dict(_case("plan", n=8, H=1024, W=1024, big=2048, patch=256), name="decode_large_bf16"),
        # the sheared variant on large images
        dict(_case("decode", "sheared", n=4, H=1024, W=1024, patch=256),
             name="decode_large_sheared"),
        # compressing the same large images (an archive being written)
        dict(_case("encode", n=8, H=1024, W=1024, big=2048, patch=256), name="encode_large_bf16"),
        # drawing images from the model
        dict(_case("sample", n=64, H=64, W=64), name="sample_small_bf16"),
        # held-out code length while a model trains
        dict(_case("bits", n=256, H=32, W=32), name="bits_heldout_bf16"),
        # a training step with the user's own optimizer: weights in, loss and gradient out
        dict(_case("nll", n=128, H=32, W=32), name="train_bf16"),
        # the FP32 model's training step
        dict(_case("adjoint", "fp32", n=64, H=32, W=32), name="train_fp32"),
        # the network under a loss of the user's own: outputs forward, their gradient back
        dict(_case("model", h=2, n=32, H=32, W=32), name="model_autograd_bf16"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode", "decode", "plan", "encode", "encode", "roundtrip", "sample", "bits",
                       "nll", "adjoint", "model"])
    prec = rng.choice(["bf16", "bf16", "fp32", "sheared"])
    h = rng.choice([1, 2, 3])
    C = rng.choice([32, 64, 64])
    R = rng.choice([0, 1, 2, 2])
    K = rng.choice([5, 10, 10])
    if kind in ("nll", "adjoint", "model"):
        if kind == "nll" and prec == "sheared":
            prec = "bf16"
        side = rng.randint(24, 64)
        most = (1 << 17) if prec != "fp32" and kind != "model" else (1 << 16)
        n = _log_int(rng, 1, max(1, most // (side * side)))
        return _case(kind, prec, h, C, R, K, n, side, rng.randint(24, 64) if n > 1 else side)
    if kind == "roundtrip":
        return _case(kind, prec, h, C, R, K, 1, rng.randint(8, 48), rng.randint(8, 40), layout="unit",
                     sched=rng.choice(["sequential", "raster"]))
    if kind == "sample":
        return _case(kind, prec, h, C, R, K, _log_int(rng, 1, 64), rng.randint(16, 128),
                     rng.randint(16, 128), patch=rng.choice([0, 64]), gen=rng.randint(0, 1 << 30))
    H, W = _log_int(rng, 16, 1200), _log_int(rng, 16, 1200)
    patch = rng.choice([0, 64, 128, 256]) if max(H, W) <= 512 else rng.choice([128, 200, 256])
    most = MAX_PX // 2 if prec != "fp32" else 1 << 20
    n = _log_int(rng, 1, max(1, min(48, most // (H * W))))
    if H * W * n > most:
        H = W = 700
        n = 1
    if kind == "bits":
        return _case(kind, prec, h, C, R, K, n, H, W, patch=patch)
    lo = 16 if n > 1 and rng.random() < 0.4 else 0
    return _case(kind, prec, h, C, R, K, n, H, W, lo=lo, patch=patch)


# ------------------------------------------------------------------ inputs

def _image(gen, H, W, n_poly):
    """One H x W x 3 uint8 image on the GPU."""
    spec = torch.fft.rfft2(torch.randn((3, H, W), generator=gen, device=DEV))
    fy = torch.fft.fftfreq(H, device=DEV)[:, None]
    fx = torch.fft.rfftfreq(W, device=DEV)[None, :]
    f = torch.sqrt(fx * fx + fy * fy)
    f[0, 0] = math.inf
    fields = torch.fft.irfft2(spec / f, s=(H, W))
    mixed = torch.einsum("ck,khw->hwc", torch.randn((3, 3), generator=gen, device=DEV), fields)
    mixed = mixed - mixed.mean(dim=(0, 1), keepdim=True)
    img = 128.0 + 40.0 * mixed / mixed.std(dim=(0, 1), keepdim=True).clamp_min(1e-6)
    y = torch.arange(H, device=DEV)[:, None] + 0.5
    x = torch.arange(W, device=DEV)[None, :] + 0.5
    v = torch.rand((n_poly, 3, 2), generator=gen, device=DEV) * torch.tensor([H, W], device=DEV)
    colour = torch.randint(0, 256, (n_poly, 3), generator=gen, device=DEV).float()
    for p in range(n_poly):
        side = []
        for a in range(3):
            (ya, xa), (yb, xb) = v[p, a], v[p, (a + 1) % 3]
            side.append((y - ya) * (xb - xa) - (x - xa) * (yb - ya) > 0)
        inside = (side[0] == side[1]) & (side[1] == side[2])
        img = torch.where(inside[..., None], colour[p], img)
    img = img + 2.0 * torch.randn(img.shape, generator=gen, device=DEV)
    return img.round().clamp(0, 255).to(torch.uint8).contiguous()


def _sizes(case):
    rng = np.random.default_rng([case["n"], case["H"], case["W"]])
    sizes = [(case["big"], case["big"])] if case["big"] else []
    for _ in range(case["n"]):
        if case["lo"]:
            sizes.append((int(rng.integers(case["lo"], case["H"] + 1)),
                          int(rng.integers(case["lo"], case["W"] + 1))))
        else:
            sizes.append((case["H"], case["W"]))
    return sizes


def _images(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(1 + seed)
    return [_image(gen, H, W, 4 if H * W <= 512 * 512 else 16) for H, W in _sizes(case)]


def _batch(case, seed):
    """N x H x W x 3 crops, several from one picture."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(2 + seed)
    n, H, W = case["n"], case["H"], case["W"]
    rng = np.random.default_rng([seed, 2])
    out = torch.empty((n, H, W, 3), dtype=torch.uint8, device=DEV)
    src = None
    for k in range(n):
        if k % 16 == 0:
            src = _image(gen, 256, 256, 4)
        y, x = int(rng.integers(0, 257 - H)), int(rng.integers(0, 257 - W))
        out[k] = src[y:y + H, x:x + W]
    return out


def _weights(case, seed):
    """A model that predicts such images: random hidden layers, and a head fitted by least squares
    (locations with channel coupling, log-scales from the residuals, components spread around)."""
    h, C, R, K = case["h"], case["C"], case["R"], case["K"]
    w = synth.xavier_weights(h, C, R, K, seed=seed).astype(np.float64)
    mats, at = {}, 0
    for name, shp in synth.weight_shapes(h, C, R, K):
        size = int(np.prod(shp))
        mats[name] = w[at:at + size].reshape(shp)
        at += size
    img = synth.make_image(seed, 96, 96)
    rng = np.random.default_rng([seed, 3])
    ys, xs = rng.integers(h, 96, 2048), rng.integers(h, 96 - h, 2048)
    v = (2.0 * img - 255.0) / 255.0
    taps = [(dy, dx) for dy in range(-h, 1) for dx in range(-h, h + 1) if dy < 0 or dx < 0]
    x = np.concatenate([v[ys + dy, xs + dx] for dy, dx in taps], axis=1)

    def elu(t):
        return np.where(t > 0, t, np.expm1(np.minimum(t, 0)))

    a = x @ mats["W0"].T + mats["b0"]
    for r in range(R):
        z = elu(a) @ mats[f"W1_{r}"].T + mats[f"b1_{r}"]
        a = a + elu(z) @ mats[f"W2_{r}"].T + mats[f"b2_{r}"]
    f = np.concatenate([elu(a), np.ones((len(a), 1))], axis=1)
    t = v[ys, xs]
    WH, bH = mats["WH"], mats["bH"]
    WH *= 0.3
    raw = np.zeros(3)  # alpha, beta, gamma before tanh
    for c in range(3):
        g = np.concatenate([f, t[:, :c]], axis=1)
        s = np.linalg.solve(g.T @ g + 1e-3 * len(g) * np.eye(g.shape[1]), g.T @ t[:, c])
        couple = np.clip(s[f.shape[1]:], -0.9, 0.9)
        if c == 1:
            raw[0] = np.arctanh(couple[0])
        if c == 2:
            raw[1:] = np.arctanh(couple)
        std = max(np.std(t[:, c] - g @ s), 4.0 / 255.0)
        for k in range(K):
            WH[(1 + c) * K + k] = s[:C] * (1.0 + 0.02 * rng.standard_normal())
            bH[(1 + c) * K + k] = s[C] + 0.7 * std * rng.standard_normal()
            bH[(4 + c) * K + k] = math.log(0.5 * std) + 0.6 * rng.standard_normal()
    for c in range(3):
        bH[(7 + c) * K:(8 + c) * K] = raw[c]
    return np.concatenate([mats[name].ravel()
                           for name, _ in synth.weight_shapes(h, C, R, K)]).astype(np.float32)


def prepare(case, seed):
    seed = int(seed)
    kind = case["kind"]
    layout = N.NLC_LAYOUT_UNIT if case["layout"] == "unit" else N.NLC_LAYOUT_ROW
    s = dict(case=case, layout=layout, sched=SCHED[case["sched"]], patch=case["patch"],
             w=_weights(case, seed))
    cd = s["codec"] = CD.Codec(case["h"], case["C"], case["R"], case["K"], PREC[case["prec"]], s["w"])
    if kind in ("nll", "adjoint", "model"):
        s["batch"] = _batch(case, seed)
        if kind != "adjoint":
            s["weights"] = torch.from_numpy(s["w"]).to(DEV).requires_grad_()
        if kind == "model":  # some loss of the user's own: a weighted sum of squares
            gen = torch.Generator(device=DEV)
            gen.manual_seed(3 + seed)
            s["target"] = torch.randn((1, 10 * case["K"]), generator=gen, device=DEV)
        return s
    if kind == "sample":
        s["sizes"], s["seed"] = _sizes(case), seed + case.get("gen", 0)
        return s
    s["imgs"] = _images(case, seed)
    s["sizes"] = [(int(t.shape[0]), int(t.shape[1])) for t in s["imgs"]]
    if kind in ("encode", "roundtrip"):  # the buffer that the program writes files from
        cap = N.nlc_compress_bound(s["sizes"], s["patch"], layout)
        s["data"] = torch.zeros(cap, dtype=torch.uint8, device=DEV)
        s["offs"] = torch.zeros(len(s["sizes"]) + 1, dtype=torch.int64, device=DEV)
    if kind in ("decode", "plan"):
        s["data"], s["offs"] = cd.compress(s["imgs"], s["patch"], layout)
        del s["imgs"]
    if kind == "plan":
        s["plan"] = cd.plan(s["sizes"], s["patch"], layout, s["sched"])
    return s


# --------------------------------------------------------------------- run

def _compress(s):
    cd = s["codec"]
    N.nlc_compress(cd.ctx, s["imgs"], s["patch"], s["layout"], s["data"], s["offs"])
    cd.check()
    return s["data"], s["offs"]


def run(s):
    cd, kind = s["codec"], s["case"]["kind"]
    if kind == "decode":
        return cd.decompress(s["data"], s["offs"], s["sizes"], s["patch"], s["layout"], s["sched"])
    if kind == "plan":
        return s["plan"].run(s["data"], s["offs"])
    if kind == "encode":
        return _compress(s)
    if kind == "roundtrip":
        data, offs = _compress(s)
        return [data, offs, cd.decompress(data, offs, s["sizes"], s["patch"], s["layout"], s["sched"])]
    if kind == "sample":
        return cd.sample(s["sizes"], s["patch"], s["seed"])
    if kind == "bits":
        return cd.forward(s["imgs"], s["patch"], params=False, bits=True)[1]
    if kind == "adjoint":
        return cd.loss_grad(s["batch"])
    s["weights"].grad = None
    if kind == "nll":
        loss = CD.LocalModelNLL.apply(s["weights"], cd, s["batch"])
        loss.backward()
        return loss.detach(), s["weights"].grad
    out = CD.LocalModel.apply(s["weights"], cd, s["batch"])
    loss = (out - s["target"]).square().mean()
    loss.backward()
    return out.detach(), s["weights"].grad


# ----------------------------------------------------- work and exact values

def _pixels(case):
    if case["lo"]:
        return case["n"] * (case["lo"] + case["H"]) * (case["lo"] + case["W"]) // 4
    return case["big"] ** 2 + case["n"] * case["H"] * case["W"]


def work(case):
    h, C, R, K = case["h"], case["C"], case["R"], case["K"]
    px = _pixels(case)
    n_w = synth.num_weights(h, C, R, K)
    flops = 2.0 * px * (6 * h * (h + 1) * C + 2 * R * C * C + 10 * K * C)
    image, container, outputs = 3.0 * px, 1.8 * px, 40.0 * K * px
    kind = case["kind"]
    if kind in ("decode", "plan", "encode"):
        nbytes = image + container
    elif kind == "roundtrip":
        nbytes, flops = 2 * (image + container), 2 * flops
    elif kind == "sample":
        nbytes = image
    elif kind == "bits":
        nbytes = image + 4.0 * px
    elif kind in ("nll", "adjoint"):
        nbytes, flops = image + 4.0 * n_w, 3 * flops
    else:  # outputs written, their gradient read
        nbytes, flops = 2 * image + 2 * outputs + 8.0 * n_w, 4 * flops
    return {"bytes": nbytes + 4.0 * n_w, "flops": flops}


def _outputs64(case, w, units):
    """Network outputs (pixels x 10K, FP64) of a list of units, in raster order."""
    h, C, R, K = case["h"], case["C"], case["R"], case["K"]
    mats, at = {}, 0
    for name, shp in synth.weight_shapes(h, C, R, K):
        size = int(np.prod(shp))
        mats[name] = w[at:at + size].reshape(shp)
        at += size
    xs = []
    for u in units:
        v = (2.0 * u.double() - 255.0) / 255.0
        p = torch.nn.functional.pad(v, (0, 0, h, h, h, 0))
        H, W = u.shape[:2]
        xs.append(torch.cat([p[h + dy:h + dy + H, h + dx:h + dx + W] for dy in range(-h, 1)
                             for dx in range(-h, h + 1) if dy < 0 or dx < 0],
                            dim=2).reshape(H * W, -1))
    elu = torch.nn.functional.elu
    a = torch.cat(xs) @ mats["W0"].T + mats["b0"]
    for r in range(R):
        z = elu(a) @ mats[f"W1_{r}"].T + mats[f"b1_{r}"]
        a = a + elu(z) @ mats[f"W2_{r}"].T + mats[f"b2_{r}"]
    return elu(a) @ mats["WH"].T + mats["bH"]


def _bits64(case, P, v):
    """-log2 of the joint discretized logistic mixture of pixels v (n x 3) under outputs P."""
    K = case["K"]
    x = (2.0 * v.double() - 255.0) / 255.0
    logpi = torch.log_softmax(P[:, :K], dim=1)
    co = torch.tanh(P[:, 7 * K:])
    m = [P[:, K:2 * K], P[:, 2 * K:3 * K] + co[:, :K] * x[:, :1],
         P[:, 3 * K:4 * K] + co[:, K:2 * K] * x[:, :1] + co[:, 2 * K:] * x[:, 1:2]]
    ls = torch.nn.functional.logsigmoid
    l = logpi
    for c in range(3):
        inv = torch.exp(-torch.clamp_min(P[:, (4 + c) * K:(5 + c) * K], -7.0))
        b = v[:, c:c + 1].double()
        lo, hi = (2 * b - 256) / 255, (2 * b - 254) / 255
        a_hi, a_lo, d = (hi - m[c]) * inv, (lo - m[c]) * inv, (2.0 / 255.0) * inv
        mid = ls(a_hi) + ls(-a_lo) + torch.log(-torch.expm1(-d))
        l = l + torch.where(b == 0, ls(a_hi), torch.where(b == 255, ls(-a_lo), mid))
    return -torch.logsumexp(l, dim=1) / math.log(2.0)


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("bits", "nll", "adjoint", "model"):
        return None  # bytes and pixels
    seed = int(seed)
    w = torch.from_numpy(_weights(case, seed)).double().to(DEV)
    if kind == "bits":
        P = case["patch"] or max(case["H"], case["W"])
        out = []
        for img in _images(case, seed):
            H, W = img.shape[:2]
            bits = torch.empty((H, W), dtype=torch.float64, device=DEV)
            for y in range(0, H, P):
                for x in range(0, W, P):
                    u = img[y:y + P, x:x + P]
                    b = _bits64(case, _outputs64(case, w, [u]), u.reshape(-1, 3))
                    bits[y:y + P, x:x + P] = b.reshape(u.shape[:2])
            out.append(bits.reshape(-1))
        return torch.cat(out)
    batch = _batch(case, seed)
    w.requires_grad_()
    if kind == "model":
        gen = torch.Generator(device=DEV)
        gen.manual_seed(3 + seed)
        target = torch.randn((1, 10 * case["K"]), generator=gen, device=DEV).double()
        out = _outputs64(case, w, list(batch))
        (out - target).square().mean().backward()
        return out.detach(), w.grad
    grad, total, px = torch.zeros_like(w), 0.0, batch.shape[0] * batch.shape[1] * batch.shape[2]
    for part in batch.split(16):
        loss = _bits64(case, _outputs64(case, w, list(part)), part.reshape(-1, 3)).sum() / (3 * px)
        grad += torch.autograd.grad(loss, w)[0]
        total = total + loss.detach()
    return (total.reshape(1), grad) if kind == "adjoint" else (total, grad)
