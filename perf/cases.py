"""The work that users of the framework have it do, as cases that can be run
and timed: transforms of image batches, the differentiable layer, the unrolled
inpainting iteration, the 3x3 convolution blocks of the learned parts, the
threshold network and the ray transform, each through its public entry points.

``listed()`` names the usual sizes (the configurations of the benchmark and of
``measure.py``); ``draw()`` gives more cases of the same ranges, odd sizes among
them.  ``exact()`` restates a case in float64 with plain torch.
"""

from __future__ import annotations

import functools
import math

import torch

DEV = "cuda:0"
DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}
DIRECTIONS = (8, 8, 16, 16)          # filters per scale: 17, 33 and 49 with the low-pass
LPD_PAIRS = ((6, 32), (7, 32), (32, 32), (32, 5), (33, 32), (32, 33), (102, 32), (32, 85))


def listed():
    return [
        # one small image: the plain transform of a single 256 x 256 picture, bound by launches
        {"name": "transform_256_b1", "kind": "transform", "rows": 256, "cols": 256, "scales": 2,
         "batch": 1, "dtype": "f32", "complex": False},
        # the headline workload: a batch of 512 x 512 images, 49 filters, there and back
        {"name": "transform_512_b16", "kind": "transform", "rows": 512, "cols": 512, "scales": 4,
         "batch": 16, "dtype": "f32", "complex": False},
        # the largest point of the throughput sweep, coefficients stored in 16 bits
        {"name": "transform_1024_b8_bf16", "kind": "transform", "rows": 1024, "cols": 1024,
         "scales": 4, "batch": 8, "dtype": "bf16", "complex": False},
        # camera-sized frames: sides that are no powers of two
        {"name": "transform_480x640_b16", "kind": "transform", "rows": 480, "cols": 640,
         "scales": 4, "batch": 16, "dtype": "f32", "complex": False},
        # prime sides, as a cropped scan may have
        {"name": "transform_509_b4", "kind": "transform", "rows": 509, "cols": 509, "scales": 4,
         "batch": 4, "dtype": "f32", "complex": False},
        # the differentiable layer inside a training step, forward and backward
        {"name": "layer_256_b32_bf16", "kind": "layer", "rows": 256, "cols": 256, "scales": 3,
         "batch": 32, "dtype": "bf16", "complex": False},
        # two unrolled inpainting iterations with the relaxed threshold, forward and backward, as
        # the threshold network is trained
        {"name": "relaxed_iht_512_b4", "kind": "relaxed", "rows": 512, "cols": 512, "scales": 4,
         "batch": 4, "iterations": 2, "complex": False},
        # one iteration of the plain inpainting loop early in its schedule, where few coefficients
        # are kept and none lies at its threshold
        {"name": "shrink_512_b2", "kind": "shrink", "rows": 512, "cols": 512, "scales": 4,
         "batch": 2, "complex": False},
        # first block of the coefficient network in a training step
        {"name": "conv_33_32_256_b32", "kind": "conv", "ci": 33, "co": 32, "rows": 256,
         "cols": 256, "batch": 32},
        # first block of the shearlet-domain primal network of the learned reconstruction
        {"name": "conv_102_32_128_b4", "kind": "conv", "ci": 102, "co": 32, "rows": 128,
         "cols": 128, "batch": 4},
        # tomography: projections and back-projections of a batch of slices
        {"name": "ray_512_b8", "kind": "ray", "n": 512, "angles": 180, "batch": 8},
        # the threshold network at inference, before a learned inpainting
        {"name": "threshold_net_512_b8", "kind": "net", "rows": 512, "cols": 512, "batch": 8,
         "filters": 49, "iterations": 15},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["transform"] * 4 + ["general"] * 4 + ["layer", "relaxed", "shrink"]
                      + ["conv"] * 2 + ["ray"] * 2 + ["net"])
    scales = rng.randint(2, 4)
    K = _filters(scales)
    if kind in ("transform", "layer", "relaxed", "shrink"):
        top = 10 if kind == "transform" else 9
        rows, cols = 1 << rng.randint(6, top), 1 << rng.randint(6, top)
        budget = {"transform": 400e6, "layer": 70e6, "relaxed": 50e6, "shrink": 26e6}[kind]
        most = max(1, min(32 if kind != "shrink" else 2, int(budget / (K * rows * cols))))
        case = {"kind": kind, "rows": rows, "cols": cols, "scales": scales,
                "batch": _log_int(rng, 1, most), "complex": False}
        if kind in ("transform", "layer"):
            case["dtype"] = rng.choice(("f32", "bf16"))
        if kind == "relaxed":
            case["iterations"] = rng.randint(1, 3)
        return case
    if kind == "general":
        rows, cols = _log_int(rng, 48, 900), _log_int(rng, 48, 900)
        most = max(1, min(16, int(50e6 / (K * rows * cols))))
        return {"kind": "transform", "rows": rows, "cols": cols, "scales": scales,
                "batch": _log_int(rng, 1, most), "dtype": rng.choice(("f32", "f32", "bf16")),
                "complex": rng.random() < 0.25}
    if kind == "conv":
        ci, co = rng.choice(LPD_PAIRS)
        rows, cols = _log_int(rng, 24, 256), _log_int(rng, 24, 256)
        if rng.random() < 0.75:
            cols += cols % 2
        most = max(1, min(32, int((2e6 if cols % 2 == 0 else 2e5) / (rows * cols) * 32 / max(ci, co))))
        return {"kind": "conv", "ci": ci, "co": co, "rows": rows, "cols": cols,
                "batch": _log_int(rng, 1, most)}
    if kind == "ray":
        n, angles = _log_int(rng, 64, 700), _log_int(rng, 30, 360)
        most = max(1, min(32, int(530e6 / (angles * 1.42 * n * n))))
        return {"kind": "ray", "n": n, "angles": angles, "batch": _log_int(rng, 1, most)}
    rows, cols = 8 * _log_int(rng, 16, 80), 8 * _log_int(rng, 16, 80)
    return {"kind": "net", "rows": rows, "cols": cols, "batch": _log_int(rng, 1, 16),
            "filters": K, "iterations": rng.choice((10, 15, 20))}


# ------------------------------------------------------------------- inputs
def _filters(scales):
    return 1 + sum(DIRECTIONS[:scales])


def _spectra(rows, cols, scales, cplx, device="cpu"):
    """[K, rows, cols] float64 directional wedges over dyadic rings and a
    low-pass, even (or, shifted in space by whole pixels, Hermitian)."""
    ky = torch.fft.fftfreq(rows, dtype=torch.float64, device=device)[:, None]
    kx = torch.fft.fftfreq(cols, dtype=torch.float64, device=device)[None, :]
    r, th = torch.sqrt(ky * ky + kx * kx), torch.atan2(ky, kx)
    low = lambda w: torch.exp(-((r / w) ** 2) * math.log(2.0))  # noqa: E731
    edge = [0.5 * 2.0 ** (j - scales) for j in range(scales + 1)]
    out = [low(edge[0])]
    for j in range(scales):
        ring = torch.sqrt((low(edge[j + 1]) - low(edge[j])).clamp_min(0)) if j + 1 < scales else \
            torch.sqrt((1.0 - low(edge[j])).clamp_min(0))
        n = DIRECTIONS[j]
        for d in range(n):
            a = torch.cos(th - math.pi * d / n) ** 2     # period pi: even under k -> -k
            out.append(ring * a ** (n // 2))
    g = torch.stack(out)
    back = torch.roll(torch.flip(g, (1, 2)), (1, 1), (1, 2))
    g = 0.5 * (g + back)
    if not cplx:
        return g
    y, x = torch.arange(rows, device=device)[:, None], torch.arange(cols, device=device)[None, :]
    i = torch.arange(len(out), device=device)[:, None, None]
    ph = 2 * math.pi * (((i % 5) * y % rows).double() / rows + ((i % 3) * x % cols).double() / cols)
    return torch.polar(g, ph)


@functools.lru_cache(maxsize=1)
def _bank(rows, cols, scales, cplx):
    """The filter bank that a program builds once for its image size."""
    from paper_2006_04591_gb300.shearlet import Bank
    g = _spectra(rows, cols, scales, cplx, DEV).cpu().numpy()
    return Bank.from_complex_spectra(g) if cplx else Bank.from_spectra(g)


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) % (1 << 31))


def _cartoons(gen, batch, rows, cols, noise=30.0 / 255.0):
    """Overlapping filled ellipses of random grey levels plus Gaussian noise."""
    u = torch.rand((batch, 14, 6), generator=gen, device=DEV)
    y = torch.arange(rows, device=DEV, dtype=torch.float32)[None, :, None]
    x = torch.arange(cols, device=DEV, dtype=torch.float32)[None, None, :]
    img = torch.zeros((batch, rows, cols), device=DEV)
    n = min(rows, cols)
    for e in range(u.shape[1]):
        p = u[:, e, :, None, None]
        dy, dx = y - p[:, 0] * rows, x - p[:, 1] * cols
        c, s = torch.cos(math.pi * p[:, 4]), torch.sin(math.pi * p[:, 4])
        ry, rx = n * (1 / 16 + 3 / 16 * p[:, 2]), n * (1 / 16 + 3 / 16 * p[:, 3])
        inside = ((c * dx + s * dy) / rx) ** 2 + ((c * dy - s * dx) / ry) ** 2 <= 1
        img = torch.where(inside, p[:, 5].expand_as(img), img)
    return img + noise * torch.randn(img.shape, generator=gen, device=DEV)


def _inputs(case, seed):
    """The case's tensors, the same for ``run`` and ``exact``."""
    g, kind = _gen(seed), case["kind"]
    if kind in ("transform", "layer"):
        s = {"x": _cartoons(g, case["batch"], case["rows"], case["cols"])}
        if kind == "layer":
            s["g"] = torch.randn(s["x"].shape, generator=g, device=DEV)
        return s
    if kind in ("relaxed", "shrink", "net"):
        clean = _cartoons(g, case["batch"], case["rows"], case["cols"], 0.0)
        mask = torch.rand(clean.shape, generator=g, device=DEV) < 0.5
        s = {"fm": clean * mask, "mask": mask.to(torch.uint8)}
        if kind == "relaxed":
            # thresholds relative to the filters' RMS, and the loss's gradient
            s["delta"] = 0.05 + 0.5 * torch.rand((case["batch"], case["iterations"],
                                                  _filters(case["scales"])), generator=g, device=DEV)
            s["g"] = 1e-3 * torch.randn(clean.shape, generator=g, device=DEV)
        elif kind == "shrink":
            # the estimate of a loop that has just begun, and its high thresholds
            s["fe"] = clean * (0.6 + 0.1 * torch.rand((case["batch"], 1, 1), generator=g, device=DEV))
            s["delta"] = 3.0 + torch.rand((case["batch"], 1), generator=g, device=DEV)
        else:
            s["mask"] = mask.float()
        return s
    if kind == "conv":
        ci, co = case["ci"], case["co"]
        shape = (case["batch"], ci, case["rows"], case["cols"])
        return {"x": torch.randn(shape, generator=g, device=DEV),
                "w": torch.randn((co, ci, 3, 3), generator=g, device=DEV) * math.sqrt(2.0 / (9 * ci)),
                "b": 0.1 * torch.randn(co, generator=g, device=DEV),
                "a": torch.full((1,), 0.25, device=DEV),
                "g": torch.randn((shape[0], co) + shape[2:], generator=g, device=DEV)}
    n = case["n"]
    bins = int(math.ceil(math.sqrt(2.0) * n))
    return {"x": _cartoons(g, case["batch"], n, n, 0.0),
            "p": torch.rand((case["batch"], case["angles"], bins), generator=g, device=DEV)}


def prepare(case, seed):
    s, kind = _inputs(case, seed), case["kind"]
    s["case"] = case
    if kind in ("transform", "layer", "relaxed", "shrink"):
        s["bank"] = _bank(case["rows"], case["cols"], case["scales"], case["complex"])
    if kind in ("relaxed", "shrink"):
        s["rms"] = s["bank"].rms_device
    if kind == "shrink":
        s["th"] = s["delta"] * s["rms"]
        s["th"][:, 0] = 0.0              # the low-pass is kept
    if kind == "layer":
        from paper_2006_04591_gb300.autograd import ShearletDec, ShearletRec
        s["dec"], s["rec"] = ShearletDec(s["bank"], DTYPES[case["dtype"]]), ShearletRec(s["bank"])
        s["x"].requires_grad_(True)
    if kind == "relaxed":
        s["delta"].requires_grad_(True)
    if kind == "conv":
        for k in ("x", "w", "b", "a"):
            s[k].requires_grad_(True)
    if kind == "ray":
        from paper_2006_04591_gb300.ray import RayTransform
        s["op"] = RayTransform(case["n"], case["angles"], device=0)
    if kind == "net":
        from paper_2006_04591_gb300.nn import ThresholdNet
        s["net"] = ThresholdNet(case["filters"], T=case["iterations"], seed=7, device=DEV)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "transform":
        c = s["bank"].decompose(s["x"], dtype=DTYPES[case["dtype"]])
        return {"coeffs": c, "image": s["bank"].reconstruct(c)}
    if kind == "layer":
        c = s["dec"](s["x"])
        y = s["rec"](c)
        (gx,) = torch.autograd.grad(y, (s["x"],), s["g"])
        return {"coeffs": c.detach(), "image": y.detach(), "gx": gx}
    if kind == "relaxed":
        from paper_2006_04591_gb300.learned import unrolled_iht
        f = unrolled_iht(s["bank"], s["fm"], s["mask"], s["delta"], 0.1, s["rms"])
        (gd,) = torch.autograd.grad(f, (s["delta"],), s["g"])
        return {"image": f.detach(), "gdelta": gd}
    if kind == "shrink":
        return s["bank"].shrink(s["fm"], s["th"], mask_u8=s["mask"], f_est=s["fe"])
    if kind == "conv":
        from paper_2006_04591_gb300 import nn
        y = nn.prelu(nn.conv3x3(s["x"], s["w"], s["b"], tc=True), s["a"])
        gx, gw, gb, ga = torch.autograd.grad(y, (s["x"], s["w"], s["b"], s["a"]), s["g"])
        return {"y": y.detach(), "gx": gx, "gw": gw, "gb": gb, "ga": ga}
    if kind == "ray":
        return {"sinogram": s["op"].forward(s["x"]), "image": s["op"].adjoint(s["p"])}
    with torch.no_grad():
        return s["net"](torch.stack([s["fm"], s["mask"]], dim=1))


# --------------------------------------------------------------------- work
def work(case):
    kind = case["kind"]
    if kind in ("transform", "layer", "relaxed", "shrink"):
        B, N, M, K = case["batch"], case["rows"], case["cols"], _filters(case["scales"])
        half = N * (M // 2 + 1) * 4
        filt = K * half * (2 if case["complex"] else 1)
        s = {"f32": 4, "bf16": 2}[case.get("dtype", "f32")]
        img, coef = 4 * B * N * M, s * B * K * N * M
        fft = 2.5 * B * N * M * math.log2(N * M)                 # one real 2D transform per image
        one = {"bytes": img + coef + filt, "flops": (K + 1) * fft}   # one direction
        if kind == "transform":
            return {"bytes": 2 * one["bytes"] + half, "flops": 2 * one["flops"]}
        if kind == "layer":
            return {"bytes": 4 * one["bytes"] + 2 * half, "flops": 4 * one["flops"]}
        if kind == "shrink":
            return {"bytes": 3.25 * img + filt + half, "flops": 2 * one["flops"]}
        # forward: coefficients written, read and gated, read; backward: the gate's gradient reads
        # coefficients and their gradient and writes one, and the first iteration needs no more
        it = case["iterations"]
        return {"bytes": it * (4 * one["bytes"] + 5 * coef) - (one["bytes"] + coef),
                "flops": (4 * it - 1) * one["flops"]}
    if kind == "conv":
        B, H, W, ci, co = case["batch"], case["rows"], case["cols"], case["ci"], case["co"]
        px = 4 * B * H * W
        return {"bytes": px * (2 * ci + 2 * co) + 8 * 9 * ci * co, "flops": 3 * 2 * 9 * ci * co * B * H * W}
    if kind == "ray":
        n, A, B = case["n"], case["angles"], case["batch"]
        D = int(math.ceil(math.sqrt(2.0) * n))
        return {"bytes": 8 * B * (n * n + A * D), "flops": 2 * 4 * B * A * n * n}
    B, N, M = case["batch"], case["rows"], case["cols"]
    return {"bytes": 8 * B * N * M, "flops": 2 * 9 * 32 * (2 + 3 * 32) * B * (N // 4) * (M // 4)}


# -------------------------------------------------------------------- exact
def _fft_dec(x, G):
    return torch.fft.ifft2(G * torch.fft.fft2(x)[:, None]).real


def _fft_rec(c, G, W):
    return torch.fft.ifft2((torch.conj(G) * torch.fft.fft2(c)).sum(1) / W).real


def _ray_samples(n, A, D, a):
    """Joseph's method at angle a: pixel pairs and weights of every (bin, sample)."""
    phi, root = math.pi * a / A, math.sqrt(2.0)
    c, s, h = math.cos(phi), math.sin(phi), 2.0 / n
    by_rows = abs(c) >= abs(s)
    t = torch.arange(n, dtype=torch.float64, device=DEV)[None, :]
    d = torch.arange(D, dtype=torch.float64, device=DEV)[:, None]
    pos, off = -root + (d + 0.5) * (2 * root / D), -1.0 + (t + 0.5) * h
    along, across = (c, s) if by_rows else (s, c)
    u = (pos - off * across) / (h * along) + 1.0 / h - 0.5
    k = torch.floor(u)
    w1 = u - k
    return by_rows, k.long(), 1.0 - w1, w1, h / abs(along)


def _ray_exact(x, p, n, A):
    B, D = x.shape[0], p.shape[2]
    sino = torch.empty((B, A, D), dtype=torch.float64, device=DEV)
    back = torch.zeros((B, n * n), dtype=torch.float64, device=DEV)
    t = torch.arange(n, device=DEV)[None, :]
    flat = x.reshape(B, -1)
    for a in range(A):
        by_rows, k, w0, w1, w = _ray_samples(n, A, D, a)
        acc = torch.zeros((B, D), dtype=torch.float64, device=DEV)
        for kk, ww in ((k, w0), (k + 1, w1)):
            ok = (kk >= 0) & (kk < n)
            kc = kk.clamp(0, n - 1)
            at = (t * n + kc) if by_rows else (kc * n + t)
            ww = torch.where(ok, ww, 0.0) * w
            acc += (flat[:, at.reshape(-1)].reshape(B, D, n) * ww).sum(2)
            back.index_add_(1, at.reshape(-1), (ww * p[:, a, :, None]).reshape(B, -1))
        sino[:, a] = acc
    return {"sinogram": sino, "image": back.reshape(B, n, n)}


def exact(case, seed):
    s, kind = _inputs(case, seed), case["kind"]
    s = {k: v.double() for k, v in s.items()}
    if kind in ("transform", "layer", "relaxed", "shrink"):
        G = _spectra(case["rows"], case["cols"], case["scales"], case["complex"], DEV)
        W = (G.abs() ** 2).sum(0)
    if kind in ("transform", "layer"):
        B = case["batch"]
        c = torch.empty((B,) + tuple(G.shape), dtype=torch.float64, device=DEV)
        y = torch.empty_like(s["x"])
        for b in range(B):
            c[b:b + 1] = _fft_dec(s["x"][b:b + 1], G)
            y[b:b + 1] = _fft_rec(c[b:b + 1], G, W)
        out = {"coeffs": c, "image": y}
        if kind == "layer":
            # backward of rec o dec: the filters over W, then their adjoint sum
            out["gx"] = torch.cat([_fft_rec(_fft_dec(s["g"][b:b + 1], G / W), G, torch.ones_like(W))
                                   for b in range(B)])
        return out
    if kind == "relaxed":
        rms = torch.sqrt((G ** 2).mean((1, 2)))
        f, d = torch.zeros_like(s["fm"]), s["delta"].requires_grad_(True)
        for t in range(case["iterations"]):
            c = _fft_dec(torch.where(s["mask"] != 0, s["fm"], f), G)
            lim = (d[:, t] * rms)[:, :, None, None]
            f = _fft_rec(c * torch.sigmoid((c.abs() / lim - 1.0) / 0.1), G, W)
        (gd,) = torch.autograd.grad(f, (d,), s["g"])
        return {"image": f.detach(), "gdelta": gd}
    if kind == "shrink":
        th = (s["delta"].float() * torch.sqrt((G ** 2).mean((1, 2))).float()).double()
        th[:, 0] = 0.0
        c = _fft_dec(torch.where(s["mask"] != 0, s["fm"], s["fe"]), G)
        return _fft_rec(torch.where(c.abs() >= th[:, :, None, None], c, 0.0), G, W)
    if kind == "conv":
        x, w, b, a = (s[k].requires_grad_(True) for k in ("x", "w", "b", "a"))
        z = torch.nn.functional.conv2d(x, w, b, padding=1)
        y = torch.where(z >= 0, z, a * z)
        gx, gw, gb, ga = torch.autograd.grad(y, (x, w, b, a), s["g"])
        return {"y": y.detach(), "gx": gx, "gw": gw, "gb": gb, "ga": ga}
    if kind == "ray":
        return _ray_exact(s["x"], s["p"], case["n"], case["angles"])
    # the threshold network from the same seeded weights: four convolution blocks on the pooled
    # image and mask, global mean, linear, softplus
    gen = torch.Generator().manual_seed(7)
    h = torch.nn.functional.avg_pool2d(torch.stack([s["fm"], s["mask"]], 1), 4)
    chans = (2, 32, 32, 32, 32)
    for l in range(4):
        w = torch.randn((chans[l + 1], chans[l], 3, 3), generator=gen) * math.sqrt(2.0 / (9 * chans[l]))
        z = torch.nn.functional.conv2d(h, w.double().to(DEV), padding=1)
        h = torch.where(z >= 0, z, 0.25 * z)
    T, K = case["iterations"], case["filters"]
    wl = (torch.randn((T * K, 32), generator=gen) * 0.01).double().to(DEV)
    return torch.nn.functional.softplus(h.mean((2, 3)) @ wl.T + 1.0).reshape(-1, T, K)
