"""What is timed: the work a user of the library has it do, through its public
entry points, over the range it is used in.

A case is a dict of plain values with a "kind":
  filter    the guided filter alone (Eq. 3-5)
  color     the guided filter with a colour guidance image
  spectrum  the 2-D real DFT and its inverse
  solve     one image, `iters` iterations
  padded    one image of any size: padded to a canvas, solved, cropped
  batch     images of uneven sizes solved together, device buffers
  host      the same from page-locked host buffers, results back on the host
  grad      the differentiable solve of a batch: result and gradient

Inputs are made on the GPU from the seed alone: shaded regions with hard edges
and a fine texture, blurred circularly by a PSF, with Gaussian noise.

A solve's result is the image u, and its ISNR curve where there is a clean
image (FP64 numbers formed from an FP32 image: returned as FP32).  The lambda_k
that a solve also reports are the path's own intermediates: they carry the
condition number of Eq. 11, which reaches 1e6 on these inputs, so that two
roundings of one spectrum move them by 1e-7 to 1e-2 of their size where u stays
the same to 1e-7.  The gradient is taken with respect to the observation: the
PSF is known (the sums behind its gradient cancel to a like degree).
"""
import math
import random

import numpy as np
import torch

import paper_1609_01839_gb300 as gfd

DEV = "cuda:0"

# true sizes of an uneven batch and the canvases they are extended to
BATCH_SIZES = (((256, 256), (256, 256)), ((384, 384), (512, 512)), ((512, 512), (512, 512)),
               ((768, 1024), (1024, 1024)))


def listed():
    return [
        # one small edge-preserving smoothing: the shortest call there is
        {"name": "filter_256_w5", "kind": "filter", "M": 256, "N": 256, "w": 5, "eps": 1e-3,
         "truncated": False},
        # smoothing of a photograph-sized image (the large workload's window and eps)
        {"name": "filter_4096_w9", "kind": "filter", "M": 4096, "N": 4096, "w": 9, "eps": 1e-4,
         "truncated": False},
        # the widest window, with windows cut at the image's edge, not square
        {"name": "filter_cut_1024x2048_w17", "kind": "filter", "M": 1024, "N": 2048, "w": 17,
         "eps": 1e-3, "truncated": True},
        # a photograph smoothed under its own colours
        {"name": "color_1024_w9", "kind": "color", "M": 1024, "N": 1024, "w": 9, "eps": 1e-3,
         "truncated": False},
        # the library's transforms for a user's own spectral work
        {"name": "spectrum_2048x1024", "kind": "spectrum", "M": 2048, "N": 1024},
        # the plain method on one small image: launches and latency
        {"name": "solve_256_10it", "kind": "solve", "M": 256, "N": 256, "psf": "uniform9",
         "psf_sigma": 0.0, "bsnr": 40.0, "w": 5, "eps": 1e-3, "iters": 10, "clean": False},
        # the plain method on an ordinary image, with its ISNR curve
        {"name": "solve_512_20it", "kind": "solve", "M": 512, "N": 512, "psf": "invquad15",
         "psf_sigma": 0.0, "bsnr": 30.0, "w": 7, "eps": 1e-3, "iters": 20, "clean": True},
        # an observation whose size is no power of two
        {"name": "padded_601x907_15it", "kind": "padded", "m": 601, "n": 907, "psf": "invquad15",
         "psf_sigma": 0.0, "bsnr": 35.0, "w": 9, "eps": 1e-3, "iters": 15},
        # the batched workload: 256 images of uneven sizes, PSFs, noise and windows
        {"name": "batch_256_15it", "kind": "batch", "images": 256, "mix": "uneven", "iters": 15},
        # a quarter of it as a service gets it: host buffers in, host buffers out
        {"name": "host_64_15it", "kind": "host", "images": 64, "mix": "uneven", "iters": 15},
        # the large-image workload: 4 images of 4096 x 4096, motion blur
        {"name": "large_4x4096_30it", "kind": "batch", "images": 4, "mix": "large", "iters": 30},
        # the differentiation workload: a training step's forward and backward
        {"name": "grad_16x512_10it", "kind": "grad", "images": 16, "M": 512, "N": 512,
         "psf": "gauss25", "psf_sigma": 1.6, "bsnr": 25.0, "w": 7, "eps": 1e-3, "iters": 10},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _pow2(rng, lo, hi):
    return 1 << rng.randint(lo.bit_length() - 1, hi.bit_length() - 1)


def _psf_choice(rng):
    kind = rng.choice(("uniform9", "gauss25", "invquad15", "motion31"))
    return kind, round(rng.uniform(1.0, 2.0), 2) if kind == "gauss25" else 0.0


def draw(rng):
    kind = rng.choice(("filter", "color", "spectrum", "solve", "solve", "padded", "batch", "host",
                       "grad"))
    w = rng.choice((3, 5, 7, 9, 11, 17))
    eps = round(10.0 ** rng.uniform(-4.0, -2.0), 6)
    cut = rng.random() < 0.3
    if kind == "filter":
        return {"kind": kind, "M": _pow2(rng, 64, 4096), "N": _pow2(rng, 64, 4096), "w": w,
                "eps": eps, "truncated": cut}
    if kind == "color":
        return {"kind": kind, "M": _pow2(rng, 64, 2048), "N": _pow2(rng, 64, 1024), "w": w,
                "eps": eps, "truncated": cut}
    if kind == "spectrum":
        return {"kind": kind, "M": _pow2(rng, 64, 4096), "N": _pow2(rng, 64, 4096)}
    psf, psf_sigma = _psf_choice(rng)
    bsnr = round(rng.uniform(30.0, 40.0), 1)
    iters = _log_int(rng, 5, 30)
    w = rng.choice((3, 5, 7, 9))
    case = {"kind": kind, "psf": psf, "psf_sigma": psf_sigma, "bsnr": bsnr, "w": w, "eps": eps,
            "iters": iters}
    if kind == "solve":
        case.update(M=_pow2(rng, 64, 2048), N=_pow2(rng, 64, 2048), clean=rng.random() < 0.3)
    elif kind == "padded":
        case.update(m=_log_int(rng, 70, 2000), n=_log_int(rng, 70, 2000))
        if psf in ("gauss25", "motion31"):  # a padded model with zeros in |H|: u itself is loose
            case.update(psf="invquad15", psf_sigma=0.0)
    elif kind == "grad":
        size = _pow2(rng, 64, 512)
        case.update(images=_log_int(rng, 1, 16), M=size, N=size, iters=_log_int(rng, 2, 10),
                    psf="gauss25", psf_sigma=1.6, bsnr=25.0)
    else:
        case = {"kind": kind, "images": _log_int(rng, 2, 200 if kind == "batch" else 60),
                "mix": "uneven", "iters": min(iters, 20)}
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _psf(kind, sigma):
    """The workloads' point-spread functions (float64, odd-sized, sum 1)."""
    if kind == "uniform9":
        return np.full((9, 9), 1.0 / 81.0)
    if kind == "gauss25":
        i = np.arange(-12, 13)
        h = np.exp(-(i[:, None] ** 2 + i[None, :] ** 2) / (2.0 * sigma * sigma))
    elif kind == "invquad15":
        i = np.arange(-7, 8)
        h = 1.0 / (1.0 + i[:, None] ** 2 + i[None, :] ** 2)
    else:  # motion31: a 21-pixel segment at 30 degrees, splatted bilinearly
        t = (np.arange(2100) + 0.5) / 100.0 - 10.5
        col, row = 15.0 + t * math.cos(math.pi / 6), 15.0 - t * math.sin(math.pi / 6)
        r0, c0 = np.floor(row).astype(int), np.floor(col).astype(int)
        h = np.zeros((31, 31))
        for dr in (0, 1):
            for dc in (0, 1):
                wt = np.abs(1 - dr - (row - r0)) * np.abs(1 - dc - (col - c0))
                np.add.at(h, (r0 + dr, c0 + dc), wt)
    return h / h.sum()


def _embed(h, M, N):
    """A centred PSF on the canvas, offsets taken modulo its size."""
    kh, kw = h.shape
    i = (torch.arange(kh, device=h.device) - kh // 2) % M
    j = (torch.arange(kw, device=h.device) - kw // 2) % N
    flat = (i[:, None] * N + j[None, :]).reshape(-1)
    c = torch.zeros(M * N, dtype=h.dtype, device=h.device)
    return c.index_add(0, flat, h.reshape(-1)).view(M, N)


def _picture(m, n, rnd, gen, channels=None):
    """Shaded regions with hard edges over a shaded background, a fine texture."""
    y, x = torch.meshgrid(torch.linspace(-1, 1, m, device=DEV), torch.linspace(-1, 1, n, device=DEV),
                          indexing="ij")
    C = channels or 1

    def shade():
        return [rnd.uniform(0.1, 0.9) + rnd.uniform(-0.2, 0.2) * x + rnd.uniform(-0.2, 0.2) * y +
                rnd.uniform(-0.2, 0.2) * x * y for _ in range(C)]
    u = torch.stack(shade())
    for _ in range(20):
        cx, cy, th = rnd.uniform(-1, 1), rnd.uniform(-1, 1), rnd.uniform(0, math.pi)
        a, b = rnd.uniform(0.05, 0.5), rnd.uniform(0.05, 0.5)
        p = (x - cx) * math.cos(th) + (y - cy) * math.sin(th)
        q = (y - cy) * math.cos(th) - (x - cx) * math.sin(th)
        if rnd.random() < 0.5:
            inside = (p.abs() < a) & (q.abs() < b)
        else:
            inside = (p / a) ** 2 + (q / b) ** 2 < 1
        u = torch.where(inside, torch.stack(shade()), u)
    t = torch.randn(m, n, generator=gen, device=DEV)
    t = t + torch.roll(t, 1, 0) + torch.roll(t, 1, 1) + torch.roll(t, (1, 1), (0, 1))
    u = (u + 0.01 * t).clamp_(0.0, 1.0)
    return u if channels else u[0].contiguous()


def _extend(u, M, N):
    """Symmetric extension at the bottom and right edges."""
    m, n = u.shape
    i = torch.arange(M, device=u.device) % (2 * m)
    j = torch.arange(N, device=u.device) % (2 * n)
    i, j = torch.where(i < m, i, 2 * m - 1 - i), torch.where(j < n, j, 2 * n - 1 - j)
    return u[i][:, j].contiguous()


def _observe(u, psf, psf_sigma, bsnr, gen):
    """y = h * u + noise on u's canvas; (y, h, sigma)."""
    M, N = u.shape
    h = torch.from_numpy(_psf(psf, psf_sigma)).to(DEV).float()
    y = torch.fft.irfft2(torch.fft.rfft2(u) * torch.fft.rfft2(_embed(h, M, N)), s=(M, N))
    sigma = float(y.std()) / 10.0 ** (bsnr / 20.0)
    return y + sigma * torch.randn(M, N, generator=gen, device=DEV), h, sigma


def _images(case, rnd, gen):
    """The problems of a batch: dicts of y, h, sigma, w, eps.  The batch's
    make-up (sizes, PSFs, windows) goes with the number of images; the scenes
    and the noise go with the seed."""
    out, mix = [], random.Random(case["images"])
    for _ in range(case["images"]):
        if case["mix"] == "large":
            (m, n), (M, N) = (4096, 4096), (4096, 4096)
            psf, ps, bsnr, w, eps = "motion31", 0.0, 35.0, 9, 1e-4
        else:
            (m, n), (M, N) = mix.choice(BATCH_SIZES)
            psf, ps = mix.choice(("uniform9", "gauss25", "invquad15")), mix.uniform(1.0, 2.0)
            bsnr, w, eps = mix.uniform(30.0, 40.0), mix.choice((5, 7, 9)), 1e-3
        u = _extend(_picture(m, n, rnd, gen), M, N)
        y, h, sigma = _observe(u, psf, ps, bsnr, gen)
        out.append({"y": y, "h": h, "sigma": sigma, "w": w, "eps": eps})
    return out


def _inputs(case, seed):
    """Everything the call is given, from the seed alone."""
    rnd = random.Random(seed)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    kind = case["kind"]
    if kind == "filter":
        # the method's own use: a smooth guidance and a noisier input of one scene
        I = _picture(case["M"], case["N"], rnd, gen)
        p = I + 0.03 * torch.randn(I.shape, generator=gen, device=DEV)
        return {"I": I, "p": p}
    if kind == "color":
        I = _picture(case["M"], case["N"], rnd, gen, 3)
        p = I.mean(0) + 0.03 * torch.randn(I.shape[1:], generator=gen, device=DEV)
        return {"I": I.contiguous(), "p": p.contiguous()}
    if kind == "spectrum":
        return {"x": _picture(case["M"], case["N"], rnd, gen)}
    if kind in ("solve", "padded"):
        m, n = (case["M"], case["N"]) if kind == "solve" else (case["m"], case["n"])
        u = _picture(m, n, rnd, gen)
        y, h, sigma = _observe(u, case["psf"], case["psf_sigma"], case["bsnr"], gen)
        return {"u": u, "y": y, "h": h, "sigma": sigma}
    if kind == "grad":
        us = torch.stack([_picture(case["M"], case["N"], rnd, gen) for _ in range(case["images"])])
        obs = [_observe(u, case["psf"], case["psf_sigma"], case["bsnr"], gen) for u in us]
        return {"u": us, "y": torch.stack([o[0] for o in obs]), "h": obs[0][1],
                "sigma": [o[2] for o in obs]}
    return {"items": _images(case, rnd, gen)}


def _on_host(t):
    return t.cpu().pin_memory()


def prepare(case, seed):
    s = {"case": case, "in": _inputs(case, seed)}
    cut = gfd.BOUNDARY_TRUNCATED if case.get("truncated") else gfd.BOUNDARY_PERIODIC
    s["ctx"] = gfd.Context(0, boundary=cut)
    i = s["in"]
    if case["kind"] == "grad":
        i["y"].requires_grad_()
        i["eps"] = torch.tensor(case["eps"], dtype=torch.float64)
    elif case["kind"] in ("batch", "host"):
        # the buffers and descriptors that a program keeps for its batch: the
        # results side by side in one buffer
        items, iters = i["items"], case["iters"]
        host = case["kind"] == "host"
        flat = torch.empty(sum(it["y"].numel() for it in items), dtype=torch.float32,
                           device="cpu" if host else DEV, pin_memory=host)
        at = 0
        for it in items:
            if host:
                it["y"], it["h"] = _on_host(it["y"]), _on_host(it["h"])
            n = it["y"].numel()
            it["u"] = flat[at:at + n].view(it["y"].shape)
            at += n
        make = s["ctx"].make_host_images if host else s["ctx"].make_images
        s["images"], s["flat"] = make(items, iters), flat
    return s


def run(s):
    case, i, ctx = s["case"], s["in"], s["ctx"]
    kind = case["kind"]
    if kind == "filter":
        return ctx.guidfilter(i["I"], i["p"], case["w"], case["eps"])
    if kind == "color":
        return ctx.guidfilter_color(i["I"], i["p"], case["w"], case["eps"])
    if kind == "spectrum":
        X = ctx.fft2_r2c(i["x"])
        return {"X": X, "x": ctx.fft2_c2r(X)}
    if kind == "solve":
        u, _, isnr = ctx.solve(i["y"], i["h"], i["sigma"], case["w"], case["eps"], case["iters"],
                                 u_orig=i["u"] if case["clean"] else None)
        return {"u": u, "isnr": None if isnr is None else isnr.float()}
    if kind == "padded":
        u, _ = ctx.solve_padded(i["y"], i["h"], i["sigma"], case["w"], case["eps"], case["iters"])
        return u
    if kind == "grad":
        u = ctx.deconv(i["y"], i["h"], i["eps"], i["sigma"], case["w"], case["iters"])
        loss = ((u - i["u"]) ** 2).mean()
        return {"u": u.detach(), "g_y": torch.autograd.grad(loss, i["y"])[0]}
    if kind == "batch":
        ctx.solve_batched_images(s["images"], case["iters"])
    else:
        ctx.solve_batched_host_images(s["images"], case["iters"])
    return s["flat"]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _pixels(case):
    kind = case["kind"]
    if kind == "padded":
        return (1 << (case["m"] - 1).bit_length()) * (1 << (case["n"] - 1).bit_length())
    if kind in ("batch", "host"):
        if case["mix"] == "large":
            return case["images"] * 4096 * 4096
        return case["images"] * sum(M * N for _, (M, N) in BATCH_SIZES) / len(BATCH_SIZES)
    return case["M"] * case["N"] * case.get("images", 1)


def work(case):
    """Bytes: each input read once and each result written once.  Operations:
    real DFTs (2.5 P log2 P each; three an iteration, two at the start, five
    more an iteration backward), about 60 a pixel for the spectral solves and
    the equation for lambda, 40 for the filter."""
    P, kind = _pixels(case), case["kind"]
    if kind == "filter":
        return {"bytes": 12.0 * P, "flops": 40.0 * P}
    if kind == "color":
        return {"bytes": 20.0 * P, "flops": 150.0 * P}
    n_img = case.get("images", 1)
    fft = 2.5 * math.log2(P / n_img) * P
    if kind == "spectrum":
        return {"bytes": 16.0 * P, "flops": 2.0 * fft}
    it = case["iters"]
    flops = 2.0 * fft + it * (3.0 * fft + 100.0 * P)
    if kind == "grad":
        return {"bytes": 16.0 * P, "flops": flops + it * (8.0 * fft + 300.0 * P)}
    return {"bytes": 8.0 * P, "flops": flops}


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------

def _box(x, w, cut):
    """Window means over the last two axes: periodic, or cut at the edges."""
    r = w // 2
    for dim in (-1, -2):
        L = x.shape[dim]
        if cut:
            c = torch.nn.functional.pad(x, (r, r) if dim == -1 else (0, 0, r, r))
            n = torch.arange(L, device=x.device)
            n = ((n + r).clamp(max=L - 1) - (n - r).clamp(min=0) + 1).to(x.dtype)
            n = n if dim == -1 else n[:, None]
        else:
            c, n = torch.cat([x.narrow(dim, L - r, r), x, x.narrow(dim, 0, r)], dim) if r else x, w
        s = c.narrow(dim, 0, L).clone()
        for k in range(1, w):
            s = s + c.narrow(dim, k, L)
        x = s / n
    return x


def _guided(I, p, w, eps, cut=False):
    mu, pb = _box(I, w, cut), _box(p, w, cut)
    a = (_box(I * p, w, cut) - mu * pb) / (_box(I * I, w, cut) - mu * mu + eps)
    return _box(a, w, cut) * I + _box(pb - a * mu, w, cut)


def _guided_color(I, p, w, eps, cut):
    mu, pb = _box(I, w, cut), _box(p, w, cut)
    cov = torch.stack([_box(I[c] * p, w, cut) - mu[c] * pb for c in range(3)], -1)
    S = torch.stack([torch.stack([_box(I[c] * I[d], w, cut) - mu[c] * mu[d] for d in range(3)], -1)
                     for c in range(3)], -2)
    S = S + eps * torch.eye(3, dtype=I.dtype, device=I.device)
    # Cramer's rule
    x = [torch.linalg.cross(S[..., (k + 1) % 3], S[..., (k + 2) % 3]) for k in range(3)]
    det = (S[..., 0] * x[0]).sum(-1)
    a = torch.stack([(x[k] * cov).sum(-1) / det for k in range(3)])
    return (_box(a, w, cut) * I).sum(0) + _box(pb - (a * mu).sum(0), w, cut)


def _lambda(a, r, T, wt):
    """The root of sum(wt r (l / (a + l))^2) = T per image (inf where the sum
    of wt r is within T): Newton in log l, kept in a bracket."""
    dims = (-2, -1)
    inf = (wt * r).sum(dims) <= T
    lo, hi = torch.full_like(T, math.log(1e-14)), torch.full_like(T, math.log(1e12))
    x = torch.full_like(T, math.log(1e-3))
    for _ in range(100):
        t = 1.0 / (1.0 + a * torch.exp(-x)[..., None, None])
        q = wt * r * t * t
        f, df = q.sum(dims), (2.0 * q * (1.0 - t)).sum(dims)
        lo, hi = torch.where(f < T, x, lo), torch.where(f < T, hi, x)
        # Newton on log f, which is nearly straight
        nx = x - torch.log(f / T) * f / df
        nx = torch.where((nx > lo) & (nx < hi), nx, 0.5 * (lo + hi))
        if float(torch.where(inf, torch.zeros_like(x), (nx - x).abs()).max()) < 1e-14:
            x = nx
            break
        x = nx
    return torch.where(inf, torch.full_like(T, math.inf), torch.exp(x))


def _solve(y, h, sigma, w, eps, iters, clean=None):
    """The method on images of one size, y (B, M, N), h (B, kh, kw), sigma (B),
    in the inputs' precision; (u, ISNR (B, iters) or None).  lambda carries its
    derivative through Eq. 11 where the inputs ask for one."""
    B, M, N = y.shape
    P = M * N
    grad = torch.is_grad_enabled() and y.requires_grad
    H = torch.fft.rfft2(torch.stack([_embed(k, M, N) for k in h]))
    Y = torch.fft.rfft2(y)
    k = torch.arange(M, device=y.device, dtype=y.dtype)[:, None]
    l = torch.arange(N // 2 + 1, device=y.device, dtype=y.dtype)[None, :]
    D2 = 4.0 * torch.sin(math.pi * k / M) ** 2 + 4.0 * torch.sin(math.pi * l / N) ** 2
    wt = torch.full((1, N // 2 + 1), 2.0 / P, device=y.device, dtype=y.dtype)
    wt[0, 0] = wt[0, -1] = 1.0 / P
    num = ((y - y.mean((-2, -1), keepdim=True)) ** 2).sum((-2, -1)) - P * sigma ** 2
    den = h.abs().sum((-2, -1)) ** 2 * (y * y).sum((-2, -1))
    T = torch.clamp(torch.sqrt(1.0 - num / den), max=1.0) * P * sigma ** 2
    a, HY = H.real ** 2 + H.imag ** 2, H.conj() * Y
    u, isnrs = torch.zeros_like(y), []
    for _ in range(iters):
        U = torch.fft.rfft2(u)
        e = H * U - Y
        r = e.real ** 2 + e.imag ** 2
        with torch.no_grad():
            lam = _lambda(a, r, T, wt)
        inside = torch.isinf(lam)
        if grad:
            t = 1.0 / (1.0 + a.detach() / lam[:, None, None])
            q = (2.0 * wt * r.detach() * t * t * (1.0 - t)).sum((-2, -1)) / lam  # df/dlambda
            f = (wt * r / (1.0 + a / lam[:, None, None]) ** 2).sum((-2, -1)) - T
            lam = torch.where(inside, lam, lam - (f - f.detach()) / q)
        L = torch.where(inside, torch.ones_like(lam), lam)[:, None, None]
        inside = inside[:, None, None]
        I = torch.fft.irfft2(torch.where(inside, U, (HY + L * D2 * U) / (a + L * D2)), s=(M, N))
        p = torch.fft.irfft2(torch.where(inside, U, (HY + L * U) / (a + L)), s=(M, N))
        u = _guided(I, p, w, eps)
        if clean is not None:
            isnrs.append(10.0 * torch.log10(((y - clean) ** 2).sum((-2, -1)) /
                                            ((u - clean) ** 2).sum((-2, -1))))
    return u, torch.stack(isnrs, -1) if isnrs else None


def exact(case, seed):
    i, kind = _inputs(case, seed), case["kind"]
    cut = bool(case.get("truncated"))
    if kind == "filter":
        return _guided(i["I"].double(), i["p"].double(), case["w"], case["eps"], cut)
    if kind == "color":
        return _guided_color(i["I"].double(), i["p"].double(), case["w"], case["eps"], cut)
    if kind == "spectrum":
        x = i["x"].double()
        F = torch.fft.rfft2(x)
        X = F[:, :-1].clone()
        X[:, 0] = F[:, 0] + 1j * F[:, -1]
        return {"X": X, "x": x}
    if kind in ("solve", "padded"):
        y = i["y"]
        m, n = y.shape
        M, N = 1 << max(3, (m - 1).bit_length()), 1 << max(3, (n - 1).bit_length())
        clean = i["u"].double()[None] if case.get("clean") else None
        sig = torch.tensor([i["sigma"]], dtype=torch.float64, device=DEV)
        u, isnr = _solve(_extend(y, M, N).double()[None], i["h"].double()[None], sig,
                              case["w"], case["eps"], case["iters"], clean)
        if kind == "padded":
            return u[0, :m, :n].contiguous()
        return {"u": u[0], "isnr": None if isnr is None else isnr[0]}
    if kind == "grad":
        us, gys = [], []
        for b in range(case["images"]):
            y = i["y"][b:b + 1].double().requires_grad_()
            sig = torch.tensor([i["sigma"][b]], dtype=torch.float64, device=DEV)
            u, _ = _solve(y, i["h"].double()[None], sig, case["w"], case["eps"], case["iters"])
            loss = ((u - i["u"][b:b + 1].double()) ** 2).mean() / case["images"]
            gys.append(torch.autograd.grad(loss, y)[0][0])
            us.append(u.detach()[0])
        return {"u": torch.stack(us), "g_y": torch.stack(gys)}
    # images of one size and window together, a few at a time
    items, groups = i["items"], {}
    for k, it in enumerate(items):
        groups.setdefault((tuple(it["y"].shape), tuple(it["h"].shape), it["w"]), []).append(k)
    us = [None] * len(items)
    for (shape, _, w), members in groups.items():
        step = max(1, (1 << 24) // (shape[0] * shape[1]))
        for c in range(0, len(members), step):
            ks = members[c:c + step]
            sig = torch.tensor([items[k]["sigma"] for k in ks], dtype=torch.float64, device=DEV)
            u, _ = _solve(torch.stack([items[k]["y"] for k in ks]).double(),
                          torch.stack([items[k]["h"] for k in ks]).double(), sig, w,
                          items[ks[0]]["eps"], case["iters"])
            for q, k in enumerate(ks):
                us[k] = u[q].reshape(-1)
    return torch.cat(us)
