"""The work that users of this framework have it do, as cases that can be timed.

A case goes through the public calls of paper_1101_2254_gb300.gf (and .learned): evaluating
stamps (steps 1-3 of the loop), fitting them one by one and in batches, the Jacobian, the
learned start with its training step, and the cubes.  Inputs are drawn and rendered here with
plain torch in 64 bits, from the seed alone.

Images, sigma maps and PSFs are float32 and every pixel sum is formed in float32, so the
numbers that the library hands over in float64 storage (chi^2, parameters, the normal
equations) come back from run() in float32, the type that they were computed in.
"""
import math

import numpy as np
import torch

from paper_1101_2254_gb300 import gf, learned

F64 = torch.float64
READ, GAIN, SKY = 0.01, 1.0, 0.05


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # one evaluation of a small stamp, as a program with its own optimiser calls it
        # thousands of times: launches and latency
        dict(name="eval-64", kind="eval", H=64, W=64, P=25, disk=False, os=5, box=8, method="auto"),
        # the same for a large bulge + disk stamp with a wide PSF (Fourier-space convolution)
        dict(name="eval-512", kind="eval", H=512, W=512, P=65, disk=True, os=10, box=20, method="auto"),
        # full-size images with very wide PSFs through the tensor-core DFT
        dict(name="eval-1024-dft", kind="evals", count=16, lo=1024, hi=1024, P=255, disk=True, os=10, box=20, method="dft"),
        # a catalogue's cut-outs, sizes uneven: evaluated at given parameters, models kept
        dict(name="evals-ragged", kind="evals", count=400, lo=32, hi=256, P=33, disk=False, os=5, box=8, method="auto"),
        # one fit while a user waits: 8 free parameters
        dict(name="fit-64", kind="fit", H=64, W=64, P=25, disk=False, os=5, box=8, method="auto", tol=1e-6),
        # one large fit: bulge + disk, 15 free parameters
        dict(name="fit-512", kind="fit", H=512, W=512, P=65, disk=True, os=10, box=20, method="auto", tol=1e-6),
        # survey stamps of one size, fitted together from perturbed starts
        dict(name="fits-64", kind="fits", count=8192, lo=64, hi=64, P=33, disk=False, os=5, box=8, method="fft", tol=1e-6),
        # uneven cut-outs fitted together
        dict(name="fits-ragged", kind="fits", count=512, lo=48, hi=256, P=33, disk=False, os=5, box=8, method="auto", tol=1e-6),
        # normal equations and analytic columns at one point, for error bars; odd sizes
        dict(name="jacobian-odd", kind="jac", H=203, W=167, P=49, disk=True, os=7, box=15, method="auto"),
        # starting points of a batch: network, default guess, the better of the two
        dict(name="starts", kind="starts", count=8192),
        # one training step's loss and gradients
        dict(name="train-grad", kind="grad", count=512),
        # an integral-field cube, each spaxel's spectrum fitted
        dict(name="cube-64", kind="cube", count=4096, n_chan=2048, lines=3, cont=2, lsf=25),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["eval", "evals", "fit", "fits", "jac", "starts", "grad", "cube"])
    if kind == "starts":
        return dict(kind=kind, count=log(16, 8192))
    if kind == "grad":
        return dict(kind=kind, count=log(16, 512))
    if kind == "cube":
        n = log(200, 3000)
        return dict(kind=kind, count=min(log(32, 4096), 8_000_000 // n), n_chan=n, lines=rng.randint(1, 3), cont=rng.randint(1, 3), lsf=2 * rng.randint(1, 25) + 1)
    disk = rng.random() < 0.4 and kind != "fits"
    c = dict(kind=kind, disk=disk, os=rng.choice([1, 3, 5, 8]), method="auto")
    if kind in ("eval", "fit", "jac"):
        least = 192 if disk else 32 if kind == "eval" else 64
        c["H"] = log(least, 400)
        c["W"] = max(least, min(512, int(c["H"] * rng.uniform(0.7, 1.3))))
        c["P"] = 2 * rng.randint(4, 32) + 1
    else:
        c["lo"] = log(32 if kind == "evals" else 64, 128)
        c["hi"] = c["lo"] if rng.random() < 0.5 else min(256, c["lo"] + rng.randint(8, 120))
        c["P"] = 2 * rng.randint(4, 20) + 1
        c["count"] = min(log(16, 2000), max(16, 4_000_000 // (c["lo"] * c["hi"])))
        if c["lo"] == c["hi"]:
            c["method"] = rng.choice(["auto", "fft"])
    if kind in ("fit", "fits"):
        c["tol"] = 1e-6
    c["box"] = rng.randint(4, 12) if c["os"] > 1 else 0
    return c


# -------------------------------------------------- the method in plain 64 bits
def bn_of(n):
    """b_n of P(2n, b) = 1/2, by bisection."""
    n = n.detach().to("cpu", F64)
    lo, hi = torch.zeros_like(n), 2.0 * n + 10.0
    for _ in range(70):
        mid = 0.5 * (lo + hi)
        below = torch.special.gammainc(2.0 * n, mid) < 0.5
        lo, hi = torch.where(below, mid, lo), torch.where(below, hi, mid)
    return 0.5 * (lo + hi)


def profile(p, x, y, sersic, b=None):
    """One component at points x, y; p: slots in the last place, broadcast over the points."""
    s = (...,) + (None,) * (x.dim())
    q, pa, c = (p[..., 5][s], p[..., 6][s], p[..., 7][s]) if sersic else (p[..., 4][s], p[..., 5][s], p[..., 6][s])
    t = pa * (math.pi / 180.0)
    dx, dy = x - p[..., 0][s], y - p[..., 1][s]
    xr, yr = dx * torch.cos(t) + dy * torch.sin(t), (dy * torch.cos(t) - dx * torch.sin(t)) / q
    C = c + 2.0
    r = (xr.abs() ** C + yr.abs() ** C) ** (1.0 / C) if bool((c != 0).any()) else torch.sqrt(xr * xr + yr * yr)
    r = r / p[..., 3][s]
    if not sersic:
        return p[..., 2][s] * torch.exp(-r)
    b = bn_of(p[..., 4]).to(p.device) if b is None else b
    return p[..., 2][s] * torch.exp(-b[s] * (r ** (1.0 / p[..., 4][s]) - 1.0))


def light(p, x, y, disk, b=None):
    v = profile(p[..., 0:8], x, y, True, b)
    return v + profile(p[..., 8:15], x, y, False) if disk else v


def render(p, psf, H, W, disk, os, box, b=None):
    """Convolved models [..., H, W] of parameters [..., slots] and PSFs [..., P, P], 64 bits."""
    P = psf.shape[-1]
    c = (P - 1) // 2
    y, x = (torch.arange(n, dtype=F64, device=p.device) - c for n in (H + 2 * c, W + 2 * c))
    yy, xx = torch.meshgrid(y, x, indexing="ij")
    grid = light(p, xx, yy, disk, b)
    if os > 1 and box > 0:
        i0, j0 = (H - box) // 2, (W - box) // 2
        off = (torch.arange(os, dtype=F64, device=p.device) + 0.5) / os - 0.5
        ys = (torch.arange(i0, i0 + box, dtype=F64, device=p.device)[:, None] + off).reshape(-1)
        xs = (torch.arange(j0, j0 + box, dtype=F64, device=p.device)[:, None] + off).reshape(-1)
        yy, xx = torch.meshgrid(ys, xs, indexing="ij")
        fine = light(p, xx, yy, disk, b)
        fine = fine.reshape(fine.shape[:-2] + (box, os, box, os)).mean((-3, -1))
        grid[..., i0 + c:i0 + c + box, j0 + c:j0 + c + box] = fine
    grid = grid + p[..., -1][..., None, None]
    s = grid.shape[-2:]
    out = torch.fft.irfft2(torch.fft.rfft2(grid) * torch.fft.rfft2(psf.to(F64), s=s), s=s)
    return out[..., 2 * c:2 * c + H, 2 * c:2 * c + W]


def spectra(p, lsf, n, cont):
    """Convolved spectra [count, n] of parameters [count, slots], 64 bits."""
    c = (lsf.numel() - 1) // 2
    x = torch.arange(-c, n + c, dtype=F64, device=p.device)
    t = (x - 0.5 * (n - 1)) / (0.5 * (n - 1))
    e = sum(p[:, j:j + 1] * t ** j for j in range(cont)) + torch.zeros_like(p[:, :1])
    for k in range(cont, p.shape[1], 3):
        e = e + p[:, k:k + 1] * torch.exp(-0.5 * ((x - p[:, k + 1:k + 2]) / p[:, k + 2:k + 3]) ** 2)
    m = len(x)
    return torch.fft.irfft(torch.fft.rfft(e) * torch.fft.rfft(lsf.to(F64), n=m), n=m)[:, 2 * c:2 * c + n]


def chi2_of(m, img, sig):
    return (((img.to(F64) - m) / sig.to(F64)) ** 2).sum((-2, -1) if m.dim() > 2 or img.dim() == 2 else -1)


def least(f, p, free, img, sig, steps=12):
    """The chi^2 at the minimum near p [count, slots] of models f(p): damped Gauss-Newton in 64 bits."""
    w = 1.0 / sig.to(F64)
    img = img.to(F64)
    flat = lambda m: ((img - m) * w).reshape(p.shape[0], -1)  # noqa: E731
    best = (flat(f(p)) ** 2).sum(-1)
    lam = torch.full_like(best, 1e-4)
    for _ in range(steps):
        J = []
        for i in free:
            h = torch.zeros_like(p)
            h[:, i] = 1e-6 * p[:, i].abs().clamp(min=1.0)
            J.append((flat(f(p - h)) - flat(f(p + h))) / (2.0 * h[:, i:i + 1]))
        J = torch.stack(J, -1)
        A, g = J.mT @ J, (J.mT @ flat(f(p))[..., None])
        d = torch.linalg.solve(A + lam[:, None, None] * torch.diag_embed(torch.diagonal(A, dim1=-2, dim2=-1)), g)[..., 0]
        q = p.clone()
        q[:, free] += d
        new = (flat(f(q)) ** 2).sum(-1)
        ok = (new < best) & torch.isfinite(new)
        p = torch.where(ok[:, None], q, p)
        best = torch.where(ok, new, best)
        lam = torch.where(ok, lam * 0.1, lam * 10.0)
    return best


# --------------------------------------------------------------------- inputs
def sersic_draw(rng, H, W, bright):
    """A galaxy as in the survey-like configuration: n ~ U[0.5, 6], r_e log-uniform, q ~ U[0.2, 1], flux over
    three decades.  bright: a resolved, bright one, whose fit ends at a well-determined minimum."""
    side = min(H, W)
    n, q = (rng.uniform(0.8, 1.7), rng.uniform(0.5, 0.75)) if bright else (rng.uniform(0.5, 6.0), rng.uniform(0.2, 1.0))
    a, b = (6.0, max(8.0, min(30.0, 0.12 * side))) if bright else (2.0, min(40.0, 0.2 * side))
    re = math.exp(rng.uniform(math.log(a), math.log(b)))
    flux = math.exp(rng.uniform(math.log(1e5 if bright else 1e2), math.log(1e6 if bright else 1e5)))
    return [0.5 * (W - 1) + rng.uniform(-1, 1), 0.5 * (H - 1) + rng.uniform(-1, 1), flux, re, n, q, rng.uniform(15.0, 165.0), 0.0]


def bulge_disk_draw(rng, H, W, bright):
    s, f = min(H, W) / 512.0, 40.0 if bright else 1.0
    cx, cy = 0.5 * W + rng.uniform(-2, 2), 0.5 * H + rng.uniform(-2, 2)
    re, rs = rng.uniform(5.0, 14.0) * max(s, 0.4), rng.uniform(30.0, 60.0) * max(s, 0.4)
    return [cx, cy, f, re, rng.uniform(1.5, 2.5) if bright else rng.uniform(2.0, 6.0), rng.uniform(0.4, 0.7), rng.uniform(15.0, 165.0), 0.0,
            cx, cy, f * rng.uniform(0.5, 3.0), rs, rng.uniform(0.3, 0.8), rng.uniform(15.0, 165.0), 0.0]


def unit_flux_ie(p):
    """Total flux in slot 2 to the intensity at r_e."""
    n, b = p[:, 4], bn_of(torch.as_tensor(p[:, 4])).numpy()
    lg = np.array([math.lgamma(2.0 * v) for v in n])
    p[:, 2] /= 2.0 * math.pi * p[:, 5] * p[:, 3] ** 2 * n * np.exp(b + lg - 2.0 * n * np.log(b))
    return p


def moffat(fwhm, P):
    """Moffat PSFs (beta 3) of sum 1, [count, P, P] float32."""
    f = torch.as_tensor(np.atleast_1d(fwhm), dtype=F64, device="cuda")[:, None, None]
    v = torch.arange(P, dtype=F64, device="cuda") - (P - 1) // 2
    a = f / (2.0 * math.sqrt(2.0 ** (1.0 / 3.0) - 1.0))
    m = (1.0 + (v[:, None] ** 2 + v ** 2) / a ** 2) ** -3.0
    return (m / m.sum((1, 2), keepdim=True)).to(torch.float32)


def noisy(m, gen):
    sig = torch.sqrt(READ ** 2 + m.clamp(min=0.0) / GAIN)
    return (m + sig * torch.randn(m.shape, dtype=F64, device=m.device, generator=gen)).to(torch.float32), sig.to(torch.float32)


def start_of(p, rng, disk):
    """Each free slot off by up to a tenth, positions by a tenth of the radius."""
    u = rng.uniform(-1.0, 1.0, p.shape)
    s = p * (1.0 + 0.1 * u)
    for o, r in ((0, 3), (8, 11))[:2 if disk else 1]:
        s[:, o:o + 2] = p[:, o:o + 2] + 0.1 * p[:, r:r + 1] * u[:, o:o + 2]
        s[:, r + 2 if o == 0 else r + 1] = np.minimum(s[:, r + 2 if o == 0 else r + 1], 1.0)
    return s


METHOD = {"auto": gf.CONV_AUTO, "fft": gf.CONV_FFT, "direct": gf.CONV_DIRECT, "dft": gf.CONV_DFT_TC}


def stamps(case, seed):
    """Parameters, sizes, PSFs and noisy images of a case's stamps, and the library's description."""
    rng, gen = np.random.default_rng(seed), torch.Generator("cuda").manual_seed(seed)
    count, disk = case.get("count", 1), case["disk"]
    if "H" in case:
        H, W = np.array([case["H"]]), np.array([case["W"]])
    else:
        size = np.random.default_rng(count)  # the sizes belong to the case
        H = np.exp(size.uniform(math.log(case["lo"]), math.log(case["hi"] + 0.999), count)).astype(int)
        H = np.clip(H, case["lo"], case["hi"])
        W = H if case["lo"] == case["hi"] else np.clip(H + size.integers(-5, 6, count), case["lo"], case["hi"])
    bright = case["kind"] in ("fit", "fits", "jac")
    if disk:
        p = np.array([bulge_disk_draw(rng, h, w, bright) + [SKY] for h, w in zip(H, W)])
    else:
        p = unit_flux_ie(np.array([sersic_draw(rng, h, w, bright) + [SKY] for h, w in zip(H, W)]))
    psf = moffat(rng.uniform(2.0, 5.0, count), case["P"])
    pd, b = torch.as_tensor(p, device="cuda"), bn_of(torch.as_tensor(p[:, 4])).cuda()
    img, sig = [], []
    if count > 1 and H.min() == H.max() and W.min() == W.max():
        step = max(1, 24_000_000 // ((H[0] + case["P"]) * (W[0] + case["P"])))
        todo = [slice(k, k + step) for k in range(0, count, step)]
    else:
        todo = [slice(k, k + 1) for k in range(count)]
    for t in todo:
        m, s = noisy(render(pd[t], psf[t], int(H[t][0]), int(W[t][0]), disk, case["os"], case["box"], b[t]), gen)
        img.append(m.reshape(-1))
        sig.append(s.reshape(-1))
    kinds = [gf.SERSIC, gf.EXPDISK, gf.SKY] if disk else [gf.SERSIC, gf.SKY]
    d = gf.make_desc(int(H[0]), int(W[0]), case["P"], kinds, case["os"], case["box"], conv_method=METHOD[case["method"]])
    fixed = np.zeros(p.shape[1], np.uint8)
    fixed[[7, 14] if disk else [7]] = 1  # boxiness held
    return dict(d=d, p=p, H=H, W=W, psf=psf, img=torch.cat(img), sig=torch.cat(sig), fixed=fixed, rng=rng, ws=gf.Workspace())


def galaxies(case, seed):
    """Survey stamps for the network, rendered without the oversampled block: the network sees images only."""
    return stamps(dict(kind="evals", count=case["count"], lo=64, hi=64, P=learned.PSF_SIZE, disk=False, os=1, box=0, method="fft"), seed)


def lines(case, seed):
    """An emission-line complex on a sloped continuum per spaxel: amplitudes fall off, centres shift."""
    rng, gen = np.random.default_rng(seed), torch.Generator("cuda").manual_seed(seed)
    n, count, k = case["n_chan"], case["count"], case["lines"]
    r = np.sqrt(rng.uniform(0.0, 1.0, count))
    p = np.zeros((count, case["cont"] + 3 * k))
    for j, (lo, hi) in enumerate(((30.0, 50.0), (-3.0, 3.0), (-2.0, 2.0))[:case["cont"]]):
        p[:, j] = rng.uniform(lo, hi, count)
    base = 0.5 * n + 0.06 * n * np.tanh(3.0 * r) * np.cos(rng.uniform(0.0, 2.0 * math.pi, count))
    w = rng.uniform(2.0, 4.0, count)
    for i in range(k):
        o = case["cont"] + 3 * i
        p[:, o] = (2500.0 * np.exp(-1.5 * r) + 300.0) * (0.35, 1.0, 0.9)[i] * rng.uniform(0.9, 1.1, count)
        p[:, o + 1] = base + (i - 1) * max(0.03 * n, 20.0)
        p[:, o + 2] = w
    v = np.arange(case["lsf"]) - (case["lsf"] - 1) // 2
    lsf = np.exp(-0.5 * (v / 1.27) ** 2)
    lsf = torch.as_tensor((lsf / lsf.sum()).astype(np.float32), device="cuda")
    img, sig = noisy(spectra(torch.as_tensor(p, device="cuda"), lsf, n, case["cont"]), gen)
    u = rng.uniform(-1.0, 1.0, p.shape)
    s = p * (1.0 + 0.1 * u)
    s[:, case["cont"] + 1::3] = p[:, case["cont"] + 1::3] + 0.1 * w[:, None] * u[:, case["cont"] + 1::3]
    return dict(p=p, lsf=lsf, img=img, sig=sig, start=torch.as_tensor(s, device="cuda"))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "cube":
        s = lines(case, seed)
        s["d"] = gf.make_spec_desc(case["n_chan"], case["lines"], case["cont"], case["lsf"])
    elif kind in ("starts", "grad"):
        s = galaxies(case, seed)
        s["w"] = gf.cnn_init(seed)
        s["b"] = learned.uniform_batch(case["count"])
        s["d"] = learned.stamp_desc()
        if kind == "grad":
            # the network's input, asinh of the stamp over its ring's noise, and scaled targets
            s["x"] = torch.asinh(s["img"].view(-1, 64, 64) / READ).contiguous()
            s["t"] = torch.as_tensor(s["rng"].uniform(-1.0, 1.0, (case["count"], 8)), dtype=torch.float32, device="cuda")
    else:
        s = stamps(case, seed)
        if kind in ("fit", "fits"):
            s["start"] = start_of(s["p"], s["rng"], case["disk"])
            s["opts"] = gf.default_opts(ftol=case["tol"], xtol=case["tol"])
        elif kind == "jac":
            s["start"] = start_of(s["p"], s["rng"], case["disk"])[0]
        if kind in ("evals", "fits"):
            s["b"] = gf.make_batch(s["H"], s["W"], psf_size=case["P"])
        else:
            s["psf"] = s["psf"][0].contiguous()
    s["kind"] = kind
    return s


def run(s):
    kind = s["kind"]
    if kind == "eval":
        x2, m = gf.evaluate(s["d"], s["p"][0], s["img"], s["sig"], s["psf"], ws=s["ws"])
        return dict(chi2=x2.float(), model=m)
    if kind == "evals":
        x2, m = gf.evaluate_batch(s["d"], s["b"], s["p"], s["img"], s["sig"], s["psf"], want_model=True, ws=s["ws"])
        return dict(chi2=x2.float(), model=m)
    if kind == "fit":
        p, r = gf.lm_fit(s["d"], s["start"][0], s["fixed"], s["img"], s["sig"], s["psf"], s["opts"], ws=s["ws"])
        return dict(params=p.astype(np.float32), chi2=np.float32(r["chi2"]), status=r["status"])
    if kind == "fits":
        p, r = gf.lm_fit_batch(s["d"], s["b"], s["start"], s["fixed"], s["img"], s["sig"], s["psf"], s["opts"], ws=s["ws"])
        return dict(params=p.astype(np.float32), chi2=r.chi2.astype(np.float32), status=r.status)
    if kind == "jac":
        r = gf.jacobian(s["d"], s["start"], s["fixed"], s["img"], s["sig"], s["psf"], analytic=True, ws=s["ws"])
        return dict(J=r["J"], A=r["A"].float(), g=r["g"].float(), chi2=r["chi2"].float())
    if kind == "starts":
        out, choice, dflt = learned.starts(s["w"], s["b"], s["img"], s["sig"], s["psf"], s["d"], ws=s["ws"])
        return dict(starts=out.float(), choice=choice, default=dflt.float())
    if kind == "grad":
        loss, grad = gf.cnn_loss_grad(s["w"], s["x"], s["t"], ws=s["ws"])
        return dict(loss=loss, grad=grad)
    p, res = gf.spec_fit(s["d"], s["start"], None, s["img"], s["sig"], s["lsf"])
    return dict(params=p.float(), chi2=res.view(torch.float64)[:, 0].float(), status=res.view(torch.int32)[:, 6])


def exact(case, seed):
    kind = case["kind"]
    if kind in ("starts", "grad"):
        return None  # a bf16 network
    s = prepare(case, seed)
    if kind == "cube":
        p = torch.as_tensor(s["p"], device="cuda")
        f = lambda q: spectra(q, s["lsf"], case["n_chan"], case["cont"])  # noqa: E731
        step = max(1, 2_000_000 // case["n_chan"])
        x2 = [least(lambda q: f(q), p[k:k + step], list(range(p.shape[1])), s["img"][k:k + step], s["sig"][k:k + step])
              for k in range(0, len(p), step)]
        return dict(params=None, chi2=torch.cat(x2), status=None)
    disk, os, box = case["disk"], case["os"], case["box"]
    p = torch.as_tensor(s["p"], device="cuda")
    if kind == "evals":
        at, x2, models = 0, [], []
        for k in range(len(p)):
            n = int(s["H"][k] * s["W"][k])
            m = render(p[k], s["psf"][k], int(s["H"][k]), int(s["W"][k]), disk, os, box)
            x2.append(chi2_of(m, s["img"][at:at + n].view(m.shape), s["sig"][at:at + n].view(m.shape)))
            models.append(m.reshape(-1))
            at += n
        return dict(chi2=torch.stack(x2), model=torch.cat(models))
    if kind == "fits":
        return None  # thousands of fits: too long in 64 bits here
    H, W = case["H"], case["W"]
    img, sig = s["img"].view(H, W), s["sig"].view(H, W)
    free = [i for i in range(p.shape[1]) if not s["fixed"][i]]
    if kind == "eval":
        m = render(p[0], s["psf"], H, W, disk, os, box)
        return dict(chi2=chi2_of(m, img, sig)[None], model=m)
    if kind == "fit":
        x2 = least(lambda q: render(q, s["psf"], H, W, disk, os, box), p, free, img[None], sig[None])
        return dict(params=None, chi2=x2[0], status=None)
    p = torch.as_tensor(s["start"], device="cuda")
    f = lambda q: render(q, s["psf"], H, W, disk, os, box)  # noqa: E731
    J = []
    for i in free:
        h = torch.zeros_like(p)
        h[i] = 1e-5 * max(1.0, abs(float(p[i])))
        J.append((f(p + h) - f(p - h)) / (2.0 * h[i]))
    J, m = torch.stack(J), f(p)
    w = sig.to(F64) ** -2
    A = torch.einsum("ihw,jhw,hw->ij", J, J, w)
    return dict(J=J, A=A, g=torch.einsum("ihw,hw->i", J, w * (img.to(F64) - m)), chi2=chi2_of(m, img, sig)[None])


# ----------------------------------------------------------------------- work
def work(case):
    """Bytes: inputs once, outputs once.  Flops: per model evaluation of a pixel about 40 for each
    component and the FFT convolution's 5 N log2 N; a fit at least evaluates its columns and one
    trial per step over some 8 steps, each of them needing the image and sigma once."""
    kind = case["kind"]
    if kind == "grad":
        macs = 32 * 32 * 32 * 9 + 16 * 16 * 64 * 32 * 9 + 8 * 8 * 64 * 64 * 9 + 4 * 4 * 128 * 64 * 9 + 2048 * 32 + 256
        return dict(bytes=case["count"] * (4 * 4096 + 64.0) + 8 * 195432.0, flops=6.0 * macs * case["count"])
    if kind == "starts":
        macs = 32 * 32 * 32 * 9 + 16 * 16 * 64 * 32 * 9 + 8 * 8 * 64 * 64 * 9 + 4 * 4 * 128 * 64 * 9 + 2048 * 32 + 256
        fft = 2.0 * (5.0 * 9216 * math.log2(9216.0) + 40.0 * 9216)
        return dict(bytes=case["count"] * (8.0 * 4096 + 4.0 * 33 * 33 + 160), flops=case["count"] * (2.0 * macs + fft))
    if kind == "cube":
        npar = case["cont"] + 3 * case["lines"]
        per = case["n_chan"] * (20.0 * case["lines"] + 2.0 * case["lsf"]) + case["n_chan"] * npar * (npar + 3.0) + 2.0 * npar * case["lsf"] * case["n_chan"] * 0.1
        return dict(bytes=case["count"] * (8.0 * case["n_chan"] + 16.0 * npar + 32), flops=6.0 * case["count"] * per)
    count = case.get("count", 1)
    if "H" in case:
        h, w = case["H"], case["W"]
    else:
        lo, hi = case["lo"], case["hi"] + 1.0
        h = w = math.sqrt((hi * hi - lo * lo) / (2.0 * math.log(hi / lo)))  # the mean area of log-uniform sides
    grid, comps = (h + case["P"] - 1) * (w + case["P"] - 1), 2 if case["disk"] else 1
    one = grid * (40.0 * comps + 5.0 * math.log2(grid)) + 40.0 * comps * (case["os"] * case["box"]) ** 2
    pix, nf = count * h * w, 15 - 1 if case["disk"] else 8
    if kind in ("eval", "evals"):
        return dict(bytes=12.0 * pix + 4.0 * count * case["P"] ** 2, flops=count * one)
    columns = (nf - 1) * one + h * w * nf * (nf + 3.0)
    if kind == "jac":
        return dict(bytes=pix * (8.0 + 4.0 * nf) + 4.0 * case["P"] ** 2, flops=columns)
    return dict(bytes=8.0 * (8.0 * pix + 4.0 * count * case["P"] ** 2), flops=8.0 * count * (columns + one))
