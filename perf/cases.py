"""The work that users of this framework have it do, as measurable cases.

Each case is one call (or one step of a pipeline) through the public entry
points of paper_2603_08593_gb300, with inputs drawn on the GPU from a seed:
star fields, noise, masks and stamps of the recipe that the repository's own
configurations use (sky 1000 ADU, read noise 6 ADU, power-law fluxes, PSF
widths that vary over the chip, saturation masks, bad columns, bleed trails).

  subtract    Plan.subtract of one or many CCD pairs, mixed or FP64
  templates   one science frame against several templates, median-combined,
              with the constant-photometric-ratio kernel
  apply       Plan.apply: a fitted kernel applied to a frame again
  detect      Detector on a difference image
  classify    RBModel.logits on the candidates' stamps
  train       RBModel.backward of one mini-batch and its gradients
  rotinv      RIModel.logits, the rotation-invariant classifier
  photometry  limiting_mag and aperture_flux on the differences of an exposure
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2603_08593_gb300 import binding as B

DEV = "cuda"
F64 = torch.float64
SKY, READ_NOISE = 1000.0, 6.0
SAT_CLIP, SAT_MASK = 6.5e4, 6.0e4
FWHM = 2.0 * math.sqrt(2.0 * math.log(2.0))
ZP = 25.0


def listed():
    return [
        # a cutout around one alert, differenced on its own: the smallest call, all latency
        dict(name="cutout", kind="subtract", H=160, W=192, L=5, DK=1, DB=1, batch=1, prec="mixed", graph=False,
             mask=0.02, columns=0),
        # the plain FP64 fit of a 512 x 512 pair without a mask, the configuration that parity is judged on
        dict(name="pair512_fp64", kind="subtract", H=512, W=512, L=7, DK=1, DB=1, batch=1, prec="fp64", graph=False,
             mask=0.0, columns=0),
        # a strip of a CCD at the survey's kernel size in FP64
        dict(name="strip_fp64", kind="subtract", H=512, W=2048, L=11, DK=2, DB=2, batch=1, prec="fp64", graph=False,
             mask=0.03, columns=2),
        # one DECam CCD pair at the survey's kernel size, the framework's headline call
        dict(name="ccd", kind="subtract", H=4096, W=2048, L=11, DK=2, DB=2, batch=1, prec="mixed", graph=False,
             mask=0.0, columns=2),
        # a share of an exposure: CCDs with uneven masks in one graph-captured call
        dict(name="exposure", kind="subtract", H=4096, W=2048, L=11, DK=2, DB=2, batch=10, prec="mixed", graph=True,
             mask=0.15, columns=2),
        # one science frame against five templates of odd size, kernel sum held constant
        dict(name="templates", kind="templates", H=1021, W=1193, L=9, DK=1, DB=1, batch=5, mask=0.03),
        # a stored kernel applied to a frame again
        dict(name="apply", kind="apply", H=4096, W=2048, L=11, DK=2, DB=2, batch=1),
        # candidates of one CCD's difference image
        dict(name="detect", kind="detect", H=4096, W=2048, batch=1, psf_sigma=0.76),
        # the stamps of an exposure, scored
        dict(name="classify", kind="classify", n=10000, max_batch=4096),
        # one mini-batch of classifier training
        dict(name="train", kind="train", n=256),
        # the rotation-invariant classifier on one CCD's candidates
        dict(name="rotinv", kind="rotinv", n=1000),
        # limiting magnitudes and forced fluxes on the differences of some CCDs
        dict(name="photometry", kind="photometry", H=4096, W=2048, batch=4, n=1024, forced=300, radius=1.31),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["subtract", "subtract", "subtract", "subtract", "templates", "apply", "detect", "classify",
                       "train", "rotinv", "photometry"])
    H, W = _log_int(rng, 128, 4096), _log_int(rng, 128, 2048)
    if kind in ("subtract", "templates", "apply"):
        # enough pixels for the fit to be well determined
        fits = [(L, D) for L in (3, 5, 7, 9, 11) for D in (0, 1, 2) if H * W >= 60 * (L * L * _nm(D) + _nm(D))]
        L, D = rng.choice(fits[-6:])
        if kind == "templates":
            return dict(kind=kind, H=min(H, 1500), W=W, L=L, DK=D, DB=D, batch=rng.randint(2, 7), mask=0.03)
        if kind == "apply":
            return dict(kind=kind, H=H, W=W, L=L, DK=D, DB=D, batch=rng.randint(1, 3))
        prec = rng.choice(["mixed", "mixed", "mixed", "fp64"])
        if prec == "fp64":
            H = min(H, 1024)
        batch = rng.randint(1, 4) if prec == "mixed" else 1
        return dict(kind=kind, H=H, W=W, L=L, DK=D, DB=rng.choice([D, 2]), batch=batch, prec=prec,
                    graph=rng.random() < 0.5, mask=rng.choice([0.0, 0.02, 0.1, 0.3]), columns=rng.randint(0, 3))
    if kind == "detect":
        return dict(kind=kind, H=H, W=W, batch=rng.randint(1, 3), psf_sigma=rng.uniform(0.6, 1.6))
    if kind == "classify":
        return dict(kind=kind, n=_log_int(rng, 1, 20000), max_batch=4096)
    if kind == "train":
        return dict(kind=kind, n=_log_int(rng, 32, 1024))
    if kind == "rotinv":
        return dict(kind=kind, n=_log_int(rng, 1, 4000))
    return dict(kind=kind, H=H, W=W, batch=rng.randint(1, 6), n=_log_int(rng, 64, 2048), forced=_log_int(rng, 10, 1000),
                radius=rng.uniform(1.0, 6.0))


# ------------------------------------------------------------------ inputs
def _nm(d):
    return (d + 1) * (d + 2) // 2


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 2654435761 % (1 << 62))
    return g


def _uniform(g, lo, hi, n):
    return lo + (hi - lo) * torch.rand(n, generator=g, device=DEV, dtype=F64)


def _points(H, W, xs, ys, flux, sig, radius=8):
    """Sum of pixel-integrated Gaussians.  Light is added in whole units of 1/64 ADU, so that the order in which the
    GPU adds the stars does not show."""
    img = torch.zeros(H * W, dtype=torch.int64, device=DEV)
    off = torch.arange(-radius, radius + 1, device=DEV)
    px, py = (torch.floor(v + 0.5).long()[:, None] + off[None, :] for v in (xs, ys))
    s = (sig * math.sqrt(2.0))[:, None]
    fx, fy = (0.5 * (torch.erf((p + 0.5 - v[:, None]) / s) - torch.erf((p - 0.5 - v[:, None]) / s))
              for p, v in ((px, xs), (py, ys)))
    val = torch.round(64.0 * flux[:, None, None] * fy[:, :, None] * fx[:, None, :]).long()
    ok = ((py >= 0) & (py < H))[:, :, None] & ((px >= 0) & (px < W))[:, None, :]
    idx = py[:, :, None] * W + px[:, None, :]
    img.index_add_(0, idx[ok], val[ok])
    return (img.to(F64) / 64.0).reshape(H, W)


def _noisy(model, g):
    return torch.poisson((SKY + model).float(), generator=g) + READ_NOISE * torch.randn(model.shape, generator=g, device=DEV)


def _dilate(m, r, disc=False):
    H, W = m.shape
    p = F.pad(m, (r, r, r, r))
    out = m.clone()
    for dy in range(-r, r + 1):
        for dx in range(-r, r + 1):
            if not disc or dy * dy + dx * dx <= r * r:
                out |= p[r + dy:r + dy + H, r + dx:r + dx + W]
    return out


def _field(H, W, g, density=1.0 / 420):
    """Star positions, fluxes N(>F) ~ F^-1.5 on [1e3, 1e6] ADU and the PSF widths along the chip."""
    n = max(12, int(H * W * density))
    xs, ys, u = _uniform(g, -0.5, W - 0.5, n), _uniform(g, -0.5, H - 0.5, n), _uniform(g, 0.0, 1.0, n)
    flux = 1e3 * (1.0 - u * (1.0 - 1e-3 ** 1.5)) ** (-1.0 / 1.5)
    return xs, ys, flux


def _pair(H, W, seed, mask, columns, science=None):
    """One reference / science pair and its bad-pixel mask, all on the GPU."""
    g, rng = _gen(seed), np.random.default_rng(int(seed))
    xs, ys, flux = _field(H, W, _gen(seed if science is None else science))
    lo, hi = rng.uniform(0.95, 1.05), rng.uniform(1.35, 1.45)
    grow = 0.5 + 0.05 * rng.uniform(-1, 1)
    fw = lo + (hi - lo) * torch.clamp(ys / max(H - 1, 1), 0, 1)
    R = _noisy(_points(H, W, xs, ys, flux, fw / FWHM), g)
    gs = _gen(seed + 1 if science is None else science + 1)
    fs = 1.55 + 0.4 * torch.clamp(ys / max(H - 1, 1), 0, 1) + (grow - 0.5 if science is None else 0.0)
    model = _points(H, W, xs + 0.1, ys, flux, fs / FWHM)
    nt = max(1, min(50, H * W // 40000))        # transients at SNR 5-50
    snr = torch.exp(_uniform(gs, math.log(5.0), math.log(50.0), nt))
    sig = torch.full((nt,), 1.8 / FWHM, dtype=F64, device=DEV)
    model += _points(H, W, _uniform(gs, 8, W - 9, nt), _uniform(gs, 8, H - 9, nt),
                     snr * 32.19 * math.sqrt(4 * math.pi) * sig, sig)
    S = _noisy(model, gs)
    bad = _dilate((R > SAT_MASK) | (S > SAT_MASK), 3, disc=True)
    for c in rng.integers(0, W, columns):
        bad[:, int(c)] = True
    if mask > 0:
        for i in torch.argsort(flux, descending=True)[:max(1, flux.numel() // 400)].tolist():   # bleed trails
            x0, y0 = int(xs[i]), int(ys[i])
            half, ln = int(rng.integers(1, 3)), int(rng.integers(10, max(11, min(400, H // 3))))
            sl = (slice(max(0, y0 - ln), min(H, y0 + ln)), slice(max(0, x0 - half), min(W, x0 + half + 1)))
            R[sl] = S[sl] = SAT_CLIP
            bad[sl] = True
        for k in range(64):                      # strips along the edges, up to the masked fraction
            need = (mask - float(bad.float().mean())) * H * W
            if need <= 0:
                break
            if k % 2:
                w = int(min(W // 2, max(2, need / H * rng.uniform(0.3, 1.0))))
                bad[:, :w] = True
            else:
                h = int(min(H // 2, max(2, need / W * rng.uniform(0.3, 1.0))))
                wd = int(rng.integers(W // 4, W + 1))
                x = int(rng.integers(0, W - wd + 1))
                bad[H - h:, x:x + wd] = True
    return torch.clamp(R, max=SAT_CLIP).float(), torch.clamp(S, max=SAT_CLIP).float(), bad.to(torch.uint8)


def _pairs(case, seed):
    t = [_pair(case["H"], case["W"], seed * 64 + i, case.get("mask", 0.0) * (0.5 + i % 3 / 2.0), case.get("columns", 1),
               seed * 64 + 63 if case["kind"] == "templates" else None) for i in range(case["batch"])]
    R, S, bad = (torch.stack(v).contiguous() for v in zip(*t))
    if case["kind"] == "subtract" and case["mask"] == 0.0 and case["columns"] == 0:
        bad = None
    return R, S, bad


def _theta(case, seed):
    """A smooth kernel whose width varies over the chip, its background in original units."""
    L, NK, NB = case["L"], _nm(case["DK"]), _nm(case["DB"])
    rng = np.random.default_rng(seed + 5)
    u = np.arange(L) - (L - 1) // 2
    th = np.zeros((case["batch"], L * L * NK + NB))
    for b in range(case["batch"]):
        for p in range(NK):
            s = 0.8 + 0.2 * rng.random()
            k = np.exp(-(u[:, None] ** 2 + u[None, :] ** 2) / (2 * s * s))
            th[b, p:L * L * NK:NK] = (1.0 if p == 0 else 0.05 * rng.normal()) * (k / k.sum()).ravel() \
                + 1e-4 * rng.normal(size=L * L)
        th[b, L * L * NK:] = rng.normal(0, 5.0, NB)
    return torch.from_numpy(th).to(DEV)


def _stamps(n, seed):
    """Candidate stamps in raw ADU: a star or galaxy core in both frames, and half of them a transient in the science
    frame, the rest cosmic-ray hits or misregistered stars."""
    g = _gen(seed)
    off = torch.arange(31, device=DEV, dtype=torch.float32) - 15

    def blob(flux, x, y, s):
        e = lambda c: torch.exp(-(off[None, :] - c[:, None]) ** 2 / (2 * s * s))  # noqa: E731
        return flux[:, None, None] * e(y)[:, :, None] * e(x)[:, None, :] / (2 * math.pi * s * s)

    u = lambda lo, hi: lo + (hi - lo) * torch.rand(n, generator=g, device=DEV)  # noqa: E731
    label = (torch.rand(n, generator=g, device=DEV) < 0.5).float()
    host = 10 ** u(2.5, 5.0)
    x, y = u(-4, 4), u(-4, 4)
    shift = (1 - label) * u(0.3, 1.0)
    ref = SKY + blob(host, x, y, 0.55)
    hit = (1 - label) * (torch.rand(n, generator=g, device=DEV) < 0.4).float()
    sci = SKY + blob(host, x + shift, y, 0.8) + blob(label * 32.19 * 2.8 * 10 ** u(0.5, 2.0), u(-.5, .5), u(-.5, .5), 0.8)
    sci = sci + torch.randn(n, 31, 31, generator=g, device=DEV) * torch.sqrt(sci)
    ref = ref + torch.randn(n, 31, 31, generator=g, device=DEV) * torch.sqrt(ref)
    sci[:, 15, 15] += 1e4 * hit
    diff = sci - SKY - blob(host, x, y, 0.8) + 32.0 * torch.randn(n, 31, 31, generator=g, device=DEV)
    return torch.stack([sci, ref, diff], 1).contiguous(), label


_RB = [("w1", (32, 3, 3, 3)), ("b1", (32,)), ("w2", (64, 32, 3, 3)), ("b2", (64,)), ("w3", (64, 64, 3, 3)), ("b3", (64,)),
       ("w4", (128, 576)), ("b4", (128,)), ("w5", (1, 128)), ("b5", (1,))]
_RI = _RB[:2] + [("wa", (32, 32, 3, 3)), ("ba", (32,)), ("wb", (32, 32, 3, 3)), ("bb", (32,))] + _RB[2:4] + \
    [("wc", (64, 64, 3, 3)), ("bc", (64,)), ("wd", (64, 64, 3, 3)), ("bd", (64,))] + _RB[6:]


def _weights(shapes, seed):
    rng = np.random.default_rng(seed + 11)
    out = []
    for name, s in shapes:
        lim = math.sqrt(6.0 / max(1, int(np.prod(s[1:]))))
        out.append(rng.normal(0, 0.05, s) if name[0] == "b" else rng.uniform(-lim, lim, s))
    return np.concatenate([v.ravel() for v in out]).astype(np.float32)


def _difference(H, W, seed):
    """A difference image: noise, residuals of the bright stars, transients."""
    R, S, bad = _pair(H, W, seed, 0.02, 2)
    g = _gen(seed + 3)
    D = torch.randn(H, W, generator=g, device=DEV) * torch.sqrt(torch.clamp(R + S, min=1.0))
    n = max(4, H * W // 20000)
    sig = torch.full((n,), 0.76, dtype=F64, device=DEV)
    D += _points(H, W, _uniform(g, 0, W - 1, n), _uniform(g, 0, H - 1, n), 10 ** _uniform(g, 2.3, 4.0, n), sig).float()
    return D, S, R, bad


def prepare(case, seed):
    k = case["kind"]
    st = dict(case=case)
    if k in ("subtract", "templates"):
        st["R"], S, st["bad"] = _pairs(case, seed)
        st["S"] = S[0].contiguous() if k == "templates" else S
        st["stream"] = torch.cuda.Stream() if case.get("graph") else torch.cuda.current_stream()
        st["plan"] = p = B.Plan(case["H"], case["W"], case["L"], case["DK"], case["DB"], batch=case["batch"],
                                prec=case.get("prec", "mixed"), graph=bool(case.get("graph")), stream=st["stream"],
                                const_ratio=k == "templates")
        new = lambda *s, t=F64: torch.empty(*s, dtype=t, device=DEV)  # noqa: E731
        st["out"] = dict(A=new(p.batch, p.N, p.N), b=new(p.batch, p.N), theta=new(p.batch, p.N),
                         info=new(p.batch, t=torch.int32), D=new(p.batch, p.H, p.W, t=torch.float32))
        if k == "templates":
            st["scale"] = torch.from_numpy(np.random.default_rng(seed).uniform(0.8, 1.2, case["batch"])).float().to(DEV)
    elif k == "apply":
        st["R"], st["S"], _ = _pairs(dict(case, mask=0.0), seed)
        st["theta"] = _theta(case, seed)
        st["sky"] = torch.tensor([[1000.0, 1001.0]], dtype=F64, device=DEV).repeat(case["batch"], 1)
        st["plan"] = B.Plan(case["H"], case["W"], case["L"], case["DK"], case["DB"], batch=case["batch"], d_batch=1)
        st["D"] = torch.empty_like(st["S"])
    elif k == "detect":
        t = [_difference(case["H"], case["W"], seed * 64 + i) for i in range(case["batch"])]
        st["D"], st["S"], st["R"], st["bad"] = (torch.stack(v).contiguous() for v in zip(*t))
        st["det"] = d = B.Detector(case["H"], case["W"], batch=case["batch"])
        for t in (d.xy, d.snr, d.stamps):        # entries past a CCD's count are left as they were
            t.zero_()
    elif k in ("classify", "train", "rotinv"):
        st["stamps"], st["labels"] = _stamps(case["n"], seed)
        cls, shapes = (B.RIModel, _RI) if k == "rotinv" else (B.RBModel, _RB)
        st["model"] = cls(max_batch=case.get("max_batch", min(1024, case["n"])), seed=1)
        st["model"].set_weights(_weights(shapes, seed))
    else:
        t = [_difference(case["H"], case["W"], seed * 64 + i) for i in range(case["batch"])]
        st["D"], _, _, st["bad"] = (torch.stack(v).contiguous() for v in zip(*t))
        st["pos"] = B.random_positions(case["batch"], case["H"], case["W"], case["n"], seed)
        st["forced"] = B.random_positions(case["batch"], case["H"], case["W"], case["forced"], seed + 1, margin=2.0)
    torch.cuda.synchronize()
    return st


# ------------------------------------------------------------------ one pass
def run(st):
    c, k = st["case"], st["case"]["kind"]
    if k == "subtract":
        with torch.cuda.stream(st["stream"]):
            o = st["plan"].subtract(st["R"], st["S"], st["bad"], out=st["out"])
            if c["prec"] == "fp64":
                return o
            # a mixed plan sums in FP32 and its A and b are scratch of the call; a program keeps the fitted kernel
            # beside D in single precision
            return dict(D=o["D"], info=o["info"], theta=o["theta"].float())
    if k == "templates":
        comb, o = B.multi_template_difference(st["plan"], st["R"], st["S"], st["bad"], st["scale"])
        return dict(comb=comb, D=o["D"], info=o["info"], theta=o["theta"].float())
    if k == "apply":
        return st["plan"].apply(st["R"], st["S"], st["theta"], st["sky"], D=st["D"])
    if k == "detect":
        xy, snr, count, stamps = st["det"](st["D"], st["S"], st["R"], st["bad"], psf_sigma=c["psf_sigma"], thresh=5.0, guard=5)
        return dict(xy=xy, snr=snr, count=count, stamps=stamps)
    if k in ("classify", "rotinv"):
        return st["model"].logits(st["stamps"])
    if k == "train":
        loss = st["model"].backward(st["stamps"], st["labels"])
        return dict(loss=loss, grads=st["model"].get_grads())
    sigma, mlim, ngood = B.limiting_mag(st["D"], c["radius"], ZP, pos=st["pos"], bad=st["bad"])
    flux, flag = B.aperture_flux(st["D"], st["forced"], c["radius"], bad=st["bad"])
    return dict(sigma=sigma, mlim=mlim, ngood=ngood, flux=flux, flag=flag)


def work(case):
    """Bytes: each input read once, each output written once.  Flops: of a subtraction the factorisation, and per
    pixel one multiply-add for each of the L^2 taps (their coefficients combined) in the fit's residual and in D and
    for each distinct product sum of the normal matrix; of a network its layers."""
    k = case["kind"]
    if k in ("subtract", "templates", "apply"):
        px = case["H"] * case["W"] * case["batch"]
        LL, NK = case["L"] ** 2, _nm(case["DK"])
        N = LL * NK + _nm(case["DB"])
        if k == "apply":
            return dict(bytes=12 * px + 8 * N * case["batch"], flops=2 * LL * px)
        out = 8 * case["batch"] * ((N * N + 2 * N) if case.get("prec") == "fp64" else N)
        masked = k == "templates" or case["mask"] > 0 or case["columns"] > 0
        extra = case["H"] * case["W"] * 4 if k == "templates" else 0
        sums = 2 * case["L"] * (case["L"] - 1) + 1          # half-plane offset differences
        return dict(bytes=(12 + masked) * px + out + extra, flops=2 * px * (3 * LL + sums) + case["batch"] * N ** 3 / 3)
    if k == "detect":
        return dict(bytes=5 * case["H"] * case["W"] * case["batch"] + 4096 * case["batch"] * (31 * 31 * 12 + 12),
                    flops=2 * case["H"] * case["W"] * case["batch"] * 2 * (2 * math.ceil(3 * case["psf_sigma"]) + 1))
    if k in ("classify", "train"):
        f = 2 * (31 * 31 * 27 * 32 + 225 * 288 * 64 + 49 * 576 * 64 + 576 * 128 + 128)
        n = case["n"]
        return dict(bytes=n * (11532 + 4) + 4 * 130305 * (2 if k == "train" else 1), flops=f * n * (3 if k == "train" else 1))
    if k == "rotinv":
        f = 4 * 2 * (961 * 27 * 32 + 225 * 288 * (32 + 32 + 64) + 49 * 576 * 128) + 2 * (576 * 128 + 128)
        return dict(bytes=case["n"] * 11536 + 4 * 185729, flops=f * case["n"])
    side = 2 * math.ceil(case["radius"] + 1) + 1
    n = case["batch"] * (case["n"] + case["forced"])
    return dict(bytes=n * (side * side * 5 + 16 + 12), flops=n * side * side * 2)


# ------------------------------------------------------------------ the same in 64 bits, in plain torch
def _powers(H, W, D, rows=None):
    x = 2.0 * torch.arange(W, device=DEV, dtype=F64) / max(W - 1, 1) - 1.0
    y = 2.0 * torch.arange(H, device=DEV, dtype=F64) / max(H - 1, 1) - 1.0
    y = y if rows is None else y[rows]
    return [(x[None, :] ** (n - b)) * (y[:, None] ** b) for n in range(D + 1) for b in range(n + 1)]


def _taps(img, w):
    """img(x - u) for the L^2 offsets u, zero outside, one by one."""
    H, W = img.shape
    P = F.pad(img, (w, w, w, w))
    for uy in range(-w, w + 1):
        for ux in range(-w, w + 1):
            yield P[w - uy:w - uy + H, w - ux:w - ux + W]


def _fit64(R, S, bad, case, const_ratio):
    """One CCD's A, b, theta (original units) and D in 64 bits, from the design rows."""
    H, W, L, DK, DB = (case[k] for k in ("H", "W", "L", "DK", "DB"))
    w, NK, NB = (L - 1) // 2, _nm(DK), _nm(DB)
    N = L * L * NK + NB
    good = torch.ones(H, W, dtype=torch.bool, device=DEV) if bad is None else bad == 0
    sR, sS = (torch.round(v.double()[good].mean()) for v in (R, S))
    Rm, Rt, S0 = torch.where(good, R.double() - sR, 0.0), R.double() - sR, S.double() - sS
    fit = ~_dilate(~good, w)
    fit[:w] = fit[H - w:] = False
    fit[:, :w] = fit[:, W - w:] = False
    A, b = torch.zeros(N, N, dtype=F64, device=DEV), torch.zeros(N, dtype=F64, device=DEV)
    taps = list(_taps(Rm, w))
    step = max(1, 65536 // W)
    for y in range(0, H, step):
        rows = slice(y, min(H, y + step))
        m, phi = fit[rows], _powers(H, W, DK, rows)
        X = torch.stack([(t[rows] * f)[m] for t in taps for f in phi] + [f[m] for f in _powers(H, W, DB, rows)], 1)
        A += X.T @ X
        b += X.T @ S0[rows][m]
        del X
    if const_ratio:
        c = L * L // 2
        T = torch.zeros((L * L - 1) * NK + 1 + NB, N, dtype=F64, device=DEV)
        i = 0
        for j in [c] + [j for j in range(L * L) if j != c]:
            for p in range(1 if j == c else NK):
                T[i, j * NK + p] = 1.0
                if j != c:
                    T[i, c * NK + p] = -1.0
                i += 1
        T[i:, L * L * NK:] = torch.eye(NB, dtype=F64, device=DEV)
    else:
        T = torch.eye(N, dtype=F64, device=DEV)
    M = T @ A @ T.T
    s = torch.rsqrt(torch.diagonal(M))
    Lf = torch.linalg.cholesky(M * s[:, None] * s[None, :])
    r, th = T @ b, torch.zeros(T.shape[0], dtype=F64, device=DEV)
    for _ in range(2):
        th = th + s * torch.cholesky_solve((s * (r - M @ th))[:, None], Lf)[:, 0]
    th = T.T @ th
    phi, psi = _powers(H, W, DK), _powers(H, W, DB)
    D = S0.clone()
    for j, t in enumerate(_taps(Rt, w)):
        D -= t * sum(th[j * NK + p] * phi[p] for p in range(NK))
    D -= sum(th[L * L * NK + q] * psi[q] for q in range(NB))
    out = th.clone()
    for q in range(min(NK, NB)):
        out[L * L * NK + q] += (sS if q == 0 else 0.0) - sR * th[q:L * L * NK:NK].sum()
    return A, b, out, D


def _normalised(stamps):
    x = stamps.double()
    f = x.reshape(x.shape[0], 3, -1)
    med = f.median(2, keepdim=True).values
    mad = 1.4826 * (f - med).abs().median(2, keepdim=True).values
    return (((f - med) / torch.where(mad > 0, mad, 1.0)).clamp(-64, 64)).reshape(x.shape)


def _unpack(shapes, flat):
    out, i = {}, 0
    for name, s in shapes:
        n = int(np.prod(s))
        out[name] = flat[i:i + n].reshape(s)
        i += n
    return out


def _conv(x, p, k):
    """3 x 3 'same' convolution as nine products, without a library's convolution."""
    n, c, h, w = x.shape
    cols = F.unfold(x, 3, padding=1)
    return (p["w" + k].reshape(p["w" + k].shape[0], -1) @ cols).reshape(n, -1, h, w) + p["b" + k][None, :, None, None]


def _head(x, p):
    h = torch.relu(x.reshape(x.shape[0], -1) @ p["w4"].T + p["b4"])
    return (h @ p["w5"].T + p["b5"])[:, 0]


def _net(x, p, rotinv):
    pool = lambda v: F.max_pool2d(torch.relu(v), 2)  # noqa: E731
    if not rotinv:
        return _head(pool(_conv(pool(_conv(pool(_conv(x, p, "1")), p, "2")), p, "3")), p)
    feats = 0.0
    for q in range(4):
        a = pool(_conv(torch.rot90(x, q, (2, 3)), p, "1"))
        a = torch.relu(a + _conv(torch.relu(_conv(a, p, "a")), p, "b"))
        a = pool(_conv(a, p, "2"))
        feats = feats + F.max_pool2d(torch.relu(a + _conv(torch.relu(_conv(a, p, "c")), p, "d")), 2)
    return _head(feats / 4.0, p)


def _apertures(D, bad, pos, r):
    H, W = D.shape
    m = int(math.ceil(r + 1)) + 1
    off = torch.arange(-m, m + 1, device=DEV)
    px, py = (torch.floor(pos[:, i] + 0.5).long()[:, None] + off[None, :] for i in (0, 1))
    sub = (torch.arange(5, device=DEV, dtype=F64) + 0.5) / 5
    dx, dy = ((((p.double() - 0.5)[..., None] + sub) - pos[:, i, None, None]) ** 2 for i, p in ((0, px), (1, py)))
    wt = (dy[:, :, None, :, None] + dx[:, None, :, None, :] <= r * r).sum((3, 4)).double() / 25.0
    ok = ((py >= 0) & (py < H))[:, :, None] & ((px >= 0) & (px < W))[:, None, :]
    yi, xi = py.clamp(0, H - 1)[:, :, None], px.clamp(0, W - 1)[:, None, :]
    ok = ok & (bad[yi, xi] == 0)
    return (wt * torch.where(ok, D[yi, xi].double(), 0.0)).sum((1, 2)), ((wt > 0) & ~ok).any(2).any(1)


def _matched64(D, bad, sigma, max_cand, thresh=5.0, guard=5, edge=15):
    """The matched-filter SNR of one image's candidates, in row-major order."""
    H, W = D.shape
    good, inside = bad == 0, torch.zeros(H, W, dtype=torch.bool, device=DEV)
    inside[edge:H - edge, edge:W - edge] = True
    v = D.double()[good & inside]
    mu, var = v.mean(), v.var(unbiased=False)
    for _ in range(3):
        s = v[(v - mu).abs() <= 3.0 * var.sqrt()]
        mu, var = s.mean(), s.var(unbiased=False)
    r = int(math.ceil(3.0 * sigma))
    t = [math.exp(-i * i / (2.0 * sigma * sigma)) for i in range(-r, r + 1)]
    P = F.pad(torch.where(good, D.double(), 0.0), (r, r, r, r))
    P = sum(a * P[:, i:i + W] for i, a in enumerate(t))
    snr = sum(a * P[i:i + H] for i, a in enumerate(t)) / (torch.sqrt(var / 0.97334) * sum(a * a for a in t))
    top = F.max_pool2d(snr[None, None], 5, 1, 2)[0, 0]
    found = snr[inside & ~_dilate(~good, guard) & (snr >= thresh) & (snr >= top)][:max_cand]
    return F.pad(found, (0, max_cand - found.numel()))


def exact(case, seed):
    k, st = case["kind"], prepare(case, seed)
    if k in ("subtract", "templates"):
        N = case["L"] ** 2 * _nm(case["DK"]) + _nm(case["DB"])
        if 2.0 * N * N * case["H"] * case["W"] * case["batch"] > 1.2e13:
            return None
        bad = st["bad"]
        fits = [_fit64(st["R"][i], st["S"] if k == "templates" else st["S"][i], None if bad is None else bad[i], case,
                       k == "templates") for i in range(case["batch"])]
        A, b, th, D = (torch.stack(v) for v in zip(*fits))
        if k == "templates":
            v = torch.where(bad == 0, D * st["scale"].double()[:, None, None], float("nan"))
            n = (bad == 0).sum(0)
            s = torch.sort(v, 0).values             # not-a-numbers last
            pick = lambda i: torch.gather(s, 0, i.clamp(min=0)[None])[0]  # noqa: E731
            return dict(comb=0.5 * (pick((n - 1) // 2) + pick(n // 2)), D=D, info=None, theta=th)
        return dict(A=A, b=b, theta=th, info=None, D=D) if case["prec"] == "fp64" else dict(D=D, info=None, theta=th)
    if k == "apply":
        w, NK, NB, LL = (case["L"] - 1) // 2, _nm(case["DK"]), _nm(case["DB"]), case["L"] ** 2
        phi, psi, out = _powers(case["H"], case["W"], case["DK"]), _powers(case["H"], case["W"], case["DB"]), []
        for i in range(case["batch"]):
            sR, th = st["sky"][i, 0], st["theta"][i]
            D = st["S"][i].double() - sum(th[LL * NK + q] * psi[q] for q in range(NB))
            sums = [th[p:LL * NK:NK].sum() for p in range(NK)]
            for q in range(min(NK, NB)):
                D -= sR * sums[q] * psi[q]
            for j, t in enumerate(_taps(st["R"][i].double() - sR, w)):
                D -= t * sum(th[j * NK + p] * phi[p] for p in range(NK))
            out.append(D)
        return torch.stack(out)
    if k == "detect":
        got = [_matched64(st["D"][i], st["bad"][i], case["psf_sigma"], st["det"].max_cand) for i in range(case["batch"])]
        return dict(xy=None, snr=torch.stack(got), count=None, stamps=None)
    if k in ("classify", "rotinv", "train"):
        shapes = _RI if k == "rotinv" else _RB
        flat = torch.from_numpy(_weights(shapes, seed)).double().to(DEV).requires_grad_(k == "train")
        x = _normalised(st["stamps"])
        if k == "train":
            z = _net(x, _unpack(shapes, flat), False)
            loss = F.binary_cross_entropy_with_logits(z, st["labels"].double())
            loss.backward()
            return dict(loss=loss.detach().reshape(1), grads=flat.grad)
        with torch.no_grad():
            return torch.cat([_net(x[i:i + 512], _unpack(shapes, flat), k == "rotinv") for i in range(0, len(x), 512)])
    got = []
    for i in range(case["batch"]):
        f, bad = _apertures(st["D"][i], st["bad"][i], st["pos"][i], case["radius"])
        s = f[~bad].std()
        got.append((s, ZP - 2.5 * torch.log10(5.0 * s), _apertures(st["D"][i], st["bad"][i], st["forced"][i], case["radius"])[0]))
    s, m, f = (torch.stack(v) for v in zip(*got))
    return dict(sigma=s, mlim=m, ngood=None, flux=f, flag=None)
