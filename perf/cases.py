"""Performance cases of the Haar-tSVD denoiser: what a user's program has it do, through its public entry points.

listed() names the cases, draw() gives more of the same ranges, prepare() makes the inputs a caller
has in hand, run() is one pass, work() what a pass cannot do without, and exact() the same outputs in
64-bit torch arithmetic without this package's code.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2508_10307_gb300 as htsvd

DEV = "cuda:0"
DEFAULTS = dict(stride=3, window=18, K=32, tau_mult=0.0, match="auto", agg="uniform", sigma=25.0)


def listed():
    return [
        # A gray thumbnail or image tile at a known noise level: the smallest call, latency and launches.
        dict(name="gray128", kind="image", H=128, W=128, C=1, stride=3, window=21, K=16, tau_mult=2.7),
        # A photograph-sized image of odd extent at the method's default parameters, sparsity weights.
        dict(name="rgb_default_odd", kind="image", H=321, W=481, C=3, agg="sparsity"),
        # A 512 x 512 photograph whose noise level is not known: grouping returned beside the estimate.
        dict(name="rgb512_sigma_est", kind="image", H=512, W=512, C=3, stride=2, window=31, sigma=15.0, est=True),
        # One gray full-HD frame (a microscope's or a monochrome camera's).
        dict(name="gray1080", kind="image", H=1080, W=1920, C=1, window=31, sigma=20.0),
        # One 4K colour frame at the quality setting: the largest image.
        dict(name="rgb4k", kind="image", H=2160, W=3840, C=3, window=31),
        # A folder of photographs of uneven sizes, each at its own noise level, as one batch call.
        dict(name="batch_uneven", kind="batch", n=12, lo=256, hi=1024, C=3),
        # Training through the denoiser: forward and backward on a float image, gradients of the image
        # and of the per-group weights.
        dict(name="grad512", kind="grad", H=512, W=512, C=3),
        # A full-HD colour clip, grouping over the neighbouring frames, noise level per frame.
        dict(name="video1080", kind="video", F=4, H=1080, W=1920, C=3, T=1, window=31, sigma=15.0, est=True),
        # A hyperspectral scene of 34 bands.
        dict(name="hsi34", kind="cube", H=520, W=696, C=34, sigma=12.0),
        # A T1-weighted head scan at the method's MRI setting.
        dict(name="mri176", kind="volume", D=176, H=208, W=176, stride=2, window=5, sigma=11.5),
        # Choosing a threshold: one image at eight multipliers.
        dict(name="sweep512", kind="sweep", H=512, W=512, C=3, stride=2, window=31, sigma=15.0, n=8),
        # The image cut into parts, each at its own estimated noise level (the adaptive variant).
        dict(name="adaptive768", kind="adaptive", H=768, W=768, C=3, sub=256, window=31, sigma=15.0, est=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["image"] * 7 + ["batch", "grad", "grad", "video", "cube", "volume", "sweep", "adaptive"])
    c = dict(kind=kind, C=rng.choice([1, 3, 3]), stride=rng.choice([2, 3, 3, 4]), window=rng.randint(15, 31),
             K=rng.choice([8, 16, 32, 32]), sigma=round(rng.uniform(5.0, 50.0), 1),
             agg=rng.choice(["uniform", "uniform", "sparsity"]))
    if kind == "image":
        c.update(H=_log(rng, 64, 1600), W=_log(rng, 64, 2000), est=rng.random() < 0.3,
                 match=rng.choice(["auto", "auto", "auto", "full", "green"]))
    elif kind == "batch":
        c.update(n=rng.randint(2, 12), lo=_log(rng, 64, 256), hi=_log(rng, 256, 900))
    elif kind == "grad":
        c.update(H=_log(rng, 48, 640), W=_log(rng, 48, 640))
    elif kind == "video":
        c.update(F=rng.randint(2, 4), H=_log(rng, 96, 720), W=_log(rng, 96, 1280), T=rng.choice([1, 1, 2]),
                 est=rng.random() < 0.5, window=rng.randint(15, 25))
    elif kind == "cube":
        c.update(H=_log(rng, 48, 360), W=_log(rng, 48, 360), C=rng.randint(4, 40), stride=rng.choice([3, 4]),
                 window=rng.randint(12, 18))
    elif kind == "volume":
        c.update(D=_log(rng, 24, 160), H=_log(rng, 24, 160), W=_log(rng, 24, 160), stride=rng.choice([2, 3]),
                 window=rng.randint(4, 6), est=rng.random() < 0.3)
        del c["C"]
    elif kind == "sweep":
        c.update(H=_log(rng, 64, 512), W=_log(rng, 64, 512), n=rng.randint(2, 8))
    else:
        c.update(H=_log(rng, 128, 900), W=_log(rng, 128, 900), sub=rng.randint(96, 256), est=True)
    return c


def _full(case):
    c = dict(DEFAULTS, **case)
    if c["kind"] == "volume":
        c["C"] = 4                                     # the tube of a 4 x 4 x 4 cube
    return c


def _params(c):
    p = dict(stride=c["stride"], window=c["window"], K=c["K"], tau_mult=c["tau_mult"], agg_mode=c["agg"],
             match_mode=c["match"])
    if c["kind"] == "volume":
        p["ps"] = 4
    return p


# ---- inputs: smooth objects, textures and edges under sensor noise, on the 0..255 scale

def _layer(rs, axes):
    """One smooth layer over the given coordinate axes: soft ellipsoids and plane-wave textures on a flat ground."""
    nd = len(axes)
    grid = [a.view([-1 if i == d else 1 for i in range(nd)]) for d, a in enumerate(axes)]
    ext = [float(a.numel()) for a in axes]
    img = torch.full([a.numel() for a in axes], 128.0, device=DEV)
    for _ in range(20):
        rho2 = 0.0
        for g, n in zip(grid, ext):
            rho2 = rho2 + ((g - rs.uniform(0, n)) / (rs.uniform(0.05, 0.4) * n)) ** 2
        img += rs.uniform(-80, 80) * torch.sigmoid(8.0 - 8.0 * torch.sqrt(rho2))
    for _ in range(3):
        d = rs.normal(size=nd)
        d /= np.linalg.norm(d)
        wave = rs.uniform(0, 2 * np.pi)
        period = rs.uniform(4, 16)
        for g, k in zip(grid, d):
            wave = wave + (2 * np.pi * k / period) * g
        img += rs.uniform(5, 25) * torch.sin(wave)
    return img.clamp_(0, 255)


def _clean(seed, H, W, C):
    rs = np.random.RandomState(seed % (1 << 31))
    axes = [torch.arange(n, dtype=torch.float32, device=DEV) for n in (H, W)]
    base = _layer(rs, axes)
    if C == 1:
        return base.unsqueeze(-1)
    if C == 3:                                          # colour planes share most of their content
        return torch.stack([128 + 0.8 ** 0.5 * (base - 128) + 0.2 ** 0.5 * (_layer(rs, axes) - 128)
                            for _ in range(3)], dim=-1).clamp_(0, 255)
    b = torch.arange(C, dtype=torch.float32, device=DEV)   # three endmember spectra
    cube = 20.0 + 30.0 * b / max(C - 1, 1) + torch.zeros(H, W, C, device=DEV)
    for _ in range(3):
        ab = _layer(rs, axes) / 255.0
        spec = rs.uniform(60, 140) * torch.exp(-0.5 * ((b - rs.uniform(0, C)) / (rs.uniform(0.15, 0.6) * C)) ** 2)
        cube += ab.unsqueeze(-1) * spec
    return cube.clamp_(0, 255)


def _noisy(x, sigma, seed, quantise=True):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed + 7919)
    y = x + sigma * torch.randn(x.shape, generator=gen, device=DEV)
    return y.round_().clamp_(0, 255).to(torch.uint8) if quantise else y.contiguous()


def _batch_shapes(c, seed):
    # the sizes belong to the case, the pictures to the seed
    rs = np.random.RandomState(c["n"] * 7919 + c["lo"] * 31 + c["hi"])
    return [(int(rs.randint(c["lo"], c["hi"] + 1)), int(rs.randint(c["lo"], c["hi"] + 1)),
             float(rs.uniform(10, 50))) for _ in range(c["n"])]


def prepare(case, seed):
    c = _full(case)
    kind = c["kind"]
    st = dict(case=c, params=_params(c), sigma=None if c.get("est") else c["sigma"])
    if kind == "batch":
        shapes = _batch_shapes(c, seed)
        st["x"] = [_noisy(_clean(seed + 101 * i, h, w, c["C"]), s, seed + 101 * i)
                   for i, (h, w, s) in enumerate(shapes)]
        st["sigma"] = [s for _, _, s in shapes]
    elif kind == "video":                               # content drifting one pixel a frame, fresh noise
        wide = _clean(seed, c["H"], c["W"] + c["F"], c["C"])
        st["x"] = torch.stack([_noisy(wide[:, t:t + c["W"]], c["sigma"], seed + 13 * t) for t in range(c["F"])])
    elif kind == "volume":
        rs = np.random.RandomState(seed % (1 << 31))
        axes = [torch.arange(c[k], dtype=torch.float32, device=DEV) for k in "DHW"]
        rho2 = sum((((a - a.numel() / 2) / (0.45 * a.numel())) ** 2).view([-1 if i == d else 1 for i in range(3)])
                   for d, a in enumerate(axes))
        head = torch.sigmoid(8.0 - 8.0 * torch.sqrt(rho2))   # soft outline, no signal outside
        st["x"] = _noisy(_layer(rs, axes) * head, c["sigma"], seed)
    else:
        st["x"] = _noisy(_clean(seed, c["H"], c["W"], c["C"]), c["sigma"], seed, quantise=kind != "grad")
    if kind == "grad":
        gen = torch.Generator(device=DEV)
        gen.manual_seed(seed + 17)
        n = htsvd.num_groups(c["H"], c["W"], st["params"])
        st["x"].requires_grad_(True)
        st["w"] = (0.5 + torch.rand(n, generator=gen, device=DEV)).requires_grad_(True)
        st["gout"] = torch.randn(st["x"].shape, generator=gen, device=DEV)
    if kind == "sweep":
        st["mults"] = [2.0 + 3.0 * i / c["n"] for i in range(c["n"])]
    return st


def run(st):
    c, p, x, sigma = st["case"], st["params"], st["x"], st["sigma"]
    kind = c["kind"]
    if kind == "image":
        if c.get("est"):
            out, info = htsvd.denoise(x, None, p, return_info=True)
            return {"out": out, "idx": info["idx"], "sigma": info["sigma"]}
        return htsvd.denoise(x, sigma, p)
    if kind == "batch":
        return htsvd.denoise_batch(x, sigma, p)
    if kind == "grad":
        out = htsvd.HtsvdFn.apply(x, st["w"], sigma, p)
        gx, gw = torch.autograd.grad(out, (x, st["w"]), st["gout"])
        return {"out": out.detach(), "grad_x": gx, "grad_w": gw}
    if kind == "video":
        return htsvd.denoise_video(x, sigma, p, T=c["T"])
    if kind == "cube":
        return htsvd.denoise_cube(x, sigma, p)
    if kind == "volume":
        return htsvd.denoise_volume(x, sigma, p)
    if kind == "sweep":
        return htsvd.denoise_tau_sweep(x, st["mults"], sigma, p)
    out, sigmas = htsvd.denoise_adaptive(x, (c["sub"], c["sub"]), p, return_sigmas=True)
    return {"out": out, "sigmas": sigmas}


# ---- what a pass cannot do without

def _image_work(H, W, C, c, frames=1, ps=8, D=None):
    """Bytes of one image's input and output; operations of matching (one multiply-add per pixel of a
    candidate), of one projection each way per distinct patch, and of the group transform both ways with
    its threshold."""
    ax = [n for n in (D, H, W) if n is not None]
    refs = math.prod((n - ps) // c["stride"] + 1 + ((n - ps) % c["stride"] != 0) for n in ax)
    pos = math.prod(n - ps + 1 for n in ax)
    win = math.prod(min(c["window"], n - ps + 1) for n in ax)
    planes = C if c["match"] == "full" or C not in (1, 3) else 1
    vals = ps * ps * (C if D is None else ps)
    cc = C if D is None else ps
    match = refs * win * frames * 2.0 * (vals if D is not None else ps * ps * planes)
    patch = 2.0 * vals * ps * (1 if cc == 1 else 2) * 2 + 2.0 * vals * cc
    group = c["K"] * vals * 5.0
    n = math.prod(ax) * (1 if D is not None else C)
    return dict(bytes=5.0 * n, flops=match + min(refs * c["K"], pos) * 2 * patch + refs * group)


def work(case):
    c = _full(case)
    kind = c["kind"]
    if kind == "batch":
        each = [_image_work(h, w, c["C"], c) for h, w, _ in _batch_shapes(c, 0)]
        return {k: sum(e[k] for e in each) for k in ("bytes", "flops")}
    if kind == "volume":
        return _image_work(c["H"], c["W"], 4, c, ps=4, D=c["D"])
    if kind == "video":
        near = sum(min(c["F"] - 1, t + c["T"]) - max(0, t - c["T"]) + 1 for t in range(c["F"]))
        one = _image_work(c["H"], c["W"], c["C"], c, frames=near / c["F"])
        return {k: c["F"] * v for k, v in one.items()}
    one = _image_work(c["H"], c["W"], c["C"], c)
    n = c["H"] * c["W"] * c["C"]
    if kind == "grad":                                  # float image and cotangent in; estimate and gradients out
        return dict(bytes=16.0 * n, flops=3.0 * one["flops"])
    if kind == "sweep":
        return dict(bytes=n * (1.0 + 4.0 * c["n"]), flops=c["n"] * one["flops"])
    return one


# ---- the same outputs in 64 bits, from the method's definition

def _bounds(n, part):
    t = max(1, n // part)
    return [((i * n) // t, ((i + 1) * n) // t) for i in range(t)]


def _grid(n, ps, s):
    v = list(range(0, n - ps + 1, s))
    return torch.tensor(v if v[-1] == n - ps else v + [n - ps], device=DEV)


def _starts(ref, n, ps, win):
    npos = n - ps + 1
    w = min(win, npos)
    return (ref - (win - 1) // 2).clamp(min=0).clamp(max=npos - w) if npos > win else torch.zeros_like(ref), w


class _Stack:
    """Patches of a stack of arrays [F, *extent, C] by linear position (frame-major)."""

    def __init__(self, x, ps, nd):
        self.ps, self.nd, self.C = ps, nd, x.shape[-1]
        self.ext = list(x.shape[1:1 + nd])
        self.stride = [math.prod(self.ext[d + 1:]) for d in range(nd)]
        self.flat = x.reshape(-1, self.C)
        off = torch.zeros(1, dtype=torch.int64, device=DEV)
        order = list(range(nd)) if nd == 2 else [1, 2, 0]   # volumes: rows y, columns x, tube z
        for d in order:
            off = (off[:, None] + torch.arange(ps, device=DEV) * self.stride[d]).reshape(-1)
        self.off = off

    def __call__(self, lin):
        """[..., ps, ps, tube] patches at linear positions."""
        g = self.flat[lin.unsqueeze(-1) + self.off]
        tube = self.C if self.nd == 2 else self.ps
        return g.reshape(*lin.shape, self.ps, self.ps, tube)

    def add(self, lin, vals, wts):
        num = torch.zeros(self.flat.shape, dtype=torch.float64, device=DEV)
        den = torch.zeros(self.flat.shape[0], dtype=torch.float64, device=DEV)
        pos = (lin.unsqueeze(-1) + self.off).reshape(-1)
        num = num.index_add(0, pos, vals.reshape(-1, self.C))
        den = den.index_add(0, pos, wts.unsqueeze(-1).expand(*lin.shape, self.off.numel()).reshape(-1))
        return num, den


def _references(c, ext, ps):
    ax = [_grid(n, ps, c["stride"]) for n in ext]
    mesh = torch.meshgrid(*ax, indexing="ij")
    return [m.reshape(-1) for m in mesh]


def _group(q, c, ps, nd, t=0, T=0):
    """Grouping of frame t of the quantised stack q [F, *extent, C]: global linear positions [N, K]."""
    F, ext, C, K = q.shape[0], list(q.shape[1:1 + nd]), q.shape[-1], c["K"]
    ref = _references(c, ext, ps)
    strd = [math.prod(ext[d + 1:]) for d in range(nd)]
    npix = math.prod(ext)
    me = t * npix + sum(r * s for r, s in zip(ref, strd))
    cand = torch.zeros(ref[0].numel(), 1, dtype=torch.int64, device=DEV)
    for d in range(nd):
        st, w = _starts(ref[d], ext[d], ps, c["window"])
        cand = (cand[:, :, None] + ((st[:, None] + torch.arange(w, device=DEV)) * strd[d])[:, None, :]).flatten(1)
    cand = torch.cat([cand + f * npix for f in range(max(0, t - T), min(F - 1, t + T) + 1)], dim=1)
    qi = q.to(torch.int16)
    match = c["match"] if C in (1, 3) and nd == 2 else "full"
    if nd == 3 or C == 1 or match == "full":
        which = [(qi, torch.ones_like(me, dtype=torch.bool))]
    elif match == "green":
        which = [(qi[..., 1:2], torch.ones_like(me, dtype=torch.bool))]
    else:
        e = _Stack(q.double(), ps, nd)(me).square().sum((1, 2))
        green = (1.2 * 1.2 * e[:, 1] >= e[:, 0]) & (1.2 * 1.2 * e[:, 1] >= e[:, 2])
        which = [(qi[..., 1:2], green), (qi.sum(-1, keepdim=True, dtype=torch.int16), ~green)]
    idx = torch.empty(me.numel(), K, dtype=torch.int64, device=DEV)
    for plane, sel in which:
        S = _Stack(plane.contiguous(), ps, nd)
        rows = sel.nonzero().flatten()
        step = max(1, (1 << 26) // (cand.shape[1] * S.off.numel() * S.C))
        for r in rows.split(step):
            d = S(cand[r]).flatten(2).int() - S(me[r]).flatten(1).int()[:, None]
            ssd = (d * d).sum(-1)
            key = (ssd << 32) | cand[r]
            key[cand[r] == me[r, None]] = torch.iinfo(torch.int64).max
            top = key.topk(K - 1, dim=1, largest=False, sorted=True).values
            idx[r] = torch.cat([me[r, None], top & 0xFFFFFFFF], dim=1)
    return idx


def _canonical(A):
    Q = torch.linalg.eigh(A.cpu()).eigenvectors.flip(-1)
    for k in range(Q.shape[-1]):
        m = Q[:, k].abs()
        a = int((m >= m.max() * (1 - 1e-6)).nonzero()[0])
        Q[:, k] = Q[:, k] * (Q[a, k].conj() / Q[a, k].abs())
    return Q.to(DEV)


def _bases(P):
    X = torch.fft.fft(P.double(), dim=-1)
    U, V = [], []
    for f in range(P.shape[-1] // 2 + 1):
        x = X[..., f]
        r, k = x.transpose(0, 1).flatten(1), x.permute(2, 0, 1).flatten(1)
        U.append(_canonical(r @ r.conj().T))
        V.append(_canonical(k.conj() @ k.T))
    return U, V


def _project(G, U, V, inverse):
    """U^T * G * V per patch (t-products along the last mode), or its inverse."""
    X = torch.fft.rfft(G, dim=-1)
    S = []
    for f in range(X.shape[-1]):
        x = X[..., f]
        u, v = (U[f], V[f].conj().T) if inverse else (U[f].conj().T, V[f])
        S.append(u @ x @ v)
    return torch.fft.irfft(torch.stack(S, dim=-1), n=G.shape[-1], dim=-1)


def _haar(K):
    H = torch.tensor([[1.0, 1.0], [1.0, -1.0]], dtype=torch.float64) / math.sqrt(2)
    while H.shape[0] < K:
        n = H.shape[0]
        H = torch.cat([torch.kron(H, torch.tensor([[1.0, 1.0]], dtype=torch.float64)),
                       torch.kron(torch.eye(n, dtype=torch.float64), torch.tensor([[1.0, -1.0]], dtype=torch.float64))])
        H /= math.sqrt(2)
    return H.to(DEV)


def _sigma(P):
    p = P.double().flatten(1)
    mu = p.mean(0)
    lam = torch.linalg.eigvalsh((p.T @ p / p.shape[0] - torch.outer(mu, mu)).cpu())
    best = 1
    for r in range(1, lam.numel() + 1):
        med = lam[(r - 1) // 2] if r % 2 else 0.5 * (lam[r // 2 - 1] + lam[r // 2])
        if lam[:r].mean() <= 1.02 * med:
            best = r
    return math.sqrt(max(float(lam[:best].mean()), 0.0))


def _prepared(q, c, ps, nd, t=0, T=0):
    """Grouping, bases and estimated noise level of frame t."""
    idx = _group(q, c, ps, nd, t, T)
    P = _Stack(q, ps, nd)(idx[:, 0])
    return idx, _bases(P), P


def _filter(x, idx, bases, tau, c, ps, nd, w=None, t=0):
    """Numerator / denominator of frame t of the stack x after thresholding every group at tau."""
    S, H = _Stack(x.double(), ps, nd), _haar(c["K"])
    npix = math.prod(S.ext)
    num = den = 0.0
    tube = S.C if nd == 2 else ps
    for lo in range(0, idx.shape[0], step := max(1, (1 << 27) // (c["K"] * ps * ps * tube))):
        i = idx[lo:lo + step]
        Y = torch.einsum("mk,nkabc->nmabc", H, _project(S(i), *bases, inverse=False))
        keep = (Y.detach().abs() >= tau).double()
        G = _project(torch.einsum("mk,nmabc->nkabc", H, Y * keep), *bases, inverse=True)
        wg = torch.ones(i.shape[0], dtype=torch.float64, device=DEV)
        if w is not None:
            wg = w[lo:lo + step]
        elif c["agg"] == "sparsity":
            wg = 1.0 / keep.sum((1, 2, 3, 4)).clamp(min=1.0)
        inside = ((i >= t * npix) & (i < (t + 1) * npix)).double() * wg[:, None]
        a, b = S.add(i, G * inside[:, :, None, None, None], inside)
        num, den = num + a, den + b
    sl = slice(t * npix, (t + 1) * npix)
    return (num[sl] / den[sl, None]).reshape(*S.ext, S.C)


def _mult(c, C, ps):
    return c["tau_mult"] if c["tau_mult"] > 0 else math.sqrt(2 * math.log(C * c["K"] * ps * ps))


def _denoised(q, c, sigma, ps=8, nd=2, t=0, T=0):
    idx, bases, P = _prepared(q, c, ps, nd, t, T)
    sg = _sigma(P) if sigma is None else sigma
    tau = _mult(c, q.shape[-1] if nd == 2 else ps, ps) * sg
    return _filter(q, idx, bases, tau, c, ps, nd, t=t), idx, sg


def exact(case, seed):
    c = _full(case)
    st = prepare(case, seed)
    x, kind, sigma = st["x"], c["kind"], st["sigma"]
    if kind == "image":
        out, idx, sg = _denoised(x[None], c, sigma)
        return {"out": out, "idx": idx.int(), "sigma": sg} if c.get("est") else out
    if kind == "batch":
        return [_denoised(y[None], c, s)[0] for y, s in zip(x, sigma)]
    if kind == "grad":
        xd = x.detach().double().requires_grad_(True)
        wd = st["w"].detach().double().requires_grad_(True)
        q = x.detach().round().clamp(0, 255).to(torch.uint8)
        idx, bases, _ = _prepared(q[None], c, 8, 2)
        out = _filter(xd[None], idx, bases, _mult(c, c["C"], 8) * sigma, c, 8, 2, w=wd)
        gx, gw = torch.autograd.grad(out, (xd, wd), st["gout"].double())
        return {"out": out.detach(), "grad_x": gx, "grad_w": gw}
    if kind == "video":
        return torch.stack([_denoised(x, c, sigma, t=t, T=c["T"])[0] for t in range(c["F"])])
    if kind == "cube":
        return _denoised(x[None], c, sigma)[0]
    if kind == "volume":
        return _denoised(x[None, ..., None], c, sigma, ps=4, nd=3)[0].squeeze(-1)
    if kind == "sweep":
        idx, bases, _ = _prepared(x[None], c, 8, 2)
        return torch.stack([_filter(x[None], idx, bases, m * sigma, c, 8, 2) for m in st["mults"]])
    out = torch.empty(x.shape, dtype=torch.float64, device=DEV)
    sigmas = []
    for y0, y1 in _bounds(c["H"], c["sub"]):
        for x0, x1 in _bounds(c["W"], c["sub"]):
            o, _, sg = _denoised(x[None, y0:y1, x0:x1].contiguous(), c, None)
            out[y0:y1, x0:x1] = o
            sigmas.append(sg)
    return {"out": out, "sigmas": sigmas}
