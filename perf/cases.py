"""What a user of this library has it do: the workloads that its speed is measured on.

Every case is one whole call of a public entry point on inputs that are on the
GPU (or, where the case says so, in host arrays). Solves run a fixed number of
iterations under the stop rule that the workload really uses, with a tolerance
that is not met that early, so that two runs do the same work: the stop rule
is evaluated as in earnest. Sizes are the repository's own workloads (64^2
reference problem, 512^2 inpainting batch, 1024^2 and 2048^2 frame images, the
uneven batch, the 256^2 comparison with the Reeves-Sorel variants, the
warm-start network at 16 x 512^2 and 16 x 256^2), with shorter iteration
counts, and odd image sizes between them.
"""
from __future__ import annotations

import math
import os

import numpy as np
import torch

import paper_1210_2687_gb300 as ad

POW2 = (64, 128, 256, 512, 1024, 2048)
SIDES = tuple(n for n in range(64, 2049, 32)
              if (n & -n) >= 32 and n // (n & -n) in (1, 3, 5))   # sides solved exactly
CG = ("tv_cg", "haar_cg")
L2_BYTES = 129e6
WEIGHTS = os.path.join(os.path.dirname(os.path.abspath(ad.__file__)), "weights", "warmstart_tv.npz")


def _solve(name, **kw):
    c = {"kind": "solve", "H": 512, "W": 512, "count": 1, "reg": "tv", "levels": 4, "blur": "box", "side": 9,
         "missing": 0.0, "lam": 1e-3, "mu1": 0.0, "mu2": 0.0, "stop": "iters", "check": 1, "iters": 50, "host": False}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the reference problem: one small image, latency of the whole call
        _solve("tv_64", H=64, W=64, side=9, lam=1e-3, mu1=1.0, mu2=1e-2, iters=200),
        # the paper's setting: one 256^2 image, 19 x 19 blur, its objective rule every iteration
        _solve("tv_256_paper", H=256, W=256, side=19, lam=2e-4, stop="rel_obj", iters=80),
        # the headline workload: a batch of 512^2 images with 40 % missing pixels, rel-x rule
        _solve("tv_512_batch", count=64, blur="gauss", side=19, missing=0.4, lam=1e-5, stop="rel_x", check=10,
               iters=60),
        # one large photograph
        _solve("tv_2048", H=2048, W=2048, side=13, lam=5e-5, iters=40),
        # a size that is not a power of two, solved on its own domain
        _solve("tv_384_batch", H=384, W=384, count=16, blur="motion", side=15, missing=0.25, lam=3e-5, stop="rel_x",
               check=10, iters=60),
        # odd image sizes in host memory, padded to the next domain: copies in and out count
        _solve("tv_ragged_host", H=300, W=451, count=8, blur="motion", side=11, missing=0.3, lam=1e-4, stop="rel_x",
               check=10, iters=40, host=True),
        # the variant that mask decoupling is compared with
        _solve("tv_cg_256", H=256, W=256, count=8, reg="tv_cg", side=19, lam=2e-4, stop="rel_obj", iters=40),
        # the frame prior on one image
        _solve("haar_1024", H=1024, W=1024, reg="haar", side=13, lam=5e-5, iters=50),
        _solve("haar_2048", H=2048, W=2048, reg="haar", side=13, lam=5e-5, iters=40),
        # images of every size, both priors, solved in one call
        {"name": "uneven_batch", "kind": "uneven", "count": 20, "largest": 1024, "iters": 40},
        # the learned start of 16 images, and one training batch's loss and gradients
        {"name": "cnn_predict", "kind": "predict", "count": 16, "H": 512, "W": 512},
        {"name": "cnn_gradients", "kind": "gradients", "count": 16, "H": 256, "W": 256},
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choices(("solve", "uneven", "predict", "gradients"), (7, 1, 1, 1))[0]
    if kind == "uneven":
        return {"kind": kind, "count": rng.randint(5, 24), "largest": rng.choice((256, 384, 512, 1024)),
                "iters": rng.randint(20, 40)}
    if kind in ("predict", "gradients"):
        H, W = (16 * rng.randint(4, 40) for _ in range(2))
        most = (16 << 18 if kind == "predict" else 16 << 16) // (H * W)
        return {"kind": kind, "count": max(1, min(16, rng.randint(1, max(1, most)))), "H": H, "W": W}
    reg = rng.choice(("tv", "tv", "tv", "haar", "haar", "tv_aniso", "haar_ll_free", "haar_synthesis") + CG)
    host = rng.random() < 0.2
    size = _log_uniform(rng, 64, 2048)
    H, W = (min(2048.0, max(64.0, size * rng.uniform(0.7, 1.4))) for _ in range(2))
    if host:
        H, W = int(H), int(W)
    else:
        sides = POW2 if reg in CG or rng.random() < 0.6 else SIDES
        H, W = (min(sides, key=lambda n: abs(math.log(n / v))) for v in (H, W))
    iters = rng.randint(20, 60)
    per = _domain(H, reg, host) * _domain(W, reg, host) * (67 if reg.startswith("tv") else 155)
    most = max(1, min(96, int(2e10 / (per * iters))))
    count = max(1, int(_log_uniform(rng, 1, most + 0.99)))
    iters = max(5, min(iters, int(2e10 / (per * count))))
    blur = rng.choice(("box", "gauss", "motion"))
    stop, check = rng.choice((("iters", 1), ("rel_x", 10), ("rel_x", 1), ("rel_obj", 1)))
    lam = {"tv": 1e-4, "haar": 1e-4}.get(reg.split("_")[0]) * _log_uniform(rng, 0.5, 10)
    return _solve(None, H=H, W=W, count=count, reg=reg, levels=rng.choice((4, 4, 4, 3, 2)), blur=blur,
                  side=2 * rng.randint(2, 10) + 1, missing=rng.choice((0.0, round(rng.uniform(0.0, 0.5), 3))), lam=lam,
                  stop=stop, check=check, iters=iters, host=host)


# ---- inputs ---------------------------------------------------------------------------------------------------
def _domain(n, reg, pad):
    """The side that an n-pixel side is solved on."""
    return n if not pad else min(m for m in (POW2 if reg in CG else SIDES) if m >= n)


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float32)


def _images(g, count, H, W):
    """Piecewise-constant images (20 rectangles and disks) plus smooth four-octave texture, in [0, 1]."""
    rr = torch.arange(H, device="cuda", dtype=torch.float32).view(1, H, 1)
    cc = torch.arange(W, device="cuda", dtype=torch.float32).view(1, 1, W)
    img = _rand(g, count, 1, 1).expand(count, H, W).clone()
    for _ in range(20):
        p = _rand(g, count, 6).view(count, 6, 1, 1)
        r0, r1 = torch.minimum(p[:, 0], p[:, 1]) * H, torch.maximum(p[:, 0], p[:, 1]) * H
        c0, c1 = torch.minimum(p[:, 2], p[:, 3]) * W, torch.maximum(p[:, 2], p[:, 3]) * W
        rect = (rr >= r0) & (rr <= r1) & (cc >= c0) & (cc <= c1)
        rad = 2 + p[:, 1] * (min(H, W) / 4 - 2)
        disk = (rr - p[:, 0] * H) ** 2 + (cc - p[:, 2] * W) ** 2 <= rad * rad
        img = torch.where(torch.where(p[:, 4] < 0.5, rect, disk), p[:, 5], img)
    tex, amp, tot = 0.0, 1.0, 0.0
    for period in (64, 32, 16, 8):
        lat = _rand(g, count, 1, H // period + 2, W // period + 2)
        t = torch.nn.functional.interpolate(lat, size=(H, W), mode="bilinear", align_corners=True)
        tex, amp, tot = tex + amp * t[:, 0], amp / 2, tot + amp
    return (0.6 * img + 0.4 * tex / tot).clamp(0, 1)


def _kernel(blur, side, seed):
    """A unit-sum blur kernel of an odd side."""
    h = side // 2
    t = np.arange(-h, h + 1, dtype=np.float64)
    if blur == "gauss":
        k = np.exp(-(t[:, None] ** 2 + t[None, :] ** 2) / (2 * (side / 6.0) ** 2))
    elif blur == "motion":
        a, s = math.radians(15 + 37 * (seed % 5)), np.linspace(-h, h, 64 * side)
        k = np.maximum(0, 1 - abs(t[:, None, None] + s * math.sin(a))) * np.maximum(0, 1 - abs(t[None, :, None] - s * math.cos(a)))
        k = k.sum(-1)
    else:
        k = np.ones((side, side))
    return (k / k.sum()).astype(np.float32)


def _spectrum(k, H, W):
    """DFT of the kernel placed with its centre at (0, 0) of an H x W domain (half spectrum, float64)."""
    a = torch.zeros(H, W, dtype=torch.float64, device="cuda")
    h, w = k.shape[0] // 2, k.shape[1] // 2
    r, c = (torch.arange(-h, h + 1) % H).cuda(), (torch.arange(-w, w + 1) % W).cuda()
    a[r[:, None], c[None, :]] = torch.from_numpy(k).double().cuda()
    return torch.fft.rfft2(a)


def _valid(H, W, k):
    m = torch.zeros(H, W, dtype=torch.bool, device="cuda")
    h, w = k.shape[0] // 2, k.shape[1] // 2
    m[h:H - h, w:W - w] = True
    return m


def _observe(g, count, H, W, k, missing):
    """Images, their observations at BSNR 40 dB (float32, 0 where unobserved) and masks (uint8)."""
    x = _images(g, count, H, W)
    y = torch.fft.irfft2(torch.fft.rfft2(x) * _spectrum(k, H, W).to(torch.complex64), s=(H, W))
    m = _valid(H, W, k) & (_rand(g, count, H, W) >= missing)
    n = m.sum((1, 2), keepdim=True).clamp(min=1)
    mean = (y * m).sum((1, 2), keepdim=True) / n
    sigma = (((y - mean) ** 2 * m).sum((1, 2), keepdim=True) / n / 1e4).sqrt()
    y = y + sigma * torch.randn(count, H, W, generator=g, device="cuda")
    return x, torch.where(m, y, 0.0).contiguous(), m.to(torch.uint8).contiguous()


def _penalties(case):
    """(lambda, mu1, mu2) as the float32 values that the plan is given."""
    lam = np.float32(case["lam"])
    mu2 = np.float32(case["mu2"]) if case["mu2"] > 0 else np.float32(10 * lam)
    mu1 = np.float32(case["mu1"]) if case["mu1"] > 0 else np.float32(min(1.0, 3 * mu2))
    return float(lam), float(mu1), float(mu2)


def _parts(case):
    """The cases of equal problems that an uneven batch is made of: five sizes, both priors, three kernel families."""
    sides = [s for s in (128, 256, 384, 512, 1024) if s <= case["largest"]]
    out = []
    for i in range(case["count"]):
        n, reg = sides[i % len(sides)], ("tv", "haar")[(i // len(sides)) % 2]
        blur = ("box", "gauss", "motion")[i % 3]
        out.append(_solve(None, H=n, W=n, reg=reg, blur=blur, side=(13, 17, 15)[i % 3], missing=0.1 * (i % 6),
                          lam=1e-4 if reg == "haar" else 3e-5, stop="rel_x", check=10, iters=case["iters"]))
    return out


def _problems(case, seed):
    """[(case of one group, its kernel, ybar, mask)] of a solve."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    out = []
    for j, c in enumerate(_parts(case) if case["kind"] == "uneven" else [case]):
        k = _kernel(c["blur"], c["side"], seed + j)
        _, y, m = _observe(g, c["count"], c["H"], c["W"], k, c["missing"])
        out.append((c, k, y, m))
    return out


def _net_inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    x, y, m = _observe(g, case["count"], case["H"], case["W"], _kernel("box", 9, seed), 0.25)
    return x, y, m, g


def _targets(x, g):
    """Training targets (image and three dual channels of order one)."""
    d = 0.3 * torch.randn(*x.shape, 3, generator=g, device="cuda")
    return torch.cat([x[..., None], d], dim=-1).contiguous()


# ---- the calls ------------------------------------------------------------------------------------------------
def prepare(case, seed):
    torch.cuda.init()
    if case["kind"] in ("predict", "gradients"):
        x, y, m, g = _net_inputs(case, seed)
        w = np.load(WEIGHTS)
        n, H, W = y.shape
        net = ad.Cnn(n * H * W, training=case["kind"] == "gradients")
        net.set_params(w["params"])
        s = {"kind": case["kind"], "net": net, "y": y, "m": m}
        if case["kind"] == "predict":
            s.update(scales=[float(v) for v in w["scales"]], x0=torch.empty(n, H, W, device="cuda"),
                     d0=torch.empty(n, 3 * H * W, device="cuda"))
        else:
            s.update(target=_targets(x, g), grads=torch.empty(net.param_count(), device="cuda"))
        return s
    s = {"kind": "solve", "plans": [], "y": [], "m": [], "x": [], "out": []}
    for c, k, y, m in _problems(case, seed):
        lam, mu1, mu2 = _penalties(c)
        x = torch.zeros_like(y)
        if c["host"]:
            y, m, x = (v.cpu().numpy() for v in (y, m, x))
        for i in range(c["count"]):
            s["plans"].append(ad.Plan(c["H"], c["W"], k, lam, mu1, mu2, c["reg"], levels=c["levels"], stop=c["stop"],
                                      max_iters=c["iters"], check_every=c["check"], pad=c["host"]))
            s["y"].append(y[i])
            s["m"].append(m[i])
            s["x"].append(x[i])
        s["out"].append(x)
    return s


def run(state):
    s = state
    if s["kind"] == "predict":
        s["net"].predict_start(s["y"], s["m"], s["scales"], s["x0"], s["d0"])
        return {"x0": s["x0"], "d0": s["d0"]}
    if s["kind"] == "gradients":
        loss = s["net"].gradients(s["y"], s["m"], s["target"], (1.0, 1.0, 1.0, 1.0), s["grads"])
        return {"loss": loss, "grads": s["grads"]}
    if len(s["plans"]) == 1:
        res = [ad.solve(s["plans"][0], s["y"][0], s["m"][0], s["x"][0])]
    else:
        res = ad.solve_batch(s["plans"], s["y"], s["m"], s["x"])
    return {"x": s["out"], "iters": np.array([r.iters for r in res], np.int32),
            "objective": np.array([r.objective for r in res], np.float32)}


def work(case):
    if case["kind"] in ("predict", "gradients"):
        px = case["count"] * case["H"] * case["W"]
        flops = 2 * 9 * (2 * 32 + 6 * 32 * 32 + 32 * 4)
        if case["kind"] == "predict":
            return {"bytes": px * (4 + 1 + 16), "flops": px * flops}
        return {"bytes": px * (4 + 1 + 16), "flops": px * (3 * flops - 2 * 9 * 2 * 32)}
    total = {"bytes": 0.0, "flops": 0.0}
    state = 0.0
    parts = _parts(case) if case["kind"] == "uneven" else [case]
    for c in parts:
        H, W = _domain(c["H"], c["reg"], c["host"]), _domain(c["W"], c["reg"], c["host"])
        n, tv = c["count"] * H * W, c["reg"].startswith("tv")
        nb = 2 if tv else 3 * c["levels"] + 1
        state += n * (4 * nb + 4 + 4 + 6 + 8)      # duals, M^T y, spectra, one complex field
    for c in parts:
        H, W = _domain(c["H"], c["reg"], c["host"]), _domain(c["W"], c["reg"], c["host"])
        n, tv = c["count"] * H * W, c["reg"].startswith("tv")
        nb = 2 if tv else 3 * c["levels"] + 1
        io = c["count"] * c["H"] * c["W"] * 9      # y, mask and x once
        # state that does not stay on the chip goes through memory once per iteration: duals in and
        # out, M^T y and mask, spectra, the complex field between the row and column transforms
        it = n * (8 * nb + 8 + 5 + 6 + 32) if state > L2_BYTES else 0
        per = 10 * math.log2(H * W) + (60 if tv else 30 + 16 * nb)
        if c["reg"] in CG:
            it, per = it + (n * (32 + 6) if it else 0), per + 10 * math.log2(H * W) + 20
        total["bytes"] += io + it * c["iters"]
        total["flops"] += n * per * c["iters"]
    return total


# ---- the same in 64 bits --------------------------------------------------------------------------------------
def _soft(v, t):
    return torch.sign(v) * (v.abs() - t).clamp(min=0)


def _analysis(x, levels):
    out, a = [], x
    for j in range(levels):
        s = 1 << j
        r = torch.roll(a, -s, -1)
        lo, hi = (a + r) / 2, (a - r) / 2
        rl, rh = torch.roll(lo, -s, -2), torch.roll(hi, -s, -2)
        out += [(hi + rh) / 2, (lo - rl) / 2, (hi - rh) / 2]
        a = (lo + rl) / 2
    return out + [a]


def _synthesis(c, levels):
    a = c[3 * levels]
    for j in reversed(range(levels)):
        s = 1 << j
        up = lambda v: torch.roll(v, s, -2)  # noqa: E731
        b0, b1, b2 = c[3 * j:3 * j + 3]
        lo = (a + up(a) + b1 - up(b1)) / 2
        hi = (b0 + up(b0) + b2 - up(b2)) / 2
        a = (lo + torch.roll(lo, s, -1) + hi - torch.roll(hi, s, -1)) / 2
    return a


def _iterate(c, k, y, m):
    """x and the objective after the case's iterations from u0 = d0 = 0, in float64, for equal problems."""
    lam, mu1, mu2 = _penalties(c)
    reg, L = c["reg"], c["levels"]
    tv, cg = reg.startswith("tv"), reg in CG
    H0, W0 = c["H"], c["W"]
    H, W = _domain(H0, reg, c["host"]), _domain(W0, reg, c["host"])
    yb = torch.zeros(y.shape[0], H, W, dtype=torch.float64, device="cuda")
    ob = torch.zeros(y.shape[0], H, W, dtype=torch.bool, device="cuda")
    ob[:, :H0, :W0] = (m != 0) & _valid(H0, W0, k)
    yb[:, :H0, :W0] = y.double()
    yb *= ob
    lm, gam, tau = _spectrum(k, H, W), mu2 / mu1, lam / mu2
    F, Fi = torch.fft.rfft2, lambda v: torch.fft.irfft2(v, s=(H, W))  # noqa: E731
    fr = lambda n, full: 4 * torch.sin(math.pi * torch.arange(n if full else n // 2 + 1, device="cuda", dtype=torch.float64) / n) ** 2  # noqa: E731
    den = lm.abs() ** 2 + gam * ((fr(H, True)[:, None] + fr(W, False)[None, :]) if tv else 1.0)
    Dh, Dv = lambda v: torch.roll(v, -1, -1) - v, lambda v: torch.roll(v, -1, -2) - v  # noqa: E731
    zero = torch.zeros_like(yb)
    u1, d1, xi, x = zero, zero, zero, zero
    nb = 2 if tv else 3 * L + 1
    u2, d2 = [zero] * nb, [zero] * nb
    dot = lambda a, b: (a * b).sum((1, 2), keepdim=True)  # noqa: E731
    for _ in range(c["iters"]):
        z1, z2 = u1 + d1, [a + b for a, b in zip(u2, d2)]
        if tv:
            w = gam * (torch.roll(z2[0], 1, -1) - z2[0] + torch.roll(z2[1], 1, -2) - z2[1])
        else:
            pz = _synthesis(z2, L)
            w = gam * pz
        r = F(z1) * lm.conj() + F(w)
        if cg:
            S = lambda v: torch.where(ob, 0.0, Fi(lm * lm.conj() * F(v) / den) - v)  # noqa: E731
            p = torch.where(ob, 0.0, Fi(lm * r / den)) - S(xi)
            rr, q = dot(p, p), dot(p, S(p))
            xi = xi + torch.where(rr > 0, rr / torch.where(q == 0, 1.0, q), 0.0) * p
            r = r - lm.conj() * F(xi)
        X = r / den
        x, ax = Fi(X), Fi(lm * X)
        if cg:
            ax = torch.where(ob, ax, 0.0)
            u1 = torch.where(ob, (yb + mu1 * (ax - d1)) / (1 + mu1), 0.0)
        else:
            u1 = (yb + mu1 * (ax - d1)) / (ob + mu1)
        d1 = d1 - (ax - u1)
        if tv:
            v = [Dh(x), Dv(x)]
        else:
            v = _analysis(x - pz, L) if reg == "haar_synthesis" else _analysis(x, L)
            if reg == "haar_synthesis":
                v = [a + b for a, b in zip(v, z2)]
        s = [a - b for a, b in zip(v, d2)]
        if reg in ("tv", "tv_cg"):
            n = torch.sqrt(s[0] ** 2 + s[1] ** 2)
            f = torch.where(n > tau, (n - tau) / torch.where(n > 0, n, 1.0), 0.0)
            u2 = [f * s[0], f * s[1]]
        else:
            u2 = [_soft(a, tau) for a in s]
            if reg == "haar_ll_free":
                u2[-1] = s[-1]
        d2 = [a - b for a, b in zip(u2, s)]
    if reg in ("tv", "tv_cg"):
        pen = torch.sqrt(v[0] ** 2 + v[1] ** 2).sum((1, 2))
    else:
        pen = sum(a.abs().sum((1, 2)) for a in (v[:-1] if reg == "haar_ll_free" else v))
    obj = 0.5 * ((ob * (yb - ax)) ** 2).sum((1, 2)) + lam * pen
    return x[:, :H0, :W0].contiguous(), obj


class _Stored(torch.autograd.Function):
    """A value that the network stores in BF16, and so its gradient where `both`; the arithmetic is in 64 bits."""

    @staticmethod
    def forward(ctx, v, both):
        ctx.both = both
        return v.to(torch.bfloat16).double()

    @staticmethod
    def backward(ctx, g):
        return (g.to(torch.bfloat16).double() if ctx.both else g), None


def _network(params, y, m):
    """The network's output (count, 4, H, W): weights and activations are BF16 by its definition."""
    a, o = torch.stack([torch.where(m != 0, y, 0.0).double(), (m != 0).double()], 1), 0
    a = a.to(torch.bfloat16).double()
    for l in range(8):
        ci, co = 2 if l == 0 else 32, 4 if l == 7 else 32
        w, o = _Stored.apply(params[o:o + co * ci * 9].view(co, ci, 3, 3), False), o + co * ci * 9
        b, o = params[o:o + co], o + co
        z, p = b.view(1, co, 1, 1), torch.nn.functional.pad(a, (1, 1, 1, 1))
        for t in range(9):
            sh = p[:, :, t // 3:t // 3 + y.shape[1], t % 3:t % 3 + y.shape[2]]
            z = z + torch.einsum("oi,nihw->nohw", w[:, :, t // 3, t % 3], sh)
        a = _Stored.apply(torch.relu(z), True) if l < 7 else z
    return a


def exact(case, seed):
    if case["kind"] in ("predict", "gradients"):
        x, y, m, g = _net_inputs(case, seed)
        wts = np.load(WEIGHTS)
        params = torch.from_numpy(wts["params"]).double().cuda()
        n, H, W = y.shape
        if case["kind"] == "predict":
            s = [float(np.float32(v)) for v in wts["scales"]]
            x0 = torch.empty(n, H, W, dtype=torch.float64, device="cuda")
            d0 = torch.empty(n, 3 * H * W, dtype=torch.float64, device="cuda")
            for i in range(n):
                o = _network(params, y[i:i + 1], m[i:i + 1])[0]
                x0[i] = s[0] * o[0]
                d0[i] = torch.cat([s[1] * o[1].reshape(-1), s[2] * o[2:4].permute(1, 2, 0).reshape(-1)])
            return {"x0": x0, "d0": d0}
        target = _targets(x, g).double()
        params.requires_grad_(True)
        total = 0.0
        for i in range(n):
            o = _network(params, y[i:i + 1], m[i:i + 1])[0].permute(1, 2, 0)
            e = (o - target[i]).detach()
            o.backward((2 * e / (n * H * W)).to(torch.bfloat16).double())
            total += float((e ** 2).sum() / (n * H * W))
        return {"loss": total, "grads": params.grad}
    xs, objs, iters = [], [], 0
    for c, k, y, m in _problems(case, seed):
        x, obj = _iterate(c, k, y, m)
        xs.append(x)
        objs.append(obj)
    return {"x": xs, "iters": None, "objective": torch.cat(objs)}
