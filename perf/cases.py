"""Performance cases of the MLBA deblurring library.

Each case is a piece of work a program hands to the library through its Python
binding: a restoration of one image (``Context``: new data in, a few
iterations, the restored image out), a batch of images restored together
(``Batch``), or one operator applied to device tensors (A and its adjoint, the
spectral preconditioner, one framelet step).  Sizes, PSFs, boundary
conditions and algorithms are those of the repository's benchmark workloads
and of the paper's experiments; ``draw`` spreads the same kinds over the whole
range of sizes and options.

Inputs are synthetic observations g = A f + eta of piecewise-smooth images,
made on the GPU from the seed.  ``exact`` is a plain FP64 torch restatement
of the definitions (FFT convolutions with zero padding, dense cosine /
antireflective bases, gathers and scatter-adds for the framelets).
"""
import math

import numpy as np
import torch

import paper_1504_07234_gb300 as mlba

MU = 10.0 / 255.0
SIZES = (128, 192, 256, 384, 512, 768, 1024)      # image sizes of the batch workload


# ---------------------------------------------------------------------------
# the cases

def _restore(name, n, psf, p, size, bc, precond, levels, iters, dtype="f32", z_store="f32",
             alpha=0.05, angle=0.0, nu=0.01, transform="auto", formulation="synthesis",
             blur_path="direct"):
    c = dict(kind="restore", n=n, psf=psf, p=p, size=size, angle=angle, nu=nu, bc=bc,
             precond=precond, levels=levels, iters=iters, dtype=dtype,
             z_store="f64" if dtype == "f64" else z_store, alpha=alpha, transform=transform,
             formulation=formulation, blur_path=blur_path)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the plain FP64 workload: a thumbnail-sized image, rectangular A,
        # Algorithm 1; launches and latency are all of it
        _restore("rect64_f64", 64, "gauss", 9, 2.0, "rect", "bccb", 1, 20, dtype="f64", alpha=0.3,
                 transform="dft"),
        # one small image, reflective BCs, nonstationary Algorithm 4-NS (DCT)
        _restore("reflective256_ns", 256, "disk", 15, 6.0, "reflective", "tikh_ns", 2, 20, nu=0.02,
                 transform="dct"),
        # the paper's Example 4: 226 x 226 field of view, antireflective BCs
        # (antireflective transform), 31 x 31 Gaussian, four framelet levels
        _restore("antireflective226_l4", 226, "gauss", 31, 2.5, "antireflective", "tikh", 4, 15,
                 nu=0.02),
        # the paper's Example 1 setting in its own precision: 256 x 256, zero
        # BCs, Algorithm 3, four levels, FP64
        _restore("zero256_f64_l4", 256, "disk", 17, 7.0, "zero", "sym", 4, 6, dtype="f64", alpha=0.3),
        # a megapixel image, motion blur, Algorithm 1, Bregman variable in BF16
        # (the first two iterations: rounding z to 8 bits makes later iterates
        # depend on the last bit of every sum before it)
        _restore("rect1024_bf16", 1024, "motion", 21, 21.0, "rect", "bccb", 2, 2, z_store="bf16",
                 alpha=0.5, angle=0.9),
        # the same image with the Krylov preconditioner (Algorithm 2)
        _restore("rect1024_krylov", 1024, "motion", 21, 21.0, "rect", "krylov", 2, 3, angle=0.9),
        # 64 images of mixed size, PSF, BC and algorithm advanced together:
        # the throughput workload
        dict(name="batch64", kind="batch", count=64, spec=4, lo=128, hi=1024, iters=8, levels=2,
             z_store="f32"),
        # a large image, 31 x 31 Gaussian, nonstationary alpha_n, two levels ...
        _restore("rect4096_ns", 4096, "gauss", 31, 5.0, "rect", "tikh_ns", 2, 4, transform="dct"),
        # ... and with the paper's four levels
        _restore("rect4096_ns_l4", 4096, "gauss", 31, 5.0, "rect", "tikh_ns", 4, 4, transform="dct"),
        # A f and A^T t on device tensors: the operators of a caller's own loop,
        # odd size, general PSF
        dict(name="blur1499", kind="blur", n=1499, psf="disk", p=19, size=8.0, angle=0.0,
             bc="reflective", dtype="f32", blur_path="direct"),
        # C^T (C C^T + alpha I)^{-1} r on a device tensor
        dict(name="precond1000", kind="precond", n=1000, psf="motion", p=15, size=15.0, angle=0.4,
             transform="dft", which="tikh", alpha=0.05, dtype="f32"),
        # one framelet step on the caller's z (band-major planes), odd size
        dict(name="frame751", kind="frame", n=751, levels=2, dtype="f32", z_store="f32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _largest_prime(n):
    big, f = 1, 2
    while f * f <= n:
        while n % f == 0:
            big, n = f, n // f
        f += 1
    return max(big, n) if n > 1 else big


def _draw_n(rng, lo, hi, dtype):
    """Any size (odd ones too); large ones without a large prime factor, whose
    direct-sum transform passes would cost more than the largest listed case."""
    n = _log_int(rng, lo, hi)
    while (n > 300 and _largest_prime(n) > 31) if dtype == "f32" else _largest_prime(n) > 13:
        n += 1
    return n


def _draw_psf(rng):
    fam = rng.choice(("gauss", "disk", "motion"))
    if fam == "gauss":
        s = round(rng.uniform(1.0, 5.0), 3)
        return fam, 2 * int(math.ceil(3.0 * s)) + 1, s, 0.0
    if fam == "disk":
        r = rng.randint(2, 8)
        return fam, 2 * r + 3, float(r), 0.0
    k = rng.randrange(5, 22, 2)
    return fam, k, float(k), round(rng.uniform(0.0, math.pi), 3)


def draw(rng):
    kind = rng.choice(("restore",) * 5 + ("batch", "batch", "blur", "precond", "frame"))
    psf, p, size, angle = _draw_psf(rng)
    dtype = rng.choice(("f32", "f32", "f32", "f64"))
    hi = 300 if dtype == "f64" else 1600
    if kind == "batch":
        zs = rng.choice(("f32", "f32", "bf16"))
        return dict(kind="batch", count=rng.randint(2, 48), spec=rng.randrange(1 << 20),
                    lo=rng.choice((64, 100, 128)), hi=_log_int(rng, 160, 800),
                    iters=2 if zs == "bf16" else rng.randint(3, 6), levels=rng.choice((1, 2, 2, 3)), z_store=zs)
    if kind == "blur":
        return dict(kind="blur", n=_draw_n(rng, 64, hi, dtype), psf=psf, p=p, size=size, angle=angle,
                    bc=rng.choice(("zero", "periodic", "reflective", "rect", "antireflective")),
                    dtype=dtype, blur_path=rng.choice(("direct", "direct", "fft")))
    if kind == "precond":
        tr = "dft" if psf == "motion" else rng.choice(("dft", "dct"))
        return dict(kind="precond", n=_draw_n(rng, 64, hi, dtype), psf=psf, p=p, size=size, angle=angle,
                    transform=tr, which=rng.choice(("inv", "tikh")),
                    alpha=round(rng.uniform(0.01, 0.5), 4), dtype=dtype)
    if kind == "frame":
        return dict(kind="frame", n=_log_int(rng, 48, hi), levels=rng.choice((1, 2, 2, 3, 4)), dtype=dtype,
                    z_store="f64" if dtype == "f64" else rng.choice(("f32", "bf16")))
    bc = rng.choice(("zero", "periodic", "reflective", "rect", "rect", "antireflective"))
    if bc == "rect":
        precond, alpha = rng.choice((("bccb", 0.5), ("krylov", 0.05), ("sym", 0.5)))
    elif bc == "periodic":
        precond, alpha = rng.choice((("tikh_ns", 0.05), ("bccb", 0.05), ("tikh", 0.05)))
    elif psf == "motion":
        precond, alpha = "sym", 0.3
    elif bc == "antireflective":
        precond, alpha = rng.choice((("tikh", 0.05), ("sym", 0.3)))
    else:
        precond, alpha = rng.choice((("tikh_ns", 0.05), ("tikh", 0.05), ("sym", 0.3), ("krylov", 0.05)))
    n = _draw_n(rng, 64, min(hi, 500) if bc == "antireflective" else hi, dtype)
    most = 5 if dtype == "f64" or precond == "krylov" else 8 if n > 700 else 16
    form, path = "synthesis", "direct"
    if precond != "krylov":
        form = rng.choice(("synthesis",) * 7 + ("balanced",))
        path = rng.choice(("direct",) * 7 + ("fft",))
    zs = rng.choice(("f32", "f32", "bf16"))
    return _restore(None, n, psf, p, size, bc, precond, rng.choice((1, 2, 2, 4)),
                    2 if zs == "bf16" and dtype == "f32" else rng.randint(2, most), dtype=dtype,
                    z_store=zs, alpha=alpha, angle=angle,
                    nu=round(rng.uniform(0.005, 0.03), 4), formulation=form, blur_path=path)


# ---------------------------------------------------------------------------
# inputs

def _psf(fam, p, size, angle):
    c = (p - 1) // 2
    t = np.arange(p, dtype=np.float64) - c
    if fam == "gauss":
        g = np.exp(-(t * t) / (2.0 * size * size))
        g /= g.sum()
        return np.outer(g, g)
    if fam == "disk":
        h = ((t[:, None] ** 2 + t[None, :] ** 2) <= size * size).astype(np.float64)
        return h / h.sum()
    # motion: samples of a centred segment, splatted bilinearly
    h = np.zeros((p, p))
    length = int(size)
    for s in np.linspace(-(length - 1) / 2.0, (length - 1) / 2.0, 4 * length):
        y, x = c + s * math.sin(angle), c + s * math.cos(angle)
        y0, x0 = int(math.floor(y)), int(math.floor(x))
        for dy in (0, 1):
            for dx in (0, 1):
                w = (1 - abs(y - y0 - dy)) * (1 - abs(x - x0 - dx))
                if 0 <= y0 + dy < p and 0 <= x0 + dx < p:
                    h[y0 + dy, x0 + dx] += w
    return h / h.sum()


def _dtype(case):
    return torch.float64 if case["dtype"] == "f64" else torch.float32


def _gen(seed, k=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1009 + k)
    return g


def _truth(m, rng):
    """Piecewise-smooth m x m image in [0, 1]: a ramp, rectangles and disks."""
    ax = torch.arange(m, dtype=torch.float64, device="cuda")
    yy, xx = ax[:, None], ax[None, :]
    a, b = rng.uniform(-1.0, 1.0, 2)
    ramp = (a * xx + b * yy) / max(m - 1, 1)
    img = 0.4 * (ramp - ramp.min()) / (ramp.max() - ramp.min())
    for _ in range(12):
        cy, cx = rng.uniform(0, m, 2)
        h, w = rng.uniform(m / 16.0, m / 4.0, 2)
        if rng.uniform() < 0.5:
            mask = ((yy - cy).abs() <= h / 2) & ((xx - cx).abs() <= w / 2)
        else:
            mask = (yy - cy) ** 2 + (xx - cx) ** 2 <= h * h / 4
        img = torch.where(mask, float(rng.uniform()), img)
    return img.clamp(0, 1)


def _observe(n, h, bc, nu, seed, k=0):
    """(g, delta): the field of view of a blurred larger scene (periodic BCs:
    a periodic scene) plus white noise of relative norm nu."""
    rng = np.random.default_rng([int(seed), k])
    if bc == "periodic":
        clean = _blur64(_truth(n, rng), h, "periodic")
    else:
        clean = _blur64(_truth(n + h.shape[0] - 1, rng), h, "rect")
    e = torch.randn(clean.shape, generator=_gen(seed, k), dtype=torch.float64, device="cuda")
    eta = e * (nu * torch.linalg.norm(clean) / torch.linalg.norm(e))
    return clean + eta, float(torch.linalg.norm(eta))


def _batch_specs(case):
    """The problems of a batch case: size, PSF, BC, algorithm and noise drawn
    as in the benchmark's 64-problem batch."""
    rng = np.random.default_rng([int(case["spec"]), 0xba7c])
    sizes = [n for n in SIZES if case["lo"] <= n <= case["hi"]]
    out = []
    for _ in range(case["count"]):
        # the benchmark's sizes, or (ranges of another shape) any even size
        if (case["lo"], case["hi"]) == (SIZES[0], SIZES[-1]):
            n = int(rng.choice(sizes))
        else:
            n = 2 * int(rng.integers(case["lo"] // 2, case["hi"] // 2 + 1))
            while _largest_prime(n) > 31:
                n += 2
        fam = ("gauss", "disk", "motion")[int(rng.integers(0, 3))]
        if fam == "gauss":
            size = float(rng.uniform(1.0, 4.0))
            p, ang = 2 * int(math.ceil(3.0 * size)) + 1, 0.0
        elif fam == "disk":
            size, ang = float(rng.integers(2, 9)), 0.0
            p = 2 * int(size) + 3
        else:
            p = int(rng.choice(np.arange(5, 22, 2)))
            size, ang = float(p), float(rng.uniform(0.0, math.pi))
        bc = ("periodic", "reflective", "rect")[int(rng.integers(0, 3))]
        nu = float(rng.uniform(0.005, 0.03))
        if bc == "rect":
            precond, alpha = "bccb", 0.5
        elif bc == "periodic" or fam != "motion":
            precond, alpha = "tikh_ns", 0.05
        else:
            precond, alpha = "sym", 0.3
        out.append(dict(n=n, h=_psf(fam, p, size, ang), bc=bc, precond=precond, alpha=alpha, nu=nu))
    return out


def _randn(shape, seed, k, dtype, scale=1.0):
    return (scale * torch.randn(shape, generator=_gen(seed, k), dtype=torch.float64, device="cuda")).to(dtype)


def _z_dtype(case):
    return {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}[case["z_store"]]


def _op_inputs(case, seed):
    n, t = case["n"], _dtype(case)
    if case["kind"] == "blur":
        nf = n + case["p"] - 1 if case["bc"] == "rect" else n
        rng = np.random.default_rng([int(seed), 7])
        return _truth(nf, rng).to(t), _randn((n, n), seed, 1, t, 0.05)
    if case["kind"] == "precond":
        rng = np.random.default_rng([int(seed), 8])
        return ((_truth(n, rng) + _randn((n, n), seed, 2, torch.float64, 0.02)).to(t),)
    # frame: Bregman coefficients around the threshold and a correction image
    zi = _randn((8 * case["levels"] + 1, n, n), seed, 3, torch.float32 if t == torch.float32 else t, 0.04)
    rng = np.random.default_rng([int(seed), 9])
    return zi.to(_z_dtype(case)), (_truth(n, rng) * 0.2 + _randn((n, n), seed, 4, torch.float64, 0.02)).to(t)


# ---------------------------------------------------------------------------
# what a program keeps, and one pass

def prepare(case, seed):
    kind = case["kind"]
    if kind == "restore":
        h = _psf(case["psf"], case["p"], case["size"], case["angle"])
        g, delta = _observe(case["n"], h, case["bc"], case["nu"], seed)
        ctx = mlba.Context(h, case["n"], case["bc"], case["precond"], dtype=case["dtype"],
                           z_store=case["z_store"], mu=MU, alpha=case["alpha"], levels=case["levels"],
                           max_iter=case["iters"] + 1, stop=False, transform=case["transform"],
                           rect_ns_hybrid=True, formulation=case["formulation"],
                           blur_path=case["blur_path"])
        return dict(kind=kind, ctx=ctx, g=g.to(_dtype(case)), delta=delta, iters=case["iters"])
    if kind == "batch":
        probs, gs, deltas = [], [], []
        for k, s in enumerate(_batch_specs(case)):
            g, delta = _observe(s["n"], s["h"], s["bc"], s["nu"], seed, k + 1)
            g = g.float()
            gs.append(g)
            deltas.append(delta)
            probs.append(dict(psf=s["h"], g=g, delta=delta, bc=s["bc"], precond=s["precond"], mu=MU,
                              alpha=s["alpha"]))
        b = mlba.Batch(probs, dtype="f32", z_store=case["z_store"], levels=case["levels"], stop=False,
                       max_iter=case["iters"] + 1)
        return dict(kind=kind, batch=b, gs=gs, deltas=deltas, iters=case["iters"])
    if kind == "frame":
        h = _psf("gauss", 3, 0.8, 0.0)
        ctx = mlba.Context(h, case["n"], "reflective", "none", dtype=case["dtype"],
                           z_store=case["z_store"], levels=case["levels"])
        zi, u = _op_inputs(case, seed)
        return dict(kind=kind, ctx=ctx, z=zi, u=u)
    h = _psf(case["psf"], case["p"], case["size"], case["angle"])
    if kind == "blur":
        ctx = mlba.Context(h, case["n"], case["bc"], "none", dtype=case["dtype"],
                           blur_path=case["blur_path"])
        f, t = _op_inputs(case, seed)
        return dict(kind=kind, ctx=ctx, f=f, t=t)
    ctx = mlba.Context(h, case["n"], "periodic" if case["transform"] == "dft" else "reflective", "bccb",
                       dtype=case["dtype"], transform=case["transform"])
    return dict(kind=kind, ctx=ctx, r=_op_inputs(case, seed)[0], alpha=case["alpha"], which=case["which"])


def run(state):
    kind = state["kind"]
    if kind == "restore":
        ctx = state["ctx"]
        ctx.set_data(state["g"], state["delta"])
        ctx.iterate(state["iters"])
        return ctx.result(device=True)
    if kind == "batch":
        b = state["batch"]
        b.set_data_all(state["gs"], state["deltas"])
        b.reset()
        b.iterate(state["iters"])
        return [b.result(i, device=True) for i in range(b.count)]
    ctx = state["ctx"]
    if kind == "blur":
        return [ctx.blur(state["f"]), ctx.blur_adjoint(state["t"])]
    if kind == "precond":
        return ctx.precond(state["r"], state["alpha"], state["which"])
    return list(ctx.frame(state["z"], state["u"], MU))


# ---------------------------------------------------------------------------
# what a pass cannot do without

def _step_work(n, p, sep_or_taps, bc, precond, levels, ts, zs):
    nf = n + p - 1 if bc == "rect" else n
    bands = 8 * levels + 1
    # z and f read and written, g and |lambda|^2 read
    b = 2 * bands * zs * nf * nf + 2 * ts * nf * nf + 2 * ts * n * n
    lg = math.log2(max(n, 2))
    solves = 6 if precond == "krylov" else 1
    fl = nf * nf * (levels * 150.0) + solves * (4.0 * sep_or_taps * n * n + 10.0 * n * n * lg)
    return b, fl


def _taps(h):
    p = h.shape[0]
    sep = np.linalg.matrix_rank(h, tol=1e-12) == 1
    return 2 * p if sep else int((h != 0).sum())


def work(case):
    kind = case["kind"]
    if kind == "batch":
        b = f = 0.0
        for s in _batch_specs(case):
            x, y = _step_work(s["n"], s["h"].shape[0], _taps(s["h"]), s["bc"], s["precond"],
                              case["levels"], 4, 2 if case["z_store"] == "bf16" else 4)
            b, f = b + x, f + y
        return {"bytes": b * case["iters"], "flops": f * case["iters"]}
    ts = 8 if case["dtype"] == "f64" else 4
    n = case["n"]
    if kind == "frame":
        bands, zs = 8 * case["levels"] + 1, {"f64": 8, "f32": 4, "bf16": 2}[case["z_store"]]
        return {"bytes": 2.0 * bands * zs * n * n + 2 * ts * n * n, "flops": 150.0 * case["levels"] * n * n}
    h = _psf(case["psf"], case["p"], case["size"], case["angle"])
    if kind == "restore":
        zs = {"f64": 8, "f32": 4, "bf16": 2}[case["z_store"]]
        b, f = _step_work(n, case["p"], _taps(h), case["bc"], case["precond"], case["levels"], ts, zs)
        return {"bytes": b * case["iters"], "flops": f * case["iters"]}
    if kind == "blur":
        nf = n + case["p"] - 1 if case["bc"] == "rect" else n
        return {"bytes": 2.0 * ts * (n * n + nf * nf), "flops": 4.0 * _taps(h) * n * n}
    half = n // 2 + 1
    spec = ts * (n * n if case["transform"] == "dct" else 2 * n * half) if case["which"] == "tikh" else ts * n * half
    return {"bytes": 2.0 * ts * n * n + spec, "flops": 10.0 * n * n * math.log2(n)}


# ---------------------------------------------------------------------------
# the same results in 64 bits, from the definitions

def _conv(x, h, flip, size):
    """Full linear convolution (flip: correlation) of x with h, cropped to size."""
    k = torch.as_tensor(np.ascontiguousarray(h[::-1, ::-1] if flip else h), dtype=torch.float64, device="cuda")
    m = x.shape[0] + h.shape[0] - 1
    m = -(-m // 64) * 64
    y = torch.fft.irfft2(torch.fft.rfft2(x, s=(m, m)) * torch.fft.rfft2(k, s=(m, m)), s=(m, m))
    return y[:size, :size]


def _bc_index(n, c, bc):
    e = torch.arange(-c, n + c, device="cuda")
    if bc == "zero":
        return e.clamp(0, n - 1), (e >= 0) & (e < n)
    if bc == "periodic":
        return e % n, torch.ones_like(e, dtype=torch.bool)
    q = e % (2 * n)
    return torch.where(q < n, q, 2 * n - 1 - q), torch.ones_like(e, dtype=torch.bool)


def _antireflect(f, c):
    for _ in range(2):       # rows, then columns (transposed in between)
        n = f.shape[0]
        top = 2.0 * f[:1] - f[1:c + 1].flip(0)
        bot = 2.0 * f[n - 1:] - f[n - 1 - c:n - 1].flip(0)
        f = torch.cat([top, f, bot]).T
    return f


def _blur64(f, h, bc):
    p = h.shape[0]
    c = (p - 1) // 2
    if bc == "rect":
        ext = f
    elif bc == "antireflective":
        ext = _antireflect(f, c)
    else:
        ix, ok = _bc_index(f.shape[0], c, bc)
        ext = f[ix][:, ix] * (ok[:, None] & ok[None, :])
    return _conv(ext, h, False, ext.shape[0])[p - 1:, p - 1:].contiguous()


def _adjoint64(t, h, bc):
    if bc == "antireflective":
        return _blur64(t, h[::-1, ::-1], bc)
    n, p = t.shape[0], h.shape[0]
    v = _conv(t, h, True, n + p - 1)
    if bc == "rect":
        return v.contiguous()
    ix, ok = _bc_index(n, (p - 1) // 2, bc)
    v = v * (ok[:, None] & ok[None, :])
    rows = torch.zeros((n, v.shape[1]), dtype=torch.float64, device="cuda").index_add_(0, ix, v)
    return torch.zeros((n, n), dtype=torch.float64, device="cuda").index_add_(1, ix, rows)


def _cos(k, n2):
    """cos(2 pi k / n2) of integers k, reduced exactly."""
    return torch.cos(2.0 * math.pi * (k % n2).double() / n2)


class _Spectral:
    """C diagonalised by the DFT, the DCT or the antireflective transform."""

    def __init__(self, h, n, transform):
        self.tr, self.n = transform, n
        p = h.shape[0]
        c = (p - 1) // 2
        hh = torch.as_tensor(np.ascontiguousarray(h), dtype=torch.float64, device="cuda")
        i = torch.arange(n, device="cuda")
        d = torch.arange(p, device="cuda") - c
        if transform == "dft":
            pad = torch.zeros((n, n), dtype=torch.float64, device="cuda")
            pad[:p, :p] = hh
            self.lam = torch.fft.fft2(torch.roll(pad, (-c, -c), (0, 1)))
        elif transform == "dct":
            ck = _cos(i[:, None] * d[None, :], 2 * n)
            self.lam = ck @ hh @ ck.T
            s = torch.full((n, 1), math.sqrt(2.0 / n), dtype=torch.float64, device="cuda")
            s[0] = math.sqrt(1.0 / n)
            self.d = s * _cos(i[:, None] * (2 * i[None, :] + 1), 4 * n)
        else:
            kk = i.clone()
            kk[n - 1] = 0
            ck = _cos(kk[:, None] * d[None, :], 2 * (n - 1))
            self.lam = ck @ hh @ ck.T
            t = torch.sin(math.pi * ((i[:, None] * i[None, :]) % (2 * (n - 1))).double() / (n - 1))
            t[:, 0] = 1.0 - i.double() / (n - 1)
            t[:, n - 1] = i.double() / (n - 1)
            self.t, self.ti = t, torch.linalg.inv(t)
        self.sigma = self.lam.abs() ** 2

    def forward(self, r):
        if self.tr == "dft":
            return torch.fft.fft2(r) / self.n
        return self.d @ r @ self.d.T if self.tr == "dct" else self.ti @ r @ self.ti.T

    def inverse(self, x):
        if self.tr == "dft":
            return torch.fft.ifft2(x * self.n).real
        return self.d.T @ x @ self.d if self.tr == "dct" else self.t @ x @ self.t.T

    def inv(self, r, alpha):
        return self.inverse(self.forward(r) / (self.sigma + alpha))

    def tikh(self, r, alpha):
        return self.inverse(self.forward(r) * self.lam.conj() / (self.sigma + alpha))


MASKS = ((0.25, 0.5, 0.25), (math.sqrt(2.0) / 4.0, 0.0, -math.sqrt(2.0) / 4.0), (-0.25, 0.5, -0.25))


def _refl(n, shift):
    q = (torch.arange(n, device="cuda") + shift) % (2 * n)
    return torch.where(q < n, q, 2 * n - 1 - q)


def _mask(x, k, d, dim):
    a, b, c = MASKS[k]
    n = x.shape[dim]
    y = a * x.index_select(dim, _refl(n, -d)) + c * x.index_select(dim, _refl(n, d))
    return y + b * x if b else y


def _mask_t(x, k, d, dim):
    a, b, c = MASKS[k]
    n = x.shape[dim]
    y = torch.zeros_like(x) if not b else b * x
    y.index_add_(dim, _refl(n, -d), x, alpha=a)
    return y.index_add_(dim, _refl(n, d), x, alpha=c)


def _frame64(z, u, levels, mu, replace=False):
    """z <- z + W u (replace: W u) in place; returns W^T S_mu(z)."""
    soft = lambda v: torch.sign(v) * (v.abs() - mu).clamp_min(0.0)  # noqa: E731
    cur = u
    for lev in range(levels):
        rows = [_mask(cur, i, 1 << lev, 0) for i in range(3)]
        for k in range(1, 9):
            b = 8 * lev + k - 1
            w = _mask(rows[k // 3], k % 3, 1 << lev, 1)
            z[b] = w if replace else z[b] + w
        cur = _mask(rows[0], 0, 1 << lev, 1)
    z[8 * levels] = cur if replace else z[8 * levels] + cur
    s = soft(z[8 * levels])
    for lev in range(levels - 1, -1, -1):
        d = 1 << lev
        acc = 0.0
        for i in range(3):
            row = 0.0
            for j in range(3):
                x = s if (i, j) == (0, 0) else soft(z[8 * lev + 3 * i + j - 1])
                row = row + _mask_t(x, j, d, 1)
            acc = acc + _mask_t(row, i, d, 0)
        s = acc
    return s


def _alpha_root(pw, sigma, qn):
    """alpha with sum pw (alpha / (sigma + alpha))^2 = qn^2 sum pw (bisection on log alpha)."""
    total = float(pw.sum())

    def over(b):
        a = math.exp(b)
        return float((pw * (a / (sigma + a)) ** 2).sum()) - qn * qn * total
    lo, hi = math.log(1e-14), 0.0
    if over(lo) >= 0:
        return 1e-14
    while over(hi) < 0:
        lo, hi = hi, hi + 3.0
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        if over(mid) < 0:
            lo = mid
        else:
            hi = mid
    return math.exp(0.5 * (lo + hi))


def _transform_of(h, precond, transform, bc):
    sym = all(np.abs(h - x).max() <= 1e-14 * np.abs(h).max() for x in (h[::-1], h[:, ::-1]))
    if precond == "sym":
        return "ar" if bc == "antireflective" else "dct"
    if transform != "auto":
        return transform
    if bc == "periodic":
        return "dft"
    if bc == "antireflective":
        return "ar" if sym and precond != "tikh_ns" else "dft"
    return "dct" if sym else "dft"


def _mlba64(g, h, delta, bc, precond, alpha, levels, iters, transform="auto", formulation="synthesis",
            q=0.5, rho=1e-4, pcg_tol=1e-3, pcg_max=5):
    n, p = g.shape[0], h.shape[0]
    nf = n + p - 1 if bc == "rect" else n
    hs = 0.25 * (h + h[::-1] + h[:, ::-1] + h[::-1, ::-1]) if precond == "sym" else h
    pre = _Spectral(hs, n, _transform_of(h, precond, transform, bc))
    z = torch.zeros((8 * levels + 1, nf, nf), dtype=torch.float64, device="cuda")
    f = torch.zeros((nf, nf), dtype=torch.float64, device="cuda")
    a_n = alpha
    for _ in range(iters):
        r = g - _blur64(f, h, bc)
        if precond in ("bccb", "sym"):
            u = _adjoint64(pre.inv(r, alpha), h, bc)
        elif precond == "krylov":
            x, res = torch.zeros_like(r), r.clone()
            y = pre.inv(res, alpha)
            rho_k = rho_0 = float((res * y).sum())
            d = y.clone()
            for _ in range(pcg_max):
                ad = _blur64(_adjoint64(d, h, bc), h, bc) + alpha * d
                step = rho_k / float((d * ad).sum())
                x = x + step * d
                res = res - step * ad
                y = pre.inv(res, alpha)
                rho_new = float((res * y).sum())
                if math.sqrt(max(rho_new, 0.0) / rho_0) <= pcg_tol:
                    break
                d = y + (rho_new / rho_k) * d
                rho_k = rho_new
            u = _adjoint64(x, h, bc)
        elif precond == "tikh":
            u = pre.tikh(r, alpha)
        else:
            rn = float(torch.linalg.norm(r))
            if not rn <= (1.0 + 2.0 * rho) / (1.0 - 2.0 * rho) * delta:
                qn = max(q, 2.0 * rho + (1.0 + rho) * delta / rn)
                a_n = _alpha_root(pre.forward(r).abs() ** 2, pre.sigma, qn)
                if bc == "rect":
                    a_n = max(a_n, alpha)
            u = _adjoint64(pre.inv(r, a_n), h, bc) if bc == "rect" else pre.tikh(r, a_n)
        if formulation == "balanced":
            f = _frame64(z, f + u, levels, MU, replace=True)
        else:
            f = _frame64(z, u, levels, MU)
    return f


def exact(case, seed):
    kind = case["kind"]
    if kind == "restore":
        h = _psf(case["psf"], case["p"], case["size"], case["angle"])
        g, delta = _observe(case["n"], h, case["bc"], case["nu"], seed)
        return _mlba64(g.to(_dtype(case)).double(), h, delta, case["bc"], case["precond"], case["alpha"],
                       case["levels"], case["iters"], case["transform"], case["formulation"])
    if kind == "batch":
        out = []
        for k, s in enumerate(_batch_specs(case)):
            g, delta = _observe(s["n"], s["h"], s["bc"], s["nu"], seed, k + 1)
            out.append(_mlba64(g.float().double(), s["h"], delta, s["bc"], s["precond"], s["alpha"],
                               case["levels"], case["iters"]))
        return out
    ins = [x.double() for x in _op_inputs(case, seed)]
    if kind == "frame":
        z = ins[0].clone()
        f = _frame64(z, ins[1], case["levels"], MU)
        return [z, f]
    h = _psf(case["psf"], case["p"], case["size"], case["angle"])
    if kind == "blur":
        return [_blur64(ins[0], h, case["bc"]), _adjoint64(ins[1], h, case["bc"])]
    pre = _Spectral(h, case["n"], case["transform"])
    return (pre.tikh if case["which"] == "tikh" else pre.inv)(ins[0], case["alpha"])
