"""What this framework is timed on: Richardson-Lucy calls as a user's program makes them.

Every case goes through the package's public entry points, with float32 CUDA volumes and
plans kept from call to call: a program that deconvolves a stack of images from one
microscope makes one plan per volume shape and PSF, and sends image after image through it.
The sizes are the repository's own workloads (``synth``) and sizes around them.

  listed()             the cases
  draw(rng)            one more case of the same ranges
  prepare(case, seed)  the images (from the seed) and the kept plans (from the case)
  run(state)           one pass through the entry point, and its outputs
  work(case)           bytes and operations that a pass cannot do without
  exact(case, seed)    the same outputs in 64 bits, by torch.fft alone
"""
import math

import numpy as np
import torch

import paper_2510_14143_gb300 as cr
from paper_2510_14143_gb300 import synth
from paper_2510_14143_gb300.autograd import RLDeconvolve

EPS = 1e-6

#: axis lengths with kernels, from thin stacks to camera width
LENGTHS = (8, 9, 10, 12, 15, 16, 18, 20, 24, 25, 27, 30, 32, 36, 40, 45, 48, 50, 54, 60, 64, 72, 75, 80, 81, 90, 96,
           100, 108, 120, 125, 128, 135, 144, 150, 160, 192, 256, 320, 384, 512, 640, 768, 1024)
PLANE = tuple(n for n in LENGTHS if n >= 32)
STACK = tuple(n for n in LENGTHS if n <= 160)


def listed():
    return [
        # one small crop (a nucleus), 20 iterations: bound by launches and latency
        dict(name="plain_small", kind="plain", nz=32, ny=64, nx=64, psf="gaussian", n_iter=20, tuned=False),
        # an odd-sized crop with a measured (not point-symmetric) PSF: the complex-spectrum path
        dict(name="plain_odd_skewed", kind="plain", nz=81, ny=150, nx=135, psf="skewed", n_iter=30, tuned=False),
        # a camera region of interest, many iterations, launch shapes tuned once
        dict(name="plain_medium", kind="plain", nz=128, ny=256, nx=256, psf="gaussian", n_iter=100, tuned=True),
        # the full-field volume the throughput is quoted on
        dict(name="plain_large", kind="plain", nz=128, ny=1024, nx=1024, psf="gaussian", n_iter=50, tuned=True),
        # the paper's stack shape: few slices of a whole camera frame, lengths past 1024
        dict(name="plain_paper", kind="plain", nz=30, ny=2160, nx=2560, psf="gaussian", n_iter=20, tuned=True),
        # zero-padded boundaries, image of any size, a small PSF box
        dict(name="linear_ragged", kind="linear", nz=61, ny=487, nx=501, kz=25, ky=33, kx=33, psf="skewed", n_iter=20,
             tuned=False),
        # a dataset of 64 crops of uneven sizes in one call
        dict(name="batched_64", kind="batched", count=64, shape_seed=synth.SEED_BASE + 4, n_iter=50),
        # fitting the PSF and the image through 30 unrolled iterations (forward and backward)
        dict(name="grad_16", kind="grad", count=16, nz=64, ny=128, nx=128, n_iter=30, ckpt=6),
        # accelerated iterations on a half-field volume
        dict(name="accel_half_field", kind="accel", nz=64, ny=512, nx=512, psf="gaussian", n_iter=20, tuned=True),
        # likelihood-guided stopping, checked every five iterations, run to its cap
        dict(name="monitor_medium", kind="monitor", nz=64, ny=256, nx=256, psf="gaussian", n_iter=25, check=5,
             tuned=False),
        # resolution of a result: Fourier shell correlation of two volumes
        dict(name="fsc_medium", kind="fsc", nz=128, ny=256, nx=256, shells=64),
        # one blur (or its adjoint) of a volume: the building block of other restoration methods
        dict(name="convolve_adjoint", kind="convolve", nz=96, ny=320, nx=384, psf="skewed", flipped=True),
    ]


def _spread(rng, lo, hi):
    """A whole number between lo and hi, spread over its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _shape(rng, most):
    """A volume shape with lengths spread over the supported range, at most `most` voxels."""
    while True:
        near = lambda seq, v: min(seq, key=lambda n: (abs(math.log(n / v)), rng.random()))  # noqa: E731
        nx, ny = near(PLANE, _spread(rng, 32, 1024)), near(PLANE, _spread(rng, 32, 1024))
        nz = near(STACK, _spread(rng, 8, 160))
        if 1 / 4 <= nx / ny <= 4 and nz * ny * nx <= most:
            return dict(nz=nz, ny=ny, nx=nx)


def draw(rng):
    kind = rng.choice(("plain", "plain", "plain", "linear", "batched", "grad", "accel", "monitor", "fsc", "convolve"))
    psf = rng.choice(("gaussian", "skewed"))
    tuned = rng.random() < 0.3
    if kind == "linear":
        while True:
            k = dict(kz=rng.randrange(3, 26), ky=rng.randrange(5, 34), kx=rng.randrange(5, 34))
            n = dict(nz=_spread(rng, 8, 100), ny=_spread(rng, 48, 700), nx=_spread(rng, 48, 700))
            if n["nz"] * n["ny"] * n["nx"] <= 24_000_000:
                return dict(kind=kind, **n, **k, psf=psf, n_iter=rng.randrange(5, 31), tuned=False)
    if kind == "batched":
        return dict(kind=kind, count=_spread(rng, 2, 48), shape_seed=rng.randrange(1, 1 << 20), n_iter=rng.randrange(5, 51))
    if kind == "grad":
        return dict(kind=kind, count=_spread(rng, 1, 12), **_shape(rng, 1_100_000), n_iter=rng.randrange(4, 25),
                    ckpt=rng.randrange(1, 7))
    if kind == "fsc":
        s = _shape(rng, 1024 * 1024 * 64)
        return dict(kind=kind, **s, shells=max(4, min(s.values()) // 2))
    if kind == "convolve":
        return dict(kind=kind, **_shape(rng, 1024 * 1024 * 64), psf=psf, flipped=rng.random() < 0.5)
    if kind == "accel":
        return dict(kind=kind, **_shape(rng, 1024 * 1024 * 32), psf=psf, n_iter=rng.randrange(5, 31), tuned=tuned)
    if kind == "monitor":
        return dict(kind=kind, **_shape(rng, 1024 * 1024 * 16), psf=psf, n_iter=rng.randrange(5, 31),
                    check=rng.randrange(1, 8), tuned=tuned)
    return dict(kind=kind, **_shape(rng, 1024 * 1024 * 64), psf=psf, n_iter=rng.randrange(5, 51), tuned=tuned)


# ------------------------------------------------------------------ inputs


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _axes(shape, dtype):
    """Index minus floor(n/2) along each axis, shaped for broadcasting."""
    nz, ny, nx = (torch.arange(n, device="cuda", dtype=dtype) - n // 2 for n in shape)
    return nz[:, None, None], ny[None, :, None], nx[None, None, :]


def _psf(shape, kind):
    """A normalised PSF volume, peak at index n // 2: a Gaussian, or one with a weaker lobe off its centre
    (coma, as in measured PSFs), which has no point symmetry."""
    z, y, x = _axes(shape, torch.float32)
    sz, sxy = min(3.0, max(0.7, shape[0] / 12)), 2.0
    g = torch.exp(-0.5 * ((z / sz) ** 2 + (y / sxy) ** 2 + (x / sxy) ** 2))
    if kind == "skewed":
        g = g + 0.3 * torch.exp(-0.5 * (((z - 1) / (1.3 * sz)) ** 2 + ((y - 2) / 2.6) ** 2 + ((x + 1) / 2.2) ** 2))
    return (g / g.sum(dtype=torch.float64)).to(torch.float32).contiguous()


def _blur(v, sz, sxy):
    """Circular Gaussian blur of unit gain (the optics of the synthetic images)."""
    fz, fy = (torch.fft.fftfreq(n, device="cuda") for n in v.shape[:2])
    fx = torch.fft.rfftfreq(v.shape[2], device="cuda")
    s = torch.fft.rfftn(v)
    for f, sig, dims in ((fz, sz, (-1, 1, 1)), (fy, sxy, (1, -1, 1)), (fx, sxy, (1, 1, -1))):
        s *= torch.exp(-2 * (math.pi * sig * f) ** 2).view(dims)
    return torch.fft.irfftn(s, s=v.shape)


def _object(shape, g):
    """Bright blobs (sigma 2 voxels, peaks of 200 to 1000, about one in 6000 voxels) on a background of 10."""
    at = torch.rand(shape, device="cuda", generator=g) < 1.6e-4
    peak = 200 + 800 * torch.rand(shape, device="cuda", generator=g)
    sz = min(2.0, max(0.7, shape[0] / 12))
    return 10 + _blur(at * peak, sz, 2.0).clamp_(min=0) * ((2 * math.pi) ** 1.5 * 4 * sz)


def _image(shape, g):
    """A photon-count image: the blurred object with Poisson noise."""
    sz = min(3.0, max(0.7, shape[0] / 12))
    return torch.poisson(_blur(_object(shape, g), sz, 2.0).clamp_(min=0), generator=g).contiguous()


def _dims(case):
    return case["nz"], case["ny"], case["nx"]


def _shapes(case):
    return synth.batch_shapes(case["count"], case["shape_seed"])


#: plans by what they are made of, kept for the life of the program
_plans = {}


def _plan(shape, psf_shape, psf, boundary="circular", index=0, tuned=False):
    key = (tuple(shape), tuple(psf_shape), psf, boundary, index, tuned)
    if key not in _plans:
        p = _psf(psf_shape, psf)
        plan = cr.cubic_rl_plan_linear(shape, p) if boundary == "linear" else cr.cubic_rl_plan(shape, p)
        if tuned:
            im = 1 + torch.rand(shape, device="cuda", generator=_gen(1))
            cr.cubic_rl_autotune(plan, im, torch.empty_like(im))
        torch.cuda.synchronize()
        _plans[key] = plan
    return _plans[key]


def prepare(case, seed):
    g, kind = _gen(seed), case["kind"]
    s = {"case": case}
    if kind == "batched":
        shapes = _shapes(case)
        s["plans"] = [_plan(sh, sh, "gaussian", index=1 + i) for i, sh in enumerate(shapes)]
        s["images"] = [_image(sh, g) for sh in shapes]
        s["outs"] = [torch.empty_like(im) for im in s["images"]]
        return s
    shape = _dims(case)
    if kind == "grad":
        s["d"] = torch.stack([_image(shape, g) for _ in range(case["count"])]).requires_grad_()
        s["target"] = torch.stack([_object(shape, g) for _ in range(case["count"])])
        s["params"] = [torch.tensor(v, device="cuda", requires_grad=True) for v in synth.GRAD_EVAL_PSF]
        return s
    if kind == "fsc":
        obj = _object(shape, g)
        s["plan"] = _plan(shape, shape, "gaussian")
        s["a"], s["b"] = (torch.poisson(obj, generator=g) for _ in range(2))
        return s
    if kind == "linear":
        s["plan"] = _plan(shape, (case["kz"], case["ky"], case["kx"]), case["psf"], "linear", tuned=case["tuned"])
    else:
        s["plan"] = _plan(shape, shape, case["psf"], tuned=case.get("tuned", False))
    s["image"] = _image(shape, g)
    s["out"] = torch.empty_like(s["image"])
    return s


# ------------------------------------------------------------------ one pass


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind in ("plain", "linear"):
        cr.cubic_rl_deconvolve(s["plan"], s["image"], case["n_iter"], EPS, s["out"])
        return s["out"]
    if kind == "batched":
        cr.cubic_rl_deconvolve_batched(s["plans"], s["images"], case["n_iter"], EPS, s["outs"])
        return s["outs"]
    if kind == "grad":
        u = RLDeconvolve.apply(s["d"], *s["params"], case["n_iter"], EPS, case["ckpt"])
        loss = (u - s["target"]).square().mean()
        grads = torch.autograd.grad(loss, [s["d"], *s["params"]])
        return {"out": u.detach(), "d": grads[0], "psf": torch.stack(grads[1:])}
    if kind == "accel":
        cr.cubic_rl_deconvolve_accel(s["plan"], s["image"], case["n_iter"], EPS, s["out"])
        return s["out"]
    if kind == "monitor":
        n, hist = cr.cubic_rl_deconvolve_monitor(s["plan"], s["image"], case["n_iter"], EPS, cr.METRIC_NLL, 0.0,
                                                 case["check"], s["out"])
        hist = np.asarray(hist, np.float32)
        return {"out": s["out"], "n": n, "change": hist[:, 0], "nll": hist[:, 1]}
    if kind == "fsc":
        return cr.cubic_fsc(s["plan"], s["a"], s["b"], case["shells"])
    cr.cubic_rl_convolve(s["plan"], s["image"], case["flipped"], s["out"])
    return s["out"]


# ------------------------------------------------------------------ what a pass needs


def _transform(shape):
    """Operations of one real 3D transform."""
    v = math.prod(shape)
    return 2.5 * v * math.log2(max(v, 2))


def work(case):
    """Bytes: the images, the PSF's spectrum (half of it in 64 bits, or in 32 where it is real) and the results, once
    each.  Operations: the transforms and the pointwise steps."""
    kind = case["kind"]
    if kind == "batched":
        each = [work(dict(kind="plain", nz=z, ny=y, nx=x, psf="gaussian", n_iter=case["n_iter"])) for z, y, x in _shapes(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    shape = _dims(case)
    v, t = math.prod(shape), _transform(shape)
    n = case.get("n_iter", 0)
    if kind == "grad":
        # forward: 4 transforms an iteration, backward: 4 more; image, target, result and gradient
        return {"bytes": case["count"] * v * 16, "flops": case["count"] * n * (8 * t + 12 * v)}
    if kind == "fsc":
        return {"bytes": 8 * v, "flops": 2 * t + 12 * v}
    spectrum = v * (4 if case["psf"] == "skewed" else 2)
    if kind == "convolve":
        return {"bytes": 8 * v + spectrum, "flops": 2 * t + 3 * v}
    if kind == "linear":
        spectrum = 4 * case["kz"] * case["ky"] * case["kx"]
    extra = {"accel": 8, "monitor": 8}.get(kind, 0)
    return {"bytes": 8 * v + spectrum, "flops": n * (4 * t + (8 + extra) * v)}


# ------------------------------------------------------------------ the same in 64 bits


def _spectrum64(p, box):
    """Transform of a PSF (peak at floor(n/2)) placed with its peak at the origin of `box`."""
    h = torch.zeros(box, dtype=torch.float64, device="cuda")
    h[: p.shape[0], : p.shape[1], : p.shape[2]] = p
    return torch.fft.rfftn(torch.roll(h, [-(n // 2) for n in p.shape], (0, 1, 2)))


def _convolver(p, shape, box):
    h = _spectrum64(p.double(), box)
    nz, ny, nx = shape

    def conv(v, flipped):
        s = torch.fft.rfftn(v, s=box, dim=(0, 1, 2))
        s *= h.conj() if flipped else h
        return torch.fft.irfftn(s, s=box, dim=(0, 1, 2))[:nz, :ny, :nx]

    return conv


def _rl64(d, conv, n_iter, each=None):
    d = d.double()
    u = torch.full_like(d, max(float(d.mean()), EPS))
    for _ in range(n_iter):
        b = conv(u, False).clamp_(min=EPS)
        new = u * conv(d / b, True)
        if each:
            each(u, b, new)
        u = new
    return u


def _accel64(d, conv, n_iter):
    d = d.double()
    x = torch.full_like(d, max(float(d.mean()), EPS))
    prev, g1, g2 = x, None, None
    for k in range(n_iter):
        alpha = 0.0
        if k >= 2:
            den = float((g2 * g2).sum())
            alpha = min(1.0, max(0.0, float((g1 * g2).sum()) / den)) if den > 0 else 0.0
        y = (x + alpha * (x - prev)).clamp_(min=0)
        new = y * conv(d / conv(y, False).clamp_(min=EPS), True)
        prev, x, g1, g2 = x, new, new - y, g1
    return x


def _grad64(case, d, target, params):
    shape = _dims(case)
    sxy, sz, amp = (p.detach().double().requires_grad_() for p in params)
    total = d.numel()
    out, gd, gp = [], [], torch.zeros(3, dtype=torch.float64, device="cuda")
    for i in range(case["count"]):
        z, y, x = _axes(shape, torch.float64)
        g = torch.exp(-0.5 * ((x * x + y * y) / (sxy * sxy) + z * z / (sz * sz)))
        h = torch.fft.rfftn(torch.roll(amp * g / g.sum(), [-(n // 2) for n in shape], (0, 1, 2)))
        di = d[i].detach().double().requires_grad_()
        u = di.mean().clamp(min=EPS).expand(shape)
        for _ in range(case["n_iter"]):
            b = torch.fft.irfftn(torch.fft.rfftn(u) * h, s=shape)
            u = u * torch.fft.irfftn(torch.fft.rfftn(di / b.clamp(min=EPS)) * h.conj(), s=shape)
        loss = (u - target[i].double()).square().sum() / total
        grads = torch.autograd.grad(loss, [di, sxy, sz, amp])
        out.append(u.detach())
        gd.append(grads[0])
        gp += torch.stack(grads[1:])
    return {"out": torch.stack(out), "d": torch.stack(gd), "psf": gp}


def _fsc64(a, b, shells):
    shape = tuple(a.shape)
    lcm = math.lcm(*shape)
    ks = [torch.fft.fftfreq(n, d=1 / n, device="cuda", dtype=torch.float64).round().long() for n in shape[:2]]
    ks.append(torch.arange(shape[2] // 2 + 1, device="cuda"))
    r = [(k * (lcm // n)) ** 2 for k, n in zip(ks, shape)]
    t = 4 * shells * shells * (r[0][:, None, None] + r[1][None, :, None] + r[2][None, None, :])
    s = torch.sqrt(t.double() / lcm**2).floor().long()
    s = torch.where(s * s * lcm**2 > t, s - 1, s)
    s = torch.where((s + 1) ** 2 * lcm**2 <= t, s + 1, s).clamp_(max=shells).reshape(-1)
    w = torch.full((shape[2] // 2 + 1,), 2.0, dtype=torch.float64, device="cuda")
    w[0] = 1
    if shape[2] % 2 == 0:
        w[-1] = 1
    fa, fb = torch.fft.rfftn(a.double()), torch.fft.rfftn(b.double())

    def total(v):
        return torch.zeros(shells + 1, dtype=torch.float64, device="cuda").index_add_(0, s, (v * w).reshape(-1))[:shells]

    den = total(fa.abs() ** 2).sqrt() * total(fb.abs() ** 2).sqrt()
    return torch.where(den > 0, total((fa * fb.conj()).real) / den, torch.zeros_like(den))


def exact(case, seed):
    kind = case["kind"]
    if kind == "batched":
        g = _gen(seed)
        shapes = _shapes(case)
        return [_rl64(_image(sh, g), _convolver(_psf(sh, "gaussian"), sh, sh), case["n_iter"]) for sh in shapes]
    s = prepare(case, seed)
    shape = _dims(case)
    if kind == "grad":
        return _grad64(case, s["d"], s["target"], s["params"])
    if kind == "fsc":
        return _fsc64(s["a"], s["b"], case["shells"])
    if kind == "linear":
        k = (case["kz"], case["ky"], case["kx"])
        conv = _convolver(_psf(k, case["psf"]), shape, [n + m for n, m in zip(shape, k)])
    else:
        conv = _convolver(_psf(shape, case["psf"]), shape, shape)
    if kind == "convolve":
        return conv(s["image"].double(), case["flipped"])
    if kind == "accel":
        return _accel64(s["image"], conv, case["n_iter"])
    if kind == "monitor":
        change, nll = [], []
        d = s["image"].double()

        def each(u, b, new):
            change.append(float((new - u).norm() / u.norm()))
            nll.append(float((b - d * b.log()).sum()))

        u = _rl64(d, conv, case["n_iter"], each)
        return {"out": u, "n": None, "change": np.asarray(change), "nll": np.asarray(nll)}
    return _rl64(s["image"], conv, case["n_iter"])
