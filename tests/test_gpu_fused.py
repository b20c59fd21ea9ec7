"""The fused form, the warp-per-line X kernels and the two-stage Y kernels.

The fused form (one plane kernel and one convolution kernel per half iteration) against the
FP64 oracle and against the pass-by-pass form, at the lengths where it can go wrong: both
choices of the in-plane axis, odd x, odd in-plane axes, butterflies that leave lanes of a warp
idle, the smallest and largest radices, lengths and planes.

Tolerances: float32 transforms with FP64-generated twiddles, a few units of rounding times
log2(V): 1e-5 for one convolution (as for the pass-by-pass form).  Two float32 forms of the
same iteration differ by the rounding of both, at most a few times 1e-6 after some iterations;
the gradients divide by the blur and pass 4 iterations of both sweeps: 1e-4.
"""
import numpy as np
import pytest

import oracle
from paper_2510_14143_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cr():
    from paper_2510_14143_gb300 import build
    build.build()
    import paper_2510_14143_gb300 as m
    return m


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def rel_l2(a, b):
    a, b = (np.asarray(v.cpu() if isinstance(v, torch.Tensor) else v, np.float64) for v in (a, b))
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def skewed_psf(shape, seed):
    """No symmetry, bright centre: the complex-spectrum path, both products."""
    r = np.random.default_rng(seed)
    p = (r.uniform(0.0, 1.0, shape) ** 4).astype(np.float32)
    p[tuple(n // 2 for n in shape)] += 0.2 * p.sum()
    return p / p.sum()


def plans(cr, shape, psf):
    """A plan in the fused form and one pinned to the pass-by-pass form."""
    fused, passes = (cr.cubic_rl_plan(shape, dev(psf)) for _ in range(2))
    _, chosen = cr.cubic_rl_plan_variants(passes)
    cr.cubic_rl_plan_set_variants(passes, *chosen)
    return fused, passes


# (z, y, x): the plane takes the smaller of z and y (an even one before an odd one)
SHAPES = [(16, 20, 32), (20, 16, 36), (9, 24, 45), (10, 45, 75), (30, 25, 81), (81, 36, 135), (32, 27, 40), (8, 12, 50),
          (12, 8, 60), (24, 18, 125), (54, 100, 72), (40, 64, 72), (150, 160, 72), (144, 75, 64), (120, 160, 48),
          (45, 75, 64), (75, 81, 90), (81, 135, 75), (135, 75, 81), (45, 125, 80), (125, 45, 135), (12, 192, 192),
          (50, 81, 160), (96, 128, 144), (128, 135, 144), (160, 160, 150), (108, 150, 192), (90, 80, 108), (40, 60, 160),
          (15, 48, 128), (8, 9, 32), (27, 45, 36)]


@pytest.mark.parametrize("shape", SHAPES)
def test_convolve(cr, shape):
    psf = skewed_psf(shape, sum(shape))
    x = synth.random_field(shape, 11 + sum(shape), -1.0, 2.0)
    fused, passes = plans(cr, shape, psf)
    a, b = (torch.full(shape, float("nan"), device="cuda") for _ in range(2))
    for flipped in (False, True):
        cr.cubic_rl_convolve(fused, dev(x), flipped, a)
        cr.cubic_rl_convolve(passes, dev(x), flipped, b)
        assert rel_l2(a, b) <= 1e-5, flipped
        if np.prod(shape) <= 200_000:
            assert rel_l2(a, oracle.convolve(oracle.psf_spectrum(psf), x, flipped)) <= 1e-5, flipped


@pytest.mark.parametrize("shape", [(16, 20, 32), (10, 45, 75), (45, 75, 64), (30, 25, 81), (54, 100, 72), (81, 135, 75), (128, 135, 144)])
@pytest.mark.parametrize("symmetric", [True, False])
def test_deconvolve_monitor_accel(cr, shape, symmetric):
    d, xt = synth.make_volume(shape, 5, (1.5, 3.0), 10.0, 1.5, 2.0, 3 + sum(shape))
    psf = oracle.psf_gaussian(shape, 1.5, 2.0).astype(np.float32) if symmetric else skewed_psf(shape, 7)
    pair = plans(cr, shape, psf)
    outs, hists = [], []
    for plan in pair:
        u, m, acc = (torch.empty(shape, device="cuda") for _ in range(3))
        alpha = torch.empty(6, device="cuda")
        cr.cubic_rl_deconvolve(plan, dev(d), 6, 1e-6, u)
        n, hist = cr.cubic_rl_deconvolve_monitor(plan, dev(d), 6, 1e-6, cr.METRIC_REL_CHANGE, 0.0, 2, m, dev(xt))
        cr.cubic_rl_deconvolve_accel(plan, dev(d), 6, 1e-6, acc, alpha)
        assert n == 6
        outs.append((u, m, acc, alpha))
        hists.append(np.array(hist))
    for a, b in zip(*outs):
        assert rel_l2(a, b) <= 1e-5
    assert np.allclose(hists[0], hists[1], rtol=1e-5)
    if np.prod(shape) <= 200_000:
        assert rel_l2(outs[0][0], oracle.rl(d, psf, 6, 1e-6)) <= 1e-5


@pytest.mark.parametrize("shape", [(16, 20, 32), (9, 24, 45), (32, 27, 40), (27, 45, 36), (64, 75, 128)])
def test_backward(cr, shape):
    r = np.random.default_rng(sum(shape))
    d = r.uniform(2.0, 30.0, shape).astype(np.float32)
    g = r.standard_normal(shape).astype(np.float32)
    got = []
    for plan in plans(cr, shape, skewed_psf(shape, 5)):
        ck = torch.empty((2,) + shape, device="cuda")
        out, gd, gp = (torch.empty(shape, device="cuda") for _ in range(3))
        cr.cubic_rl_deconvolve_ckpt(plan, dev(d), 4, 1e-6, 2, ck, out)
        cr.cubic_rl_backward(plan, dev(d), 4, 1e-6, 2, ck, dev(g), gd, gp)
        got.append((out, gd, gp))
    for a, b in zip(*got):
        assert rel_l2(a, b) <= 1e-4


def test_psf_update_changes_both_forms(cr):
    shape = (16, 20, 32)
    x = dev(synth.random_field(shape, 3))
    sym = oracle.psf_gaussian(shape, 1.5, 2.0).astype(np.float32)
    fused, passes = plans(cr, shape, sym)
    a, b = (torch.empty(shape, device="cuda") for _ in range(2))
    for psf in (skewed_psf(shape, 1), sym, skewed_psf(shape, 2)):
        for plan, out in ((fused, a), (passes, b)):
            cr.cubic_rl_plan_update_psf(plan, dev(psf))
            cr.cubic_rl_convolve(plan, x, True, out)
        assert rel_l2(a, b) <= 1e-5
        assert rel_l2(a, oracle.convolve(oracle.psf_spectrum(psf), x.cpu().numpy(), True)) <= 1e-5


# ---- the warp-per-line X kernels: the last X shape of these lengths, odd row counts and a
# linear plan's row mapping included
@pytest.mark.parametrize("n", [256, 320, 384, 512, 640, 768, 1024])
@pytest.mark.parametrize("zy", [(3, 5), (2, 8), (9, 25)])
def test_warp_per_line_x(cr, n, zy):
    shape = zy + (n,)
    psf = skewed_psf(shape, n + sum(zy))
    plan = cr.cubic_rl_plan(shape, dev(psf))
    (nx, _, _), _ = cr.cubic_rl_plan_variants(plan)
    cr.cubic_rl_plan_set_variants(plan, nx - 1, 0, 0)
    x = synth.random_field(shape, n, -1.0, 2.0)
    out, u = (torch.full(shape, float("nan"), device="cuda") for _ in range(2))
    for flipped in (False, True):
        cr.cubic_rl_convolve(plan, dev(x), flipped, out)
        assert rel_l2(out, oracle.convolve(oracle.psf_spectrum(psf), x, flipped)) <= 1e-5
    d = synth.random_field(shape, 7, 5.0, 50.0)
    cr.cubic_rl_deconvolve(plan, dev(d), 5, 1e-6, u)
    assert rel_l2(u, oracle.rl(d, psf, 5, 1e-6)) <= 1e-5


@pytest.mark.parametrize("nx", [250, 600])
def test_warp_per_line_x_linear(cr, nx):
    shape, k = (5, 7, nx), (3, 4, 9)
    psf = skewed_psf(k, nx)
    plan = cr.cubic_rl_plan_linear(shape, dev(psf))
    d = synth.random_field(shape, nx, 5.0, 50.0)
    u = torch.empty(shape, device="cuda")
    cr.cubic_rl_deconvolve(plan, dev(d), 4, 1e-6, u)
    assert rel_l2(u, oracle.rl_same(d, psf, 4, 1e-6)) <= 1e-5


def test_fsc_long_common_multiple(cr):
    # dims whose least common multiple sends the shell arithmetic past 64 bits
    shape, shells = (125, 81, 256), 1024
    a = synth.random_field(shape, 1, 0.0, 2.0)
    b = a + synth.random_field(shape, 2, -1.0, 1.0)
    psf = np.zeros(shape, np.float32)
    psf[tuple(n // 2 for n in shape)] = 1
    got = cr.cubic_fsc(cr.cubic_rl_plan(shape, dev(psf)), dev(a), dev(b), shells)
    assert np.allclose(got.cpu().numpy(), oracle.fsc(a, b, shells)[0], atol=1e-4)


# ---- the two-stage Y kernels: the last shape of these lengths; spectrum columns that leave
# part of a column tile empty, a linear plan's rows that are not loaded or stored, column chunks
Y_LENGTHS = [125, 128, 135, 144, 150, 160, 192, 256, 320, 384, 512, 640, 768, 1024]


@pytest.mark.parametrize("n", Y_LENGTHS)
@pytest.mark.parametrize("zx", [(2, 6), (3, 45), (1, 64)])
def test_two_stage_y(cr, n, zx):
    shape = (zx[0], n, zx[1])
    psf = skewed_psf(shape, n + sum(zx))
    plan = cr.cubic_rl_plan(shape, dev(psf))
    (_, ny, _), _ = cr.cubic_rl_plan_variants(plan)
    cr.cubic_rl_plan_set_variants(plan, 0, ny - 1, 0)
    x = synth.random_field(shape, n, -1.0, 2.0)
    out, u = (torch.full(shape, float("nan"), device="cuda") for _ in range(2))
    for columns in (0, 16):
        cr.cubic_rl_plan_set_chunk(plan, columns)
        for flipped in (False, True):
            cr.cubic_rl_convolve(plan, dev(x), flipped, out)
            assert rel_l2(out, oracle.convolve(oracle.psf_spectrum(psf), x, flipped)) <= 1e-5, (columns, flipped)
    d = synth.random_field(shape, 7, 5.0, 50.0)
    cr.cubic_rl_deconvolve(plan, dev(d), 5, 1e-6, u)
    assert rel_l2(u, oracle.rl(d, psf, 5, 1e-6)) <= 1e-5


@pytest.mark.parametrize("ny", [121, 140, 187, 250, 301, 500, 1000])
def test_two_stage_y_linear(cr, ny):
    shape, k = (3, ny, 20), (3, 9, 5)
    psf = skewed_psf(k, ny)
    plan = cr.cubic_rl_plan_linear(shape, dev(psf))
    (_, n, _), chosen = cr.cubic_rl_plan_variants(plan)
    cr.cubic_rl_plan_set_variants(plan, chosen[0], n - 1, chosen[2])
    d = synth.random_field(shape, ny, 5.0, 50.0)
    u = torch.empty(shape, device="cuda")
    cr.cubic_rl_deconvolve(plan, dev(d), 4, 1e-6, u)
    assert rel_l2(u, oracle.rl_same(d, psf, 4, 1e-6)) <= 1e-5
