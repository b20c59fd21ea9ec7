"""The constant that the fused form takes off the ratio: PSFs of any sum, images without
background, a large eps, an empty image.

Tolerance: float32 transforms, a few units of rounding times log2(V) per convolution, 1e-5 after
6 iterations whatever the PSF's sum is (the iteration is scale-free: the ratio carries 1 / sum and
the correlation the sum again).
"""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [(16, 20, 32), (27, 45, 36)]


@pytest.fixture(scope="module")
def cr():
    from paper_2510_14143_gb300 import build
    build.build()
    import paper_2510_14143_gb300 as m
    return m


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def image(shape, background, seed):
    r = np.random.default_rng(seed)
    o = np.full(shape, float(background))
    for _ in range(5):
        o[tuple(r.integers(0, n) for n in shape)] += r.uniform(2e3, 1e4)
    blur = oracle.convolve(oracle.psf_spectrum(oracle.psf_gaussian(shape, 1.5, 1.2).astype(np.float32)),
                           o.astype(np.float32), False)
    return r.poisson(np.maximum(blur, 0)).astype(np.float32)


def calls(cr, plan, shape, psf, d, n, eps):
    """The plain calls that run in the fused form."""
    u, m, a, b, f = (torch.full(shape, float("nan"), device="cuda") for _ in range(5))
    cr.cubic_rl_deconvolve(plan, dev(d), n, eps, u)
    cr.cubic_rl_deconvolve_monitor(plan, dev(d), n, eps, cr.METRIC_REL_CHANGE, 0.0, 2, m)
    cr.cubic_rl_deconvolve_auto(plan, dev(d), n, eps, 0.0, 2, a)
    cr.cubic_rl_deconvolve_batched([plan], [dev(d)], n, eps, [b])
    cr.cubic_rl_deconvolve_noalloc(shape, dev(psf), dev(d), n, eps, f)
    return [v.cpu().numpy().astype(np.float64) for v in (u, m, a, b, f)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("background", [10.0, 0.3, 0.0])
@pytest.mark.parametrize("total,eps", [(1.0, 1e-6), (1.0, 30.0), (1e-3, 1e-6), (250.0, 1e-6), (1e5, 1e-6)])
def test_psf_sums_and_backgrounds(cr, shape, background, total, eps):
    d = image(shape, background, 7 + sum(shape))
    psf = (oracle.psf_gaussian(shape, 1.5, 1.2) * total).astype(np.float32)
    ref = oracle.rl(d, psf, 6, eps)
    for got in calls(cr, cr.cubic_rl_plan(shape, dev(psf)), shape, psf, d, 6, eps):
        assert np.linalg.norm(got - ref) / np.linalg.norm(ref) <= 1e-5


def test_sum_changes_with_the_psf(cr):
    shape = SHAPES[0]
    d = image(shape, 10.0, 3)
    base = oracle.psf_gaussian(shape, 1.5, 1.2)
    plan = cr.cubic_rl_plan(shape, dev(base))
    u = torch.empty(shape, device="cuda")
    for total in (1e4, 1.0, 1e-3):
        psf = (base * total).astype(np.float32)
        cr.cubic_rl_plan_update_psf(plan, dev(psf))
        cr.cubic_rl_deconvolve(plan, dev(d), 6, 1e-6, u)
        ref = oracle.rl(d, psf, 6, 1e-6)
        assert np.linalg.norm(u.cpu().numpy() - ref) / np.linalg.norm(ref) <= 1e-5


def test_empty_image_gives_zero(cr):
    shape = SHAPES[0]
    psf = oracle.psf_gaussian(shape, 1.5, 1.2).astype(np.float32)
    for got in calls(cr, cr.cubic_rl_plan(shape, dev(psf)), shape, psf, np.zeros(shape, np.float32), 3, 1e-6):
        assert (got == 0).all()
