"""Launch shapes of plans that were not tuned: other ones for volumes past L2, by the kind of the
PSF's spectrum, and for monitored and accelerated calls at x = 512.

Tolerance: two launch shapes of the same float32 transforms, a few units of rounding after 4
iterations: 1e-5. The history's relative changes are differences of iterates a few percent apart: 1e-4.
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


def rel(a, b):
    return float((a.double() - b.double()).norm() / b.double().norm())




# below the threshold (96 MiB), above it, at each Y length that changes, and with a shorter z
@pytest.mark.parametrize("shape", [(64, 384, 1024), (64, 512, 1024), (100, 384, 768), (64, 768, 640), (50, 768, 768)])
def test_spectrum_kind_and_size(cr, shape):
    sym = torch.zeros(shape, device="cuda")
    c = [n // 2 for n in shape]
    sym[c[0] - 1:c[0] + 2, c[1] - 2:c[1] + 3, c[2] - 2:c[2] + 3] = 1 / 75
    skew = sym.clone()
    skew[c[0], c[1], c[2] + 3] = 0.1
    d = 5 + 45 * torch.rand(shape, device="cuda")
    plan, ref = cr.cubic_rl_plan(shape, sym), cr.cubic_rl_plan(shape, sym)
    cr.cubic_rl_plan_set_variants(ref, 0, 0, 0)
    a, b = torch.empty_like(d), torch.empty_like(d)
    shapes = set()
    for psf in (sym, skew, sym):
        for p, out in ((plan, a), (ref, b)):
            cr.cubic_rl_plan_update_psf(p, psf)
            cr.cubic_rl_deconvolve(p, d, 4, 1e-6, out)
        assert rel(a, b) <= 1e-5
        shapes.add(cr.cubic_rl_plan_variants(plan)[1])
    assert cr.cubic_rl_plan_variants(ref)[1] == (0, 0, 0)
    # y = 512 takes the same shapes for both kinds, the others another one for a real spectrum
    past_l2 = 4 * d.numel() > 96 << 20 and shape[0] >= 64
    assert len(shapes) == (2 if past_l2 and shape[1] != 512 else 1)


@pytest.mark.parametrize("shape", [(3, 5, 512), (9, 25, 512), (4, 6, 384)])
def test_heavy_calls(cr, shape):
    psf = oracle.psf_gaussian(shape, 1.0, 1.5).astype(np.float32)
    d = synth.random_field(shape, 7, 5.0, 50.0)
    plan = cr.cubic_rl_plan(shape, dev(psf))
    before = cr.cubic_rl_plan_variants(plan)[1]
    u, x, v = (torch.empty(shape, device="cuda") for _ in range(3))
    n, hist = cr.cubic_rl_deconvolve_monitor(plan, dev(d), 5, 1e-6, cr.METRIC_NLL, 0.0, 5, u)
    cr.cubic_rl_deconvolve_accel(plan, dev(d), 5, 1e-6, x)
    cr.cubic_rl_plan_set_variants(plan, *before)  # these calls on the plain calls' shape
    n2, hist2 = cr.cubic_rl_deconvolve_monitor(plan, dev(d), 5, 1e-6, cr.METRIC_NLL, 0.0, 5, v)
    assert n == n2 == 5 and np.allclose(hist, hist2, rtol=1e-4, equal_nan=True)
    assert rel(u, v) <= 1e-5 and rel(u, dev(oracle.rl(d, psf, 5, 1e-6))) <= 1e-5
    cr.cubic_rl_deconvolve_accel(plan, dev(d), 5, 1e-6, v)
    assert rel(x, v) <= 1e-5
    assert cr.cubic_rl_plan_variants(plan)[1] == before
