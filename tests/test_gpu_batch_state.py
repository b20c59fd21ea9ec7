"""Batched calls with the same arguments after a plan changed: the cached graph must not run the
plan's former state (PSF spectrum of another kind, former workspace, another plan's buffers).

Tolerance: the batched and the plain call run the same kernels or other shapes of the same
passes in float32, a few units of rounding after 4 iterations (3e-6, as in test_gpu_batched).
"""
import numpy as np
import pytest

from paper_2510_14143_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# the fused form, and the pass-by-pass form (an axis beyond the fused form's)
SHAPES = [(16, 20, 32), (8, 12, 256)]


@pytest.fixture(scope="module")
def cr():
    from paper_2510_14143_gb300 import build
    build.build()
    import paper_2510_14143_gb300 as m
    return m


def symmetric(shape):
    """Values that mirror bitwise about the centre: the real-spectrum path."""
    g = np.meshgrid(*[np.arange(n) - n // 2 for n in shape], indexing="ij")
    p = np.exp(-0.5 * sum((a / 1.7) ** 2 for a in g)).astype(np.float32)
    return p / p.sum()


def skewed(shape, seed):
    r = np.random.default_rng(seed)
    p = (r.uniform(0.0, 1.0, shape) ** 4).astype(np.float32)
    p[tuple(n // 2 for n in shape)] += 0.2 * p.sum()
    return p / p.sum()


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def rel_l2(a, b):
    a, b = (np.asarray(v.cpu(), np.float64) for v in (a, b))
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


class Batch:
    def __init__(self, cr, psfs):
        self.cr = cr
        self.plans = [cr.cubic_rl_plan(s, dev(p)) for s, p in zip(SHAPES, psfs)]
        self.images = [dev(synth.random_field(s, 3 + sum(s), 5.0, 50.0)) for s in SHAPES]
        self.outs = [torch.empty(s, device="cuda") for s in SHAPES]

    def check(self):
        self.cr.cubic_rl_deconvolve_batched(self.plans, self.images, 4, 1e-6, self.outs)
        got = [o.clone() for o in self.outs]
        for plan, im, out in zip(self.plans, self.images, got):
            ref = torch.empty_like(im)
            self.cr.cubic_rl_deconvolve(plan, im, 4, 1e-6, ref)
            assert rel_l2(out, ref) <= 3e-6


def test_psf_updates_between_batches(cr):
    b = Batch(cr, [symmetric(s) for s in SHAPES])
    b.check()
    for make in (lambda s: skewed(s, 1), symmetric, lambda s: skewed(s, 2), lambda s: skewed(s, 3)):
        for plan, s in zip(b.plans, SHAPES):
            cr.cubic_rl_plan_update_psf(plan, dev(make(s)))
        b.check()


def test_workspace_and_wait_limit_between_batches(cr):
    b = Batch(cr, [skewed(s, 4) for s in SHAPES])
    b.check()
    for plan in b.plans:
        n = cr.cubic_rl_workspace_bytes(plan)
        cr.cubic_rl_set_workspace(plan, torch.empty(n, dtype=torch.uint8, device="cuda"))
    b.check()
    for plan in b.plans:
        cr.cubic_rl_plan_set_wait_limit(plan, 1_000_000_000)
    b.check()


def test_new_plans_in_place_of_destroyed_ones(cr):
    b = Batch(cr, [skewed(s, 5) for s in SHAPES])
    b.check()
    for seed in range(6, 10):
        for i, s in enumerate(SHAPES):
            b.plans[i].close()
            b.plans[i] = cr.cubic_rl_plan(s, dev(skewed(s, seed)))
        b.check()
