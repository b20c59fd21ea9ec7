"""Batches with volumes that run the plain call's passes (4 million voxels and more): the same
results as plain calls to the bit, on fresh plans and after their launch shapes or chunks changed.

Tolerance: other volumes share launches of other shapes, a few units of rounding (3e-6, as in
test_gpu_batched).
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# 4 194 304, 10 240, 3 932 160 (below the line), 24 576 and 4 096 000 voxels
SHAPES = [(64, 256, 256), (16, 20, 32), (60, 256, 256), (8, 12, 256), (100, 160, 256)]
ALONE = (0, 4)


@pytest.fixture(scope="module")
def cr():
    from paper_2510_14143_gb300 import build
    build.build()
    import paper_2510_14143_gb300 as m
    return m


def check(cr, plans, images, outs):
    cr.cubic_rl_deconvolve_batched(plans, images, 3, 1e-6, outs)
    for i, (plan, im, out) in enumerate(zip(plans, images, outs)):
        ref = torch.empty_like(im)
        cr.cubic_rl_deconvolve(plan, im, 3, 1e-6, ref)
        assert torch.equal(out, ref) if i in ALONE else float((out - ref).norm() / ref.norm()) <= 3e-6


def test_large_volumes_in_a_batch(cr):
    plans, images = [], []
    for s in SHAPES:
        psf = torch.empty(s, device="cuda")
        cr.cubic_psf_gaussian(s, 1.5, 1.2, 1.0, psf)
        plans.append(cr.cubic_rl_plan(s, psf))
        images.append(5 + 45 * torch.rand(s, device="cuda"))
    outs = [torch.empty_like(im) for im in images]
    check(cr, plans, images, outs)
    check(cr, plans, images, outs)  # the cached graph
    cr.cubic_rl_plan_set_variants(plans[0], 0, 0, 0)
    cr.cubic_rl_plan_set_chunk(plans[4], 32)
    check(cr, plans, images, outs)
    # a batch of such volumes alone
    cr.cubic_rl_deconvolve_batched(plans[::4], images[::4], 3, 1e-6, outs[::4])
    for i in ALONE:
        ref = torch.empty_like(images[i])
        cr.cubic_rl_deconvolve(plans[i], images[i], 3, 1e-6, ref)
        assert torch.equal(outs[i], ref)
