"""Column chunks of the Y/Z/Y sequence with every Z shape: the tiles of some are wider than the
narrowest chunk.

Tolerance: the same transforms on other tiles, 1e-5 for one float32 convolution against the oracle.
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
    return float(np.linalg.norm(a.cpu().numpy().astype(np.float64) - b) / np.linalg.norm(b))


# nz 16 to 40: 64-column Z tiles by default; 128 and 160: shapes of 32 columns; 129 to 193
# spectrum columns, so that the last chunk and the last tile are both ragged
@pytest.mark.parametrize("shape", [(16, 6, 256), (30, 5, 384), (40, 4, 320), (25, 9, 135), (128, 3, 256), (160, 2, 384)])
@pytest.mark.parametrize("symmetric", [False, True])
def test_chunks(cr, shape, symmetric):
    r = np.random.default_rng(sum(shape))
    psf = oracle.psf_gaussian(shape, 1.5, 1.2).astype(np.float32) if symmetric else \
        (r.uniform(0.0, 1.0, shape) ** 4).astype(np.float32)
    plan = cr.cubic_rl_plan(shape, dev(psf / psf.sum()))
    psf = psf / psf.sum()
    x = synth.random_field(shape, 3 + sum(shape), -1.0, 2.0)
    want = oracle.convolve(oracle.psf_spectrum(psf), x, True)
    out = torch.empty(shape, device="cuda")
    (_, ny, nz), (vx, vy, vz) = cr.cubic_rl_plan_variants(plan)
    for shapes in [None] + [(vx, vy, v) for v in range(nz)] + [(vx, v, vz) for v in range(ny)]:
        if shapes:
            cr.cubic_rl_plan_set_variants(plan, *shapes)
        for columns in (16, 32, 48, 80, 1024):
            cr.cubic_rl_plan_set_chunk(plan, columns)
            out.fill_(float("nan"))
            cr.cubic_rl_convolve(plan, dev(x), True, out)
            assert rel_l2(out, want) <= 1e-5, (shapes, columns)
            assert cr.cubic_rl_plan_chunk(plan) == columns


def test_chunk_off_returns_to_the_former_form(cr):
    """A small volume's plan runs chunks pass by pass; without them it runs as before, bit for bit."""
    shape = (16, 20, 32)
    psf = oracle.psf_gaussian(shape, 1.5, 1.2).astype(np.float32)
    plan = cr.cubic_rl_plan(shape, dev(psf))
    x = dev(synth.random_field(shape, 3, -1.0, 2.0))
    outs = []
    for columns in (0, 16, 0):
        cr.cubic_rl_plan_set_chunk(plan, columns)
        outs.append(torch.empty(shape, device="cuda"))
        cr.cubic_rl_convolve(plan, x, False, outs[-1])
    assert torch.equal(outs[0], outs[2])
    assert not torch.equal(outs[0], outs[1])  # two forms of the same transforms round differently
