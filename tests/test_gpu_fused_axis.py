"""The fused form's choice of the in-plane axis by expected time: volumes on both sides of it, both
in-plane lengths odd, even and mixed.

Tolerance: float32 transforms, 1e-5 for one convolution (as for the pass-by-pass form).
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


# the first two leave the even axis for the odd one, the last one the smaller plane
@pytest.mark.parametrize("shape", [(45, 100, 192), (45, 60, 192), (54, 64, 90), (75, 80, 144), (45, 64, 64), (45, 75, 81), (18, 32, 54)])
def test_convolve(cr, shape):
    r = np.random.default_rng(sum(shape))
    psf = (r.uniform(0.0, 1.0, shape) ** 4).astype(np.float32)
    psf /= psf.sum()
    x = synth.random_field(shape, 11 + sum(shape), -1.0, 2.0)
    plan = cr.cubic_rl_plan(shape, dev(psf))
    out = torch.full(shape, float("nan"), device="cuda")
    for flipped in (False, True):
        cr.cubic_rl_convolve(plan, dev(x), flipped, out)
        want = oracle.convolve(oracle.psf_spectrum(psf), x, flipped)
        assert np.linalg.norm(out.cpu().numpy() - want) / np.linalg.norm(want) <= 1e-5
