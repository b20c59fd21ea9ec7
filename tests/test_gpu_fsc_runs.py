"""FSC shell sums with runs of 2 and of 8 frequencies per thread: both sides of the size where the
run length changes, rows that end inside a run.

Tolerance: as for every FSC here, 1e-4 against the oracle.
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


# 64x60x150 has 38400 runs of 8, 64x64x150 40960: the line is at 38912
@pytest.mark.parametrize("shape", [(1, 8, 9), (9, 8, 10), (15, 36, 32), (50, 108, 45), (27, 81, 128), (64, 60, 150), (64, 64, 150)])
@pytest.mark.parametrize("shells", [1, 4, 1024])
def test_fsc(cr, shape, shells):
    a = synth.random_field(shape, 1, 0.0, 2.0)
    b = a + synth.random_field(shape, 2, -1.0, 1.0)
    psf = np.zeros(shape, np.float32)
    psf[tuple(n // 2 for n in shape)] = 1
    got = cr.cubic_fsc(cr.cubic_rl_plan(shape, dev(psf)), dev(a), dev(b), shells)
    assert np.allclose(got.cpu().numpy(), oracle.fsc(a, b, shells)[0], atol=1e-4)
