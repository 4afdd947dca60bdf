"""The variances of FP32 frames are as exact as FP64 sums make them.

256 components and at most 16 orbits: a component's sums are one thread's and one
group's, without a merge.  With A = sum (x - K)^2 / M2 (K the first orbit's
value), s2 and s1^2 / count are A M2 and (A - 1) M2, each rounded at most three
times by 2^-53 on the way to M2, which is rounded twice more: 6 A + 2 units at
most.  Exact sums rounded to FP64 meet it; sums of 47 bits are off by up to 64
units each.
"""
import numpy as np
import pytest
import torch

import paper_1908_03869_gb300 as sdeb
from paper_1908_03869_gb300 import build as sdeb_build
from paper_1908_03869_gb300.integrator import Integrator

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    sdeb_build.build()
    sdeb.lib()


@pytest.mark.parametrize("orbits", [3, 9, 16])
@pytest.mark.parametrize("offset,scale", [(0.0, 1.0), (3.0, 3.0), (100.0, 1.0), (0.0, 1e-6), (-7.0, 1e3)])
def test_variance_to_its_last_bits(orbits, offset, scale):
    rng = np.random.default_rng(orbits)
    x = (offset + scale * rng.standard_normal((orbits, 256))).astype(np.float32)
    pb = sdeb.Problem.make("ou", 256, orbits, 1e-3, 1, 1, 0, "fp32")
    with Integrator(pb) as it:
        it.set_params(torch.zeros((orbits, 2), device="cuda"), torch.tensor(x, device="cuda"))
        it.integrate()
        var = it.moments(begin=0, count=1)[0].cpu().numpy()[0, :, 1]
    exact = x.astype(np.longdouble)
    want = exact.var(0)
    a = ((exact - exact[0]) ** 2).mean(0) / want
    assert np.max(np.abs(var - want) / want / (6 * a + 2)) <= 2.0 ** -53
