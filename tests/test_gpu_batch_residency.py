"""The batch's resident blocks per SM follow its chains: fewer where a few
long chains decide, more where there is work for every issue slot.
"""
import pytest
import torch

import paper_1908_03869_gb300 as sdeb
from paper_1908_03869_gb300 import build as sdeb_build
from paper_1908_03869_gb300 import inputs
from paper_1908_03869_gb300.integrator import BatchIntegrator

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    sdeb_build.build()
    sdeb.lib()


def _batch(sizes, orbits):
    pbs = [sdeb.Problem.make("kuramoto", n, orbits, 0.005, steps, steps, 0, "fp32") for n, steps in sizes]
    data = [inputs.kuramoto(n, orbits, seed=i) for i, (n, _) in enumerate(sizes)]
    to = lambda i: [torch.tensor(d[i], dtype=torch.float32, device="cuda") for d in data]  # noqa: E731
    return BatchIntegrator(pbs), to(0), to(1)


def _final(it, p, x0):
    it.set_params(p, x0)
    it.integrate()
    return [it.final(i).cpu() for i in range(len(p))]


def test_residency_follows_the_chains():
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    long_chains, p, x0 = _batch([(200, 4000)] * 3 + [(40, 100)] * 3, sms // 2)
    short_ones, q, y0 = _batch([(n, 60) for n in range(8, 72)], 2 * sms)
    with long_chains, short_ones:
        assert long_chains.info()["grid"] <= 2 * sms < short_ones.info()["grid"]
        first = _final(long_chains, p, x0)
        long_chains.set_params(p, x0)
        long_chains.autotune()
        for a, b in zip(first, _final(long_chains, p, x0)):
            assert torch.allclose(a, b, rtol=0, atol=1e-3)  # another layout may be picked: FP32 rounding
        assert all(torch.isfinite(t).all() for t in _final(short_ones, q, y0))
