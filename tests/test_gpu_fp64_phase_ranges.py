"""FP64 phases outside the range of the in-line sine and cosine (a network at
rest next to 0, phases wound past 2^21) are not much slower than those inside.
65536 orbits of n = 8, 100 steps: Euler-Maruyama 0.93 ms inside, 1.45 at rest,
1.54 past 2^21; Runge-Kutta 0.81, 1.68 and 1.75 (with CUDA's sincos for every
phase: 7.5 and 3.46).  The bound leaves a factor of 1.4 over the largest of
these ratios for noise."""
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


def _time(x0, scheme):
    orbits, n = x0.shape
    pb = sdeb.Problem.make("kuramoto", n, orbits, 0.01, 100, 100, 3, "fp64", rk4=scheme == "rk4", no_frames=True)
    p = torch.zeros((orbits, n + 2), dtype=torch.float64, device="cuda")
    p[:, 0] = 1.0
    best = float("inf")
    with Integrator(pb) as it:
        for _ in range(5):
            it.set_params(p, x0)
            start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            start.record()
            it.integrate()
            end.record()
            end.synchronize()
            best = min(best, start.elapsed_time(end))
    return best


@pytest.mark.parametrize("scheme", ["em", "rk4"])
def test_no_range_of_phases_is_much_slower(scheme):
    u = torch.rand((65536, 8), dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    inside = _time(1.0 + u, scheme)
    for outside in (torch.zeros_like(u), 1e-5 * u, 1e7 + u):
        assert _time(outside, scheme) <= 3.0 * inside
