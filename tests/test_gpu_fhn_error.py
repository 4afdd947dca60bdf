"""The FP32 FitzHugh-Nagumo step on pairs of units is no further from the
64-bit result than the scalar step that it took the place of.

Root mean square errors over ten seeds (2048 orbits of 64 units, 400 steps of
0.01, relative to the states): scalar 3.438e-8 (Milstein 3.460e-8) with a standard
error of 4e-11 over the seeds; five of them, 2e-10, are allowed.  The FP64
kernel's own error is 1e-15.  And sigma / sqrt(dt) may lie past the FP32
range, as it may for the scalar step.
"""
import pytest
import torch

import paper_1908_03869_gb300 as sdeb
from paper_1908_03869_gb300 import build as sdeb_build
from paper_1908_03869_gb300.integrator import Integrator

pytestmark = pytest.mark.gpu
ORBITS, UNITS = 2048, 64


@pytest.fixture(scope="module", autouse=True)
def _built():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    sdeb_build.build()
    sdeb.lib()


def _final(p, x0, precision, seed, dt, steps, milstein):
    dtype = torch.float64 if precision == "fp64" else torch.float32
    pb = sdeb.Problem.make("fhn_net", 2 * UNITS, len(x0), dt, steps, steps, seed, precision, milstein=milstein)
    with Integrator(pb) as it:
        it.set_params(p.to(dtype), x0.to(dtype))
        it.integrate()
        return it.final().double()


def _inputs(seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    u = lambda cols, low, high: low + (high - low) * torch.rand((ORBITS, cols), generator=g, device="cuda")  # noqa: E731
    p = torch.cat([u(1, 0.6, 0.8), u(1, 0.7, 0.9), u(1, 0.05, 0.1), u(1, 0.3, 0.6), u(1, 0.0, 0.5), u(1, 0.01, 0.1)], 1)
    return p, torch.cat([u(UNITS, -2.0, 2.0), u(UNITS, -0.5, 1.5)], 1)


@pytest.mark.parametrize("milstein,scalar", [(False, 3.438e-8), (True, 3.460e-8)])
def test_error_of_the_scalar_step(milstein, scalar):
    rms = []
    for seed in range(10):
        p, x0 = _inputs(seed)
        f32, f64 = (_final(p, x0, prec, seed, 0.01, 400, milstein) for prec in ("fp32", "fp64"))
        rms.append(((f32 - f64).square().mean() / f64.square().mean()).sqrt())
    assert torch.stack(rms).mean().item() <= scalar + 2e-10


def test_constants_stay_in_range():
    p, x0 = _inputs(1)
    p[:, 5] = 1e30
    x0[:, 0] = 0.0
    f32, f64 = (_final(p, x0, prec, 1, 1e-20, 1, False) for prec in ("fp32", "fp64"))
    assert torch.isfinite(f32).all()
    assert ((f32 - f64).abs() <= 1e-5 * f64.abs().max()).all()  # normals off by 2^-20 each
