"""The FP32 FitzHugh-Nagumo step on pairs of units, at the edges of its
layouts (lanes of 1, 2, 4 and 8 units, padded last lanes), against the FP64
kernel on the same noise.

Tolerance: 300 steps of 0.01, each increment below 0.1 and rounded a few
times at 2^-24, the normals off by 2^-20 each (special-function unit) times
sigma sqrt(dt) v <= 0.02: below 300 (1e-8 + 2e-8) = 1e-5 even if every error
had the same sign.
"""
import pytest
import torch

import paper_1908_03869_gb300 as sdeb
from paper_1908_03869_gb300 import build as sdeb_build
from paper_1908_03869_gb300 import inputs
from paper_1908_03869_gb300.integrator import Integrator

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    sdeb_build.build()
    sdeb.lib()


def _final(n, p, x0, precision, milstein):
    dtype = torch.float64 if precision == "fp64" else torch.float32
    pb = sdeb.Problem.make("fhn_net", n, len(x0), 0.01, 300, 300, 3, precision, milstein=milstein)
    with Integrator(pb) as it:
        it.set_params(p.to(dtype).cuda(), x0.to(dtype).cuda())
        it.integrate()
        return it.final().double().cpu()


@pytest.mark.parametrize("milstein", [False, True])
@pytest.mark.parametrize("units", [1, 2, 3, 4, 5, 7, 8, 9, 12, 17, 63, 64, 129, 256])
def test_fp32_follows_fp64(units, milstein):
    p, x0 = (torch.tensor(a).float() for a in inputs.fhn(units, 41, seed=units))
    f32, f64 = (_final(2 * units, p, x0, prec, milstein) for prec in ("fp32", "fp64"))
    assert ((f32 - f64).abs() / f64.abs().clamp(min=1.0)).max().item() < 1e-5
